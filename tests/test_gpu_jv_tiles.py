"""FP32 J V (node tiles) against the FP64 J V (lane kernel, itself held to the oracle) on meshes
of every tile width (32 to 128 threads on hexahedra, to 256 on quadrilaterals), with ragged
last tiles, hanging nodes, and node counts past the 32-bit sort keys; with and without
advection, at a new state and through the stored linearisation, into vectors that start at
an odd 4-byte offset.  Per-field maximum error 2e-5 of the field's largest entry, the bound
of the FP32 J V against the oracle."""
import pytest

from paper_2301_05985_gb300 import workloads as W

from gpu_common import lib, torch_cuda

pytestmark = pytest.mark.gpu

MESHES = {
    "3d_octree_small": lambda: W.random_balanced_octants(3, 2, 4, 0.4, 1),
    "3d_octree_medium": lambda: W.random_balanced_octants(3, 4, 5, 0.3, 2),
    "3d_band": lambda: W.membrane_band_octants(4, 7, 0.05),
    "3d_one_element": lambda: W.uniform_octants(3, 0),
    "3d_wide_keys": lambda: W.uniform_octants(3, 8),
    "2d_octree_small": lambda: W.random_balanced_octants(2, 4, 6, 0.4, 3),
    "2d_octree_medium": lambda: W.random_balanced_octants(2, 6, 7, 0.4, 4),
    "2d_octree_large": lambda: W.random_balanced_octants(2, 7, 8, 0.3, 5),
}


@pytest.mark.parametrize("adv", [False, True])
@pytest.mark.parametrize("name", list(MESHES))
def test_jv_f32_matches_f64(name, adv):
    pnp, torch = lib(), torch_cuda()
    oc = MESHES[name]()
    mesh = pnp.Mesh(oc)
    n, dim = mesh.n_nodes, oc.dim
    ctx = pnp.Context(mesh, pnp.default_params(eps=0.05, dt=1e-3), torch.cuda.current_stream().cuda_stream)
    ctx.set_bcs(W.membrane_bcs(dim, 2.0, 2.0))
    g = torch.Generator(device="cuda").manual_seed(7)

    def rand(*shape):
        return torch.rand(*shape, generator=g, device="cuda", dtype=torch.float64)

    U, prev = 0.5 + rand(n, 3), 0.5 + rand(n, 3)
    ctx.set_field(pnp.PNP_FIELD_U_PREV, prev.cpu().numpy())
    if adv:
        ctx.set_field(pnp.PNP_FIELD_ADVECTION, (rand(n, dim) - 0.5).cpu().numpy())
    V32 = torch.empty(3 * n + 1, device="cuda")[1:].view(n, 3).copy_(rand(n, 3) - 0.5)
    ref = torch.zeros(n, 3, device="cuda", dtype=torch.float64)
    ctx.jv(U, V32.double(), ref)
    scale = ref.abs().amax(0)
    new, lin = torch.zeros(3 * n + 1, device="cuda")[1:].view(n, 3), torch.zeros(n, 3, device="cuda")
    ctx.jv(U, V32, new, pnp.PNP_F32)
    ctx.linearize(U)
    ctx.jv_linearized(V32, lin)
    torch.cuda.synchronize()
    for out in (new, lin):
        err = (out.double() - ref).abs().amax(0) / scale
        assert bool((err <= 2e-5).all()), err
