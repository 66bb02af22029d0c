"""The first FP32 J V of a context: the node tables are complete when the context is, so the
first call makes the launches of every later one (no table is built between its rows and its
J V), allocates no device memory, and has the FP64 J V's result.  Per-field maximum error 2e-5
of the field's largest entry, the bound of the FP32 J V against the oracle."""
import pytest

from paper_2301_05985_gb300 import workloads as W

from gpu_common import lib, torch_cuda

pytestmark = pytest.mark.gpu

MESHES = {
    "3d_one_element": lambda: W.uniform_octants(3, 0),
    "3d_octree": lambda: W.random_balanced_octants(3, 2, 4, 0.4, 1),
    "3d_band": lambda: W.membrane_band_octants(4, 7, 0.05),
    "2d_octree": lambda: W.random_balanced_octants(2, 6, 7, 0.4, 4),
}


@pytest.mark.parametrize("name", list(MESHES))
def test_first_call_is_like_the_next(name):
    pnp, torch = lib(), torch_cuda()
    oc = MESHES[name]()
    mesh = pnp.Mesh(oc)
    n = mesh.n_nodes
    g = torch.Generator(device="cuda").manual_seed(7)
    U = 0.5 + torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64)
    V = torch.rand(n, 3, generator=g, device="cuda") - 0.5
    out = torch.zeros(n, 3, device="cuda")
    ref = torch.zeros(n, 3, device="cuda", dtype=torch.float64)
    for i in range(3):
        ctx = pnp.Context(mesh, pnp.default_params(eps=0.05, dt=1e-3), torch.cuda.current_stream().cuda_stream)
        ctx.set_bcs(W.membrane_bcs(oc.dim, 2.0, 2.0))
        counts = []
        for _ in range(2):
            free, l0 = torch.cuda.mem_get_info()[0], pnp.kernel_launches()
            ctx.jv(U, V, out, pnp.PNP_F32)
            counts.append(pnp.kernel_launches() - l0)
            # (the process' first call also loads the kernels)
            assert i == 0 or torch.cuda.mem_get_info()[0] == free
        assert counts[0] == counts[1]
        ctx.jv(U, V.double(), ref)
        err = (out.double() - ref).abs().amax(0) / ref.abs().amax(0)
        assert bool((err <= 2e-5).all()), err
        ctx.close()
