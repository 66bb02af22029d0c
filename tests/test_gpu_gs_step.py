"""pnp_gmres at the sizes around the change from one Gram-Schmidt launch to two (65,536
unknowns), at the smallest, and with a second pass and a restart length past the 64 vectors
that a round of the one launch adds: after a fixed number of iterations the iterate is the
one of GMRES written out in torch.  Tolerance 1e-8 relative, as there."""
import pytest

from paper_2301_05985_gb300 import workloads as W

from gpu_common import lib, torch_cuda
from test_gpu_gmres_sizes import _torch_gmres

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,level,m,its,two", [(2, 2, 6, 5, 0), (2, 3, 8, 12, 1), (2, 4, 70, 80, 0), (2, 4, 70, 80, 1),
                                                 (2, 7, 12, 15, 1), (3, 4, 24, 30, 0), (3, 5, 12, 15, 1)])
def test_iterates_match_plain_gmres(dim, level, m, its, two):
    pnp, torch = lib(), torch_cuda()
    mesh = pnp.Mesh(W.uniform_octants(dim, level))
    ctx = pnp.Context(mesh, pnp.default_params(eps=0.05, dt=0.01, gmres_restart=m, gmres_max_it=its, gmres_cgs2=two),
                      torch.cuda.current_stream().cuda_stream)
    ctx.set_bcs(W.membrane_bcs(dim, 2.0, 2.0))
    g = torch.Generator(device="cuda").manual_seed(level)
    n = mesh.n_nodes
    U = 1.0 + 0.2 * torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64)
    b = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    D = torch.zeros(n, 9, dtype=torch.float64, device="cuda")
    ctx.block_diag(U, D)
    Dinv = torch.linalg.inv(D.view(n, 3, 3))

    def op(v):
        return ctx.jv(U, v.contiguous(), torch.zeros_like(v))

    def prec(v):
        return torch.einsum("nij,nj->ni", Dinv, v)

    x = torch.zeros_like(b)
    ctx.gmres(U, b, x, 1e-30, raise_on_error=False)
    ref = _torch_gmres(torch, op, prec, b, m, its)
    assert float((x - ref).norm() / ref.norm()) <= 1e-8
