"""pnp_gmres at the sizes where its reductions change shape: 3,267 unknowns (one row per
thread, iterations queued ahead of the host), 198,147 (four rows per thread) and 3,151,875
(sixteen rows; past 21 basis vectors the partials are added by a second kernel).  After a
fixed number of iterations (one restart among them) the iterate is compared with GMRES
written out in torch (modified Gram-Schmidt) on the library's J V and inverted blocks.

Tolerance 1e-8 relative: both minimise the same residual over the same space; classical and
modified Gram-Schmidt bases differ by rounding times the basis' condition (below 1e6 here)."""
import numpy as np
import pytest

from paper_2301_05985_gb300 import workloads as W

from gpu_common import lib, torch_cuda

pytestmark = pytest.mark.gpu


def _torch_gmres(torch, op, prec, b, m, its):
    x = torch.zeros_like(b)
    left = its
    while left > 0:
        r = b - op(x)
        beta = r.norm()
        V = [r / beta]
        k = min(m, left)
        H = torch.zeros(k + 1, k, dtype=torch.float64)
        for j in range(k):
            w = op(prec(V[j]))
            for i in range(j + 1):
                H[i, j] = torch.dot(V[i].reshape(-1), w.reshape(-1)).cpu()
                w = w - H[i, j].item() * V[i]
            H[j + 1, j] = w.norm().cpu()
            V.append(w / H[j + 1, j].item())
        e = torch.zeros(k + 1, 1, dtype=torch.float64)
        e[0] = beta.cpu()
        y = torch.linalg.lstsq(H, e).solution[:, 0]
        x = x + prec(sum(y[i].item() * V[i] for i in range(k)))
        left -= k
    return x


@pytest.mark.parametrize("level", [5, 8, 10])
def test_gmres_iterates_match_plain_gmres(level):
    pnp, torch = lib(), torch_cuda()
    oc = W.uniform_octants(2, level)
    mesh = pnp.Mesh(oc)
    m, its = 24, 30
    ctx = pnp.Context(mesh, pnp.default_params(eps=0.05, dt=0.01, gmres_restart=m, gmres_max_it=its),
                      torch.cuda.current_stream().cuda_stream)
    ctx.set_bcs(W.membrane_bcs(2, 2.0, 2.0))
    g = torch.Generator(device="cuda").manual_seed(level)
    n = mesh.n_nodes
    U = 1.0 + 0.2 * torch.rand(n, 3, generator=g, device="cuda", dtype=torch.float64)
    b = torch.randn(n, 3, generator=g, device="cuda", dtype=torch.float64)
    D = torch.zeros(n, 9, dtype=torch.float64, device="cuda")
    ctx.block_diag(U, D)
    Dinv = torch.linalg.inv(D.view(n, 3, 3))

    def op(v):
        out = torch.empty_like(v)
        return ctx.jv(U, v.contiguous(), out, pnp.PNP_F64)

    x = torch.zeros_like(b)
    st = ctx.gmres(U, b, x, 1e-14, pnp.PNP_F64, raise_on_error=False)
    assert st.krylov_its == its
    # the matrix actions of the iterations, the initial residual and one per cycle
    assert st.jv_evals == its + 1 + 2
    ref = _torch_gmres(torch, op, lambda v: torch.einsum("nij,nj->ni", Dinv, v), b, m, its)
    assert float((x - ref).norm() / ref.norm()) <= 1e-8
