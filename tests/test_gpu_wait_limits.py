"""Bounded waits that give up inside a solve, by a poll limit of 0 (every block still arrives, so
the counters are left as they were): the solve reports PNP_ERR_DEVICE_FLAG whichever element
kernels it runs on, and the context solves as before once the limit is back.  On the patch
kernels the only waits are those of the inner solve's Gram-Schmidt steps."""
import pytest

from paper_2301_05985_gb300 import workloads as W

from gpu_common import lib, torch_cuda

pytestmark = pytest.mark.gpu


def _system(**kw):
    pnp, torch = lib(), torch_cuda()
    oc = W.random_balanced_octants(3, 1, 4, 0.3, 12)
    mesh = pnp.Mesh(oc)
    ctx = pnp.Context(mesh, pnp.default_params(eps=0.1, dt=1e-3, **kw), torch.cuda.current_stream().cuda_stream)
    ctx.set_bcs(W.membrane_bcs(3, 2.0, 2.0))
    g = torch.Generator(device="cuda").manual_seed(3)
    U = 1.0 + 0.1 * torch.rand(mesh.n_nodes, 3, generator=g, device="cuda", dtype=torch.float64)
    b = torch.rand(mesh.n_nodes, 3, generator=g, device="cuda", dtype=torch.float64) - 0.5
    return pnp, torch, ctx, U, b, torch.zeros_like(b)


@pytest.mark.parametrize("path,precision,inner", [("lanes", "PNP_F32", 8), ("patch", "PNP_F32", 8),
                                                  ("lanes", "PNP_F64", 0), ("patch", "PNP_F64", 0)])
def test_a_wait_that_gives_up_is_reported(path, precision, inner, monkeypatch):
    if path == "patch":
        monkeypatch.setenv("PNP_ELEMENT_PATH", "patch")
    pnp, torch, ctx, U, b, x = _system(gmres_inner=inner, gmres_restart=30, gmres_max_it=300)
    prec = getattr(pnp, precision)
    before = ctx.gmres(U, b, x, 1e-6, prec, raise_on_error=False)
    assert before.status == (0 if precision == "PNP_F64" else pnp.PNP_ERR_KRYLOV_MAXIT)  # FP32: its rounding floor
    ctx.set_wait_limit(0)
    x.zero_()
    assert ctx.gmres(U, b, x, 1e-6, prec, raise_on_error=False).status == pnp.PNP_ERR_DEVICE_FLAG
    ctx.set_wait_limit(-1)
    x.zero_()
    assert ctx.gmres(U, b, x, 1e-6, prec, raise_on_error=False).status == before.status
    r = torch.zeros_like(b)
    ctx.jv(U, x, r)
    # FP32 operator in the mixed solve: its rounding on top of the solver's tolerance
    assert float((b - r).norm() / b.norm()) <= (1e-5 if prec == pnp.PNP_F64 else 1e-3)


def test_no_work_is_left_behind_an_error_return():
    """The FP64 solve of a small system queues an iteration ahead of the host.  A solve that ends
    in its first iteration (here by a wait that gives up) leaves nothing on the stream, where it
    would read the caller's U after the call, and counts the initial residual's J V and its
    own iteration's."""
    pnp, torch, ctx, U, b, x = _system(gmres_restart=30, gmres_max_it=300)
    ctx.set_wait_limit(0)
    for _ in range(5):
        st = ctx.gmres(U, b, x, 1e-6, pnp.PNP_F64, raise_on_error=False)
        assert torch.cuda.current_stream().query()
        assert st.status == pnp.PNP_ERR_DEVICE_FLAG and st.jv_evals == 2
