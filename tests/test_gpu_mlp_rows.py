"""The network forward at row counts around its 128-row tiles and the 152 tiles of a first
pass, from input rows at odd 4-byte offsets, and through the allocation-free entry: the rows
are independent of one another, so every result is bit for bit the rows' part of one large
forward (which the parity tests hold to the oracle)."""
import numpy as np
import pytest

from paper_2301_05985_gb300 import workloads as W

from gpu_common import lib, torch_cuda

pytestmark = pytest.mark.gpu

ROWS = 3 * 152 * 128 + 5


@pytest.fixture(scope="module")
def net():
    pnp, torch = lib(), torch_cuda()
    ctx = pnp.Context(pnp.Mesh(W.uniform_octants(3, 2)), pnp.default_params(), torch.cuda.current_stream().cuda_stream)
    ctx.mlp_init(seed=3)
    params = (np.random.default_rng(11).normal(size=pnp.PNP_MLP_PARAMS) * 0.08).astype(np.float32)
    ctx.mlp_set_weights(params)
    g = torch.Generator(device="cuda").manual_seed(1)
    X = torch.randn(ROWS, 216, generator=g, device="cuda")
    out = torch.full((ROWS, 3), float("nan"), device="cuda")
    ctx.mlp_forward(X, out)
    assert bool(torch.isfinite(out).all())
    return pnp, torch, ctx, params, X, out


@pytest.mark.parametrize("rows", [1, 127, 128, 129, 152 * 128, 152 * 128 + 1, 2 * 152 * 128 + 3])
@pytest.mark.parametrize("offset", [0, 1])
def test_rows_do_not_depend_on_the_tiling(net, rows, offset):
    pnp, torch, ctx, params, X, ref = net
    buf = torch.empty(216 * rows + 4, device="cuda")
    x = buf[offset:offset + 216 * rows].view(rows, 216).copy_(X[1:1 + rows])
    out = torch.full((rows + 1, 3), float("nan"), device="cuda")
    ctx.mlp_forward(x, out[:rows])
    assert torch.equal(out[:rows], ref[1:1 + rows])
    assert bool(torch.isnan(out[rows]).all())  # nothing past the rows
    if rows <= pnp.PNP_NOALLOC_MAX_ROWS:
        out.fill_(float("nan"))
        pnp.mlp_forward_noalloc(torch.from_numpy(params).cuda(), x, out[:rows], torch.cuda.current_stream().cuda_stream)
        assert torch.equal(out[:rows], ref[1:1 + rows])
