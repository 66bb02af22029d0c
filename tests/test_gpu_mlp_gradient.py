"""The network's training gradient at the edges of its tiles: 32-row tiles (one short, one
more than a tile), the row splits of the weight gradients (a first split of one block of
rows, more rows than CTAs hold at once) and the largest batch, against the oracle's FP64
backward pass; and inputs that are not 16-byte aligned give the aligned call's bits.

Tolerance 3e-2 relative per parameter block: each of up to six BF16 roundings (2^-8 spacing,
2^-9 error) between an input and a gradient entry enters with a factor near one."""
import numpy as np
import pytest

import mlp_oracle as MO
from paper_2301_05985_gb300 import workloads as W

from test_gpu_mlp import _ctx, pack, unpack

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B", [1, 31, 33, 513, 152 * 32 + 1, 65536])
def test_gradient_at_tile_edges(B):
    pnp, torch, mesh, ctx = _ctx(W.uniform_octants(3, 2))
    rng = np.random.default_rng(B)
    Ws, bs = MO.init_params(2)
    bs = [b + rng.normal(0, 0.05, b.shape) for b in bs]
    p = pack(Ws, bs)
    ctx.mlp_set_weights(p)
    X = rng.normal(size=(B, 216)).astype(np.float32)
    Y = rng.normal(size=(B, 3)).astype(np.float32)
    g = torch.full((pnp.PNP_MLP_PARAMS,), float("nan"), dtype=torch.float32, device="cuda")
    Yd = torch.from_numpy(Y).cuda()
    loss = ctx.mlp_loss_grad(torch.from_numpy(X).cuda(), Yd, g)
    Wr, br = unpack(p)
    gW, gb, lref = MO.backward([MO.bf16_round(w) for w in Wr], br, MO.bf16_round(X), Y.astype(np.float64))
    assert abs(loss - lref) <= 3e-2 * lref
    gWg, gbg = unpack(g.cpu().numpy().astype(np.float64))
    for l in range(4):
        assert np.linalg.norm(gWg[l] - gW[l]) <= 3e-2 * np.linalg.norm(gW[l]), l
        assert np.linalg.norm(gbg[l] - gb[l]) <= 3e-2 * np.linalg.norm(gb[l]), l
    if B == 513:
        buf = torch.zeros(B * 216 + 1, dtype=torch.float32, device="cuda")
        shifted = buf[1:].view(B, 216)
        shifted.copy_(torch.from_numpy(X))
        g2 = torch.zeros_like(g)
        assert ctx.mlp_loss_grad(shifted, Yd, g2) == loss and torch.equal(g, g2)
