"""Beam selection from the shares' largest, against the selection oracle bit for bit: counts around the line from which shares are
used, ragged last shares, shares of 16 and of 64 candidates, few shares per survivor (the cluster kernel's side of the rule),
ties, special values, and survivors that gather in few shares (more reach the bound than shared memory holds)."""
import numpy as np
import pytest
import torch

from oracle import select as osel
import paper_2609_12399_b200 as P

pytestmark = pytest.mark.gpu


def _run(bs, lp, W_new):
    R, W_prev, C = lp.shape
    par = torch.empty((R, W_new), dtype=torch.int32, device="cuda")
    code, sc = torch.empty_like(par), torch.empty((R, W_new), device="cuda")
    W = max(W_prev, W_new)
    ctx = P.Onela(P.make_config(R, 1, 1, 32, 32, W, 2, "fp32", "fp32", R * W * 2, 0), device="cuda")
    for r in range(R):
        ctx.onela_init_shared_state(r, 0, torch.zeros(1, 32, 32, device="cuda"))
    ctx.onela_reorder_beams(0, R, None, W_prev)
    ctx.onela_select_beams(0, R, bs.cuda(), lp.cuda(), C, W_new, par, code, sc)
    torch.cuda.synchronize()
    for r in range(R):
        p, c, s = osel.select_beams(bs[r].numpy(), lp[r].numpy(), W_new)
        assert np.array_equal(par[r].cpu().numpy(), p) and np.array_equal(code[r].cpu().numpy(), c), r
        assert np.array_equal(sc[r].cpu().numpy().view(np.uint32), s.view(np.uint32)), r


@pytest.mark.parametrize("W_prev,C,W_new", [(64, 256, 64), (5, 3277, 100), (17, 1021, 33), (48, 1023, 1024), (48, 1024, 1024), (257, 191, 1000),
                                            (512, 512, 512), (1000, 263, 777), (1024, 1024, 1024), (1, 300000, 9)])
@pytest.mark.parametrize("quant", [None, 1])
def test_sizes_and_ties(W_prev, C, W_new, quant):
    gen = torch.Generator().manual_seed(W_prev * 31 + C)
    lp = torch.log_softmax(torch.randn((2, W_prev, C), generator=gen), dim=-1)
    bs = -3.0 * torch.rand((2, W_prev), generator=gen)
    if quant:
        lp, bs = torch.round(lp), torch.round(bs)
    _run(bs, lp, W_new)


@pytest.mark.parametrize("W_prev,C", [(64, 1500), (256, 1500)])        # shares of 16, of 64
def test_crowded_shares_and_special_values(W_prev, C):
    gen = torch.Generator().manual_seed(C)
    lp = torch.rand((1, W_prev, C), generator=gen)
    lp[0, 3:12] += 5.0                                  # 13 500 neighbours stand out: whole shares reach any bound
    _run(torch.zeros(1, W_prev), lp, 1000)
    lp = torch.full((1, W_prev, C), float("-inf"))
    lp[0, 5, 100:900] = float("nan")
    lp[0, 9, 3] = float("inf")
    lp[0, 11, :700], lp[0, 12, :50] = -0.0, 0.0
    _run(torch.zeros(1, W_prev), lp, 1000)
    _run(torch.full((1, W_prev), -0.0), lp, 700)        # survivors that are -0
