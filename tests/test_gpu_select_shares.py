"""Beam selection from the shares' largest, against the selection oracle bit for bit: counts around the lines from which shares are
used, ragged last shares, one CTA's shares of 16 and of 64 candidates and the cluster's, ties, special values, and candidates that
gather in few shares, so that more reach the bound than shared memory holds (which a replay of the layout confirms)."""
import numpy as np
import pytest
import torch

from oracle import select as osel
import paper_2609_12399_b200 as P

from _select_layout import LIST, crowd, reaching

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
        got, nan = sc[r].cpu().numpy(), np.isnan(s)          # (the payload of a NaN sum is the adder's)
        assert np.array_equal(np.isnan(got), nan) and np.array_equal(got[~nan].view(np.uint32), s[~nan].view(np.uint32)), r


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


@pytest.mark.parametrize("W_prev,C,W_new", [(300, 1000, 200), (128, 1024, 600), (128, 256, 600)])     # one CTA, cluster, threads' shares
def test_crowded_shares(W_prev, C, W_new):
    """Candidates that stand out lie in fewer shares than survive: all of them reach the bound, more than shared memory holds, and
    the list goes through the request's scratch (two requests, so each through its own)."""
    gen = torch.Generator().manual_seed(C)
    lp = torch.rand((2, W_prev, C), generator=gen)
    for r in range(2):
        lp[r].view(-1)[torch.from_numpy(crowd(W_prev * C, W_new))] += 5.0
        assert reaching(lp[r].view(-1).numpy(), W_new) > LIST
    _run(torch.zeros(2, W_prev), lp, W_new)


@pytest.mark.parametrize("W_prev,C,W_new", [(64, 1500, 1000), (256, 1500, 1000), (64, 1500, 200), (300, 1000, 200), (300, 1000, 66)])
def test_special_values_and_neighbours(W_prev, C, W_new):
    """The cluster's shares and one CTA's of 16 and of 64 candidates: neighbours that stand out, infinities, NaN, zeros of either
    sign, and scores that are all the same."""
    gen = torch.Generator().manual_seed(C)
    lp = torch.rand((1, W_prev, C), generator=gen)
    lp[0, 3:12] += 5.0
    _run(torch.zeros(1, W_prev), lp, W_new)
    lp = torch.full((1, W_prev, C), float("-inf"))
    lp[0, 5, 100:900] = float("nan")
    lp[0, 9, 3] = float("inf")
    lp[0, 11, :700], lp[0, 12, :50] = -0.0, 0.0
    _run(torch.zeros(1, W_prev), lp, W_new)
    _run(torch.full((1, W_prev), -0.0), lp, W_new * 7 // 10)        # survivors that are -0
    _run(torch.zeros(1, W_prev), torch.zeros(1, W_prev, C), W_new)
    _run(torch.zeros(1, W_prev), torch.full((1, W_prev, C), float("nan")), W_new)
