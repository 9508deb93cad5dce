"""The selection kernel where its bound and its list can go wrong, against the selection oracle bit for bit: one CTA and
clusters of 2, 4 and 8, shares that stay in registers and shares that do not, counts around the sort's sizes, scores that
are all equal, candidates that gather in few threads' shares (more reach the bound than shared memory holds)."""
import numpy as np
import pytest
import torch

from oracle import select as osel
import paper_2609_12399_b200 as P

pytestmark = pytest.mark.gpu


def _run(bs, lp, W_new, static=False):
    R, W_prev, C = lp.shape
    par = torch.empty((R, W_new), dtype=torch.int32, device="cuda")
    code, sc = torch.empty_like(par), torch.empty((R, W_new), device="cuda")
    if static:
        P.onela_select_beams_static(bs.cuda(), lp.cuda(), W_new, par, code, sc)
    else:
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


@pytest.mark.parametrize("W_prev,C,W_new", [(1, 1, 1), (1, 1024, 1024), (1, 1025, 1024), (8, 512, 513), (8, 513, 31), (33, 1000, 33),
                                            (64, 1023, 1024), (128, 1025, 512), (1024, 1024, 1024), (1000, 1048, 7)])
@pytest.mark.parametrize("quant", [None, 1])
def test_sizes_and_ties(W_prev, C, W_new, quant):
    gen = torch.Generator().manual_seed(W_prev * 31 + C)
    lp = torch.log_softmax(torch.randn((2, W_prev, C), generator=gen), dim=-1)
    bs = -3.0 * torch.rand((2, W_prev), generator=gen)
    if quant:
        lp, bs = torch.round(lp), torch.round(bs)
    _run(bs, lp, W_new)
    _run(bs, lp, W_new, static=True)


@pytest.mark.parametrize("static", [False, True])
def test_equal_scores_and_crowded_shares(static):
    _run(torch.zeros(1, 64), torch.zeros(1, 64, 2048), 1000, static)
    lp = torch.full((1, 64, 2048), float("-inf"))
    lp[0, 5, 100:900] = float("nan")
    lp[0, 9, 3] = float("inf")
    _run(torch.zeros(1, 64), lp, 1000, static)
    # 131 072 candidates on 8192 threads of 16: stripe j's candidates of threads 0 .. 699 (a thread's place in the stripe
    # moves by 977 per stripe) stand out, so 700 threads hold 11 200 candidates that reach any bound for k = 600
    gen = torch.Generator().manual_seed(3)
    flat = torch.rand(64 * 2048, generator=gen)
    for j in range(16):
        place = (torch.arange(700) + j * 977) % 8192
        flat[j * 8192 + place] += 5.0 - 0.001 * torch.rand(700, generator=gen)
    _run(torch.zeros(1, 64), flat.view(1, 64, 2048), 600, static)
