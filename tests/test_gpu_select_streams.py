"""Selections of ONE request on two streams at once, each with buffers of its own: the workspace's scratch is one selection's at a
time, and the other one goes without it.  Every result against the selection oracle, bit for bit."""
import numpy as np
import pytest
import torch

from oracle import select as osel
import paper_2609_12399_b200 as P

from _select_layout import LIST, crowd, reaching

pytestmark = pytest.mark.gpu


def _context(W_prev, W_new):
    W = max(W_prev, W_new)
    ctx = P.Onela(P.make_config(1, 1, 1, 32, 32, W, 2, "fp32", "fp32", W * 2, 0), device="cuda")
    ctx.onela_init_shared_state(0, 0, torch.zeros(1, 32, 32, device="cuda"))
    ctx.onela_reorder_beams(0, 1, None, W_prev)
    torch.cuda.synchronize()
    return ctx


def _claim(ctx):
    at = ctx.workspace_ptr - ctx.workspace.data_ptr()
    return ctx.workspace[at + 16:at + 24].view(torch.int64)


def _inputs(gen, W_prev, C, W_new, crowded):
    lp, bs = torch.rand((1, W_prev, C), generator=gen), -3.0 * torch.rand((1, W_prev), generator=gen)
    if crowded:
        bs.zero_()
        lp.view(-1)[torch.from_numpy(crowd(W_prev * C, W_new))] += 5.0
        assert reaching(lp.view(-1).numpy(), W_new) > LIST
    return bs, lp


class _Call:
    def __init__(self, gen, W_prev, C, W_new, crowded):
        self.bs, self.lp = _inputs(gen, W_prev, C, W_new, crowded)
        self.args = (self.bs.cuda(), self.lp.cuda())
        self.out = (torch.empty((1, W_new), dtype=torch.int32, device="cuda"), torch.empty((1, W_new), dtype=torch.int32, device="cuda"),
                    torch.empty((1, W_new), device="cuda"))
        self.C, self.W_new = C, W_new

    def run(self, ctx, stream=None):
        ctx.onela_select_beams(0, 1, *self.args, self.C, self.W_new, *self.out, stream=stream)

    def check(self):
        p, c, s = osel.select_beams(self.bs[0].numpy(), self.lp[0].numpy(), self.W_new)
        par, code, sc = (x[0].cpu().numpy() for x in self.out)
        assert np.array_equal(par, p) and np.array_equal(code, c) and np.array_equal(sc.view(np.uint32), s.view(np.uint32))


# shares and one CTA (of 16, of 64 candidates), shares and a cluster, a cluster's own threads, and lists that shared memory cannot hold
SIZES = [(128, 1000, 128, False), (300, 1000, 200, False), (512, 256, 512, False), (48, 1024, 1024, False),
         (300, 1000, 200, True), (128, 1024, 600, True), (128, 256, 600, True)]


@pytest.mark.parametrize("W_prev,C,W_new,crowded", SIZES)
def test_two_streams(W_prev, C, W_new, crowded):
    gen = torch.Generator().manual_seed(W_prev + C)
    ctx = _context(W_prev, W_new)
    calls = [_Call(gen, W_prev, C, W_new, crowded) for _ in range(6)]
    streams = [torch.cuda.Stream(), torch.cuda.Stream()]
    torch.cuda.synchronize()
    for _ in range(20):
        for i, call in enumerate(calls):
            call.run(ctx, streams[i & 1])
    torch.cuda.synchronize()
    for call in calls:
        call.check()
    assert _claim(ctx).item() == 0


@pytest.mark.parametrize("W_prev,C,W_new,crowded", SIZES)
def test_scratch_claimed_by_another(W_prev, C, W_new, crowded):
    gen = torch.Generator().manual_seed(W_prev + C + 1)
    ctx = _context(W_prev, W_new)
    _claim(ctx)[0] = (1 << 20) + 3           # what another selection of the request would have left there
    call = _Call(gen, W_prev, C, W_new, crowded)
    call.run(ctx)
    torch.cuda.synchronize()
    call.check()
    assert _claim(ctx).item() == (1 << 20) + 3
    _claim(ctx)[0] = 0
    call.run(ctx)
    torch.cuda.synchronize()
    call.check()
    assert _claim(ctx).item() == 0
