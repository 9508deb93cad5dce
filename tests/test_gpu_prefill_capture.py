"""Prefill and export as dependent launches: captured in a CUDA graph and replayed on new inputs, and back to back on one stream
with a caller's kernels in between, the exported states are those of the same calls one at a time."""
import pytest
import torch

import paper_2609_12399_b200 as P

pytestmark = pytest.mark.gpu


def _prompt(gen, T, H, d, dtype):
    k = torch.randn((T, H, d), generator=gen, device="cuda")
    return ((k / k.norm(dim=-1, keepdim=True)).to(dtype), torch.randn((T, H, d), generator=gen, device="cuda").to(dtype),
            0.9 + 0.1 * torch.rand((T, H), generator=gen, device="cuda"), torch.sigmoid(torch.randn((T, H), generator=gen, device="cuda")))


@pytest.mark.parametrize("d,dtype,T", [(128, "bf16", 300), (64, "fp32", 130), (32, "bf16", 65)])
def test_captured_and_back_to_back(d, dtype, T):
    H, gen = 3, torch.Generator(device="cuda").manual_seed(d)
    td = torch.bfloat16 if dtype == "bf16" else torch.float32
    ctx = P.Onela(P.make_config(2, 2, H, d, d, 8, 1, dtype, dtype, 16))
    prompts = [_prompt(gen, T + 7 * i, H, d, td) for i in range(4)]
    want = []
    for i, p in enumerate(prompts):
        ctx.onela_prefill_shared_state(i >> 1, i & 1, *p)
        torch.cuda.synchronize()
        want.append(ctx.onela_export_shared_state(i >> 1, i & 1))
        torch.cuda.synchronize()

    def all_of(inputs):
        out = []
        for i, p in enumerate(inputs):
            ctx.onela_prefill_shared_state(i >> 1, i & 1, *p)
            out.append(ctx.onela_export_shared_state(i >> 1, i & 1))
        return out

    held = [tuple(torch.zeros_like(x) for x in p) for p in prompts]
    side = torch.cuda.Stream()
    side.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=side):
        got = all_of(held)
    for h, p in zip(held, prompts):
        for a, b in zip(h, p):
            a.copy_(b)
    graph.replay()
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    # inputs made by kernels right before the call, and overwritten right behind it
    for i, p in enumerate(prompts):
        for a, b in zip(held[i], p):
            torch.add(b, 0, out=a)
        ctx.onela_prefill_shared_state(i >> 1, i & 1, *held[i])
        for a in held[i]:
            a.zero_()
        got[i] = ctx.onela_export_shared_state(i >> 1, i & 1)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(got, want))
    assert ctx.onela_poll_device_status() == (0, 0)
