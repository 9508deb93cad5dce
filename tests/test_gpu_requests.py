"""256 x 256 decode: where a call of all layers touches more than the L2 keeps, older records are requested a level ahead.  A context of
many layers takes that instantiation, one of a single layer the other; the same layer gives the same bits in both, within the bar of
the fp64 oracle, at chains on both sides of the eight levels whose slots the lanes hold."""
import numpy as np
import pytest
import torch

import paper_2609_12399_b200 as P
from paper_2609_12399_b200 import inputs

from _cases import check_parity, make_case, run_oracle

pytestmark = pytest.mark.gpu


def _run(case, layers, fused):
    wl = case["wl"]
    ctx = P.Onela(P.make_config(1, layers, wl.H, wl.dk, wl.dv, wl.W, wl.D, wl.dtype, wl.dtype, wl.W * wl.D))
    assert ctx.onela_uses_tensor_core_path() == 2
    ctx.onela_init_shared_state(0, 0, case["S0"][(0, 0)].cuda())
    outs = {}
    for t in range(wl.D):
        par = None if t == 0 else case["parents"][(0, t)][None].cuda()
        ctx.onela_reorder_beams(0, 1, par, wl.W)
        tok = [case["tok"][(0, 0, t)][n][None].cuda() for n in ("k", "v", "alpha", "beta")]
        q, out = case["q"][(0, 0, t)][None].cuda(), torch.empty((1, wl.W, wl.H, wl.dv), dtype=ctx.out_dtype, device="cuda")
        if fused:
            ctx.onela_append_decode_step(0, 1, 0, *tok, q, out)
        else:
            ctx.onela_append_records(0, 1, 0, *tok)
            ctx.onela_decode_step(0, 1, 0, q, out)
        outs[(0, 0, t)] = out[0].float().cpu()
    assert ctx.onela_poll_device_status() == (0, 0)
    return outs


# bytes of a call and layer: 2 heads x 128 KB, 45 beams x (q, k, v, record, output: 12 x 256 elements); the lines are 48 and 80 MB
@pytest.mark.parametrize("dtype,D,fused", [("bf16", 10, True), ("bf16", 4, False), ("fp32", 10, False), ("fp32", 4, True)])
def test_requests_change_nothing(dtype, D, fused):
    wl = inputs.WORKLOADS[1].scaled(H=2, dk=256, dv=256, W=45, D=D, dtype=dtype, prompt_len=16, parents="zipf", zipf_s=1.3, seed=D)
    case = make_case(wl)
    ref, _ = run_oracle(case)
    many, one = _run(case, 110, fused), _run(case, 1, fused)
    check_parity(case, many, ref)
    assert all(np.array_equal(many[key].numpy(), one[key].numpy()) for key in many)
