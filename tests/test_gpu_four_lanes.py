"""64 x 64 bf16 launches of more than one wave of tiles fold with four lanes per unit (delta records: where that takes fewer waves):
ragged tiles of 32 beams (16 with delta records), chains on both sides of the eight levels whose slots a unit's lanes hold, separate
append, grouped heads, both output types - every unit against the fp64 oracle at the path's bar, ancestry rows bit for bit.  The
launches on the other side of the lines take eight lanes.  Tiles are counted for a device of 148 SMs."""
import numpy as np
import pytest

import paper_2609_12399_b200 as P
from paper_2609_12399_b200 import inputs

from _cases import check_parity, expected_slots, make_case, run_library, run_oracle
from test_gpu_grouped import _run as run_grouped

pytestmark = pytest.mark.gpu

CFG1 = inputs.WORKLOADS[1]


def _check(wl, out_dtype, flags=0, fused=True):
    case = make_case(wl)
    ref, chains = run_oracle(case)
    outs, slots, ctx = run_library(case, out_dtype=out_dtype, flags=flags, fused=fused)
    assert ctx.onela_uses_tensor_core_path() == 2
    want = expected_slots(case, chains)
    for key in want:
        assert np.array_equal(slots[key], want[key]), f"ancestry rows of {key} differ"
    check_parity(case, outs, ref)
    assert ctx.onela_poll_device_status() == (0, 0)


# tiles of a launch: R x H x ceil(W / 32); the line is 740
@pytest.mark.parametrize("R,H,W,D,out_dtype,fused", [(12, 31, 33, 3, "bf16", True),       # 744, a tile of one beam
                                                     (10, 37, 64, 2, "fp32", True),       # 740: eight lanes
                                                     (13, 29, 63, 10, "fp32", True),      # 754, levels beyond the lanes'
                                                     (13, 29, 40, 5, "bf16", False)])
def test_raw_records(R, H, W, D, out_dtype, fused):
    _check(CFG1.scaled(R=R, H=H, dk=64, dv=64, W=W, D=D, prompt_len=8, parents="zipf", zipf_s=1.3, seed=R + W), out_dtype, fused=fused)


# tiles of 16 beams: 744 are two waves either way (eight lanes, 592 a wave), 640 one of four lanes' (740), 1200 two against three
@pytest.mark.parametrize("R,H,W,D,out_dtype", [(12, 31, 17, 4, "bf16"), (12, 31, 32, 10, "fp32"), (10, 32, 17, 10, "bf16"), (8, 16, 75, 4, "fp32"),
                                               (15, 40, 19, 3, "bf16")])
def test_delta_records(R, H, W, D, out_dtype):
    _check(CFG1.scaled(R=R, H=H, dk=64, dv=64, W=W, D=D, prompt_len=8, seed=R + W), out_dtype, P.FLAG_GTR_DELTA)


@pytest.mark.parametrize("g,R,H,W,D,out_dtype,fused", [(2, 6, 64, 33, 10, "bf16", True), (4, 3, 128, 40, 9, "fp32", False), (2, 4, 62, 97, 3, "bf16", False),
                                                       (4, 5, 80, 60, 3, "bf16", True)])      # 768, 768, 992, 800 tiles
def test_grouped_heads(g, R, H, W, D, out_dtype, fused):
    """H value heads over H / g key heads: split key and value planes, the key stored by the first value head of its group."""
    _, ctx, _ = run_grouped(CFG1.scaled(R=R, L=1, H=H, dk=64, dv=64, W=W, D=D, prompt_len=8, parents="zipf", zipf_s=1.3, seed=R * W), g, out_dtype, fused)
    assert ctx.onela_uses_tensor_core_path() == 2


@pytest.mark.parametrize("R,H,W,D,out_dtype,flags", [(12, 31, 33, 10, "fp32", 0), (12, 31, 33, 3, "bf16", 0), (10, 32, 17, 10, "fp32", P.FLAG_GTR_DELTA)])
def test_results_do_not_depend_on_the_other_requests_of_a_call(R, H, W, D, out_dtype, flags):
    """Ten or twelve requests in one call (744 tiles, 640 with delta records: four lanes) and the same requests one by one (62, 64:
    eight), bit for bit."""
    case = make_case(CFG1.scaled(R=R, H=H, dk=64, dv=64, W=W, D=D, prompt_len=8, parents="zipf", zipf_s=1.3, seed=W + D))
    outs, _, _ = run_library(case, out_dtype=out_dtype, flags=flags, fused=True)
    alone, _, _ = run_library(case, out_dtype=out_dtype, flags=flags, fused=True, batched=False)
    assert all(np.array_equal(outs[key].numpy(), alone[key].numpy()) for key in outs)
