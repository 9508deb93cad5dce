"""The warp-specialised kernel at the edges of its groups (64 beams, 32 with delta records): widths around one and two groups,
chains longer than the eight levels whose indices a unit's lanes hold, both gather modes (staged ancestors: Zipf parents; the
queue: uniform ones), grouped heads - against the fp64 oracle at the path's bar."""
import numpy as np
import pytest

import paper_2609_12399_b200 as P
from paper_2609_12399_b200 import inputs

from _cases import check_parity, expected_slots, make_case, run_library, run_oracle

pytestmark = pytest.mark.gpu

CFG1 = inputs.WORKLOADS[1]


def _check(wl, out_dtype, flags=0):
    case = make_case(wl)
    ref, chains = run_oracle(case)
    outs, slots, ctx = run_library(case, out_dtype=out_dtype, flags=flags, fused=True)
    assert ctx.onela_uses_tensor_core_path() == 1
    want = expected_slots(case, chains)
    for key in want:
        assert np.array_equal(slots[key], want[key]), f"ancestry rows of {key} differ"
    check_parity(case, outs, ref)
    assert ctx.onela_poll_device_status() == (0, 0)


@pytest.mark.parametrize("W", [7, 8, 9, 63, 64, 65, 128, 129])
@pytest.mark.parametrize("parents", ["uniform", "zipf"])
def test_widths_around_a_group(W, parents):
    _check(CFG1.scaled(R=2, H=3, W=W, D=4, prompt_len=32, parents=parents, zipf_s=1.5, seed=W), "bf16" if W % 2 else "fp32")


@pytest.mark.parametrize("W", [31, 32, 33, 65])
@pytest.mark.parametrize("out_dtype", ["bf16", "fp32"])
def test_delta_records_around_a_group(W, out_dtype):
    _check(CFG1.scaled(R=2, H=3, W=W, D=4, prompt_len=32, parents="zipf", zipf_s=1.3, seed=W), out_dtype, P.FLAG_GTR_DELTA)


@pytest.mark.parametrize("parents,D", [("uniform", 5), ("uniform", 6), ("uniform", 11), ("zipf", 11), ("zipf", 9)])
@pytest.mark.parametrize("flags", [0, P.FLAG_GTR_DELTA])
def test_chains_beyond_the_levels_held_in_lanes(parents, D, flags):
    _check(CFG1.scaled(R=1, H=2, W=150, D=D, prompt_len=32, parents=parents, zipf_s=1.3, seed=D), "fp32", flags)
