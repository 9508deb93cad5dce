"""The ancestry index kernel where it can go wrong: beams beyond one round of its 1024 threads, widths around its 32-beam
words and changing between calls, chains longer than one round of 32 levels.  Ancestry rows bit for bit against the oracle's
chains; the distinct-record index through the outputs of the decode that stages from it."""
import numpy as np
import pytest

from paper_2609_12399_b200 import inputs

from _cases import check_parity, expected_slots, make_case, run_library, run_oracle

pytestmark = pytest.mark.gpu

CFG1 = inputs.WORKLOADS[1]


@pytest.mark.parametrize("R,widths,law", [(2, [1, 31, 32, 33, 65], "uniform"), (1, [1500, 2049, 1025], "zipf"), (2, [5] * 36, "uniform"),
                                          (1, [40, 3, 70] * 12, "zipf")])
def test_index_widths_and_depths(R, widths, law):
    wl = CFG1.scaled(R=R, L=1, H=1, W=max(widths), D=len(widths), prompt_len=16, parents=law, zipf_s=1.3, seed=77)
    case = make_case(wl, widths=widths)
    ref, chains = run_oracle(case)
    outs, slots, ctx = run_library(case, fused=True)
    for key, want in expected_slots(case, chains).items():
        assert np.array_equal(slots[key], want), key
    check_parity(case, outs, ref)
    assert ctx.onela_poll_device_status() == (0, 0)
