"""The gather queue of the warp-specialised kernel (chains that share too little to be staged): one older level, two, and
more than the eight whose slots a unit's lanes hold; several groups and heads per CTA and a single one; ragged widths; the
delta-record format.  Every call, every unit against the oracle."""
import pytest

import paper_2609_12399_b200 as P
from paper_2609_12399_b200 import inputs

from _cases import check_parity, make_case, run_library, run_oracle

pytestmark = pytest.mark.gpu

CFG1 = inputs.WORKLOADS[1]


@pytest.mark.parametrize("flags", [0, P.FLAG_GTR_DELTA])
@pytest.mark.parametrize("R,H,W,D", [(1, 1, 301, 11), (2, 3, 260, 4), (8, 20, 150, 3)])
def test_gather_queue(R, H, W, D, flags):
    wl = CFG1.scaled(R=R, L=1, H=H, W=W, D=D, prompt_len=16, parents="uniform", seed=5 + W)
    case = make_case(wl)
    ref, _ = run_oracle(case)
    outs, _, ctx = run_library(case, out_dtype="fp32", flags=flags, fused=True)
    check_parity(case, outs, ref)
    if not flags:
        outs, _, _ = run_library(case, out_dtype="bf16")
        check_parity(case, outs, ref)
    assert ctx.onela_poll_device_status() == (0, 0)
