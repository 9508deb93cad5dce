"""32 x 32 heads: chains shorter and longer than a unit's lanes (8 with fp32 records, 4 with bf16), one beam, a tile and one
more than a tile; append fused and separate.  Every call, every unit against the oracle."""
import pytest

from paper_2609_12399_b200 import inputs

from _cases import check_parity, make_case, run_library, run_oracle

pytestmark = pytest.mark.gpu

CFG0 = inputs.WORKLOADS[0]


@pytest.mark.parametrize("dtype", ["fp32", "bf16"])
@pytest.mark.parametrize("R,H,W,D", [(1, 1, 1, 11), (2, 3, 32, 6), (3, 2, 33, 10)])
def test_small_heads(R, H, W, D, dtype):
    wl = CFG0.scaled(R=R, L=1, H=H, W=W, D=D, dtype=dtype, prompt_len=16, parents="uniform", seed=9 + W)
    case = make_case(wl)
    ref, _ = run_oracle(case)
    for fused in (True, False):
        outs, _, ctx = run_library(case, out_dtype="fp32", fused=fused)
        check_parity(case, outs, ref, bar=5e-6)     # fp32 throughout: records are exact, a chain of 11 adds 11 x 2^-22 or so
        assert ctx.onela_poll_device_status() == (0, 0)
