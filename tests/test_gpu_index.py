"""The ancestry index kernel where it can go wrong: beams beyond one round of its 1024 threads, widths around its 32-beam
words and changing between calls, chains longer than one round of 32 levels.  Ancestry rows bit for bit against the oracle's
chains; the distinct-record index through the outputs of the decode that stages from it."""
import numpy as np
import pytest
import torch

import paper_2609_12399_b200 as P
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


@pytest.mark.parametrize("max_beam,calls", [(16384, 14), (6144, 34), (12288, 18), (200000, 3)])
def test_index_rounds_that_fill_shared_memory(max_beam, calls):
    """Bitmaps of a round of levels that come out at the 48 KB a launch gets without asking (12 levels of 4 KB, 32 of 1.5 KB,
    16 of 3 KB: the kernel's own static shared memory must fit beside them), and one level's beyond it."""
    W = 8
    ctx = P.Onela(P.make_config(1, 1, 1, 128, 128, max_beam, calls, "bf16", "fp32", W * calls))
    assert ctx.onela_uses_tensor_core_path() == 1      # (the kernel whose staging the bitmaps are for)
    ctx.onela_init_shared_state(0, 0, torch.zeros(1, 128, 128, device="cuda"))
    kv, gate = torch.zeros(1, W, 1, 128, dtype=torch.bfloat16, device="cuda"), torch.ones(1, W, 1, device="cuda")
    rng, chains = np.random.default_rng(max_beam), np.zeros((W, 0), np.int64)
    for t in range(calls):
        par = rng.integers(0, W, W)
        ctx.onela_reorder_beams(0, 1, torch.from_numpy(par.astype(np.int32))[None].cuda() if t else None, W)
        ctx.onela_append_records(0, 1, 0, kv, kv, gate, gate)
        chains = np.concatenate([chains[par] if t else chains, t * W + np.arange(W)[:, None]], axis=1)
        assert np.array_equal(ctx.onela_export_chains(0).cpu().numpy(), chains), t
    assert ctx.onela_poll_device_status() == (0, 0)
