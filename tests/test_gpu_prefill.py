"""onela_prefill_shared_state against the fp64 oracle's prefill: prompt lengths around the 64-token chunks and around the
cuts into segments (few heads: up to eight segments per head, each folded onto the one before), every head width and
record dtype, gates at their ends (alpha = 0, alpha = 1, beta = 0), scales far from one, and the operand copy of the
tiled decode kernel through a decode call."""
import numpy as np
import pytest
import torch

import oracle
import paper_2609_12399_b200 as P
from paper_2609_12399_b200 import inputs

from _cases import REL_L2_BAR, rel_l2

pytestmark = pytest.mark.gpu

# fp32 sums of up to 64 products per chunk over a forgetting horizon of some tens of tokens: a few 2^-22
BAR = 2e-6


def _check(p, d, dtype, bar=BAR):
    H = p["k"].shape[1]
    ctx = P.Onela(P.make_config(1, 1, H, d, d, 8, 2, dtype, "fp32", 16))
    ctx.onela_prefill_shared_state(0, 0, *(p[n].cuda() for n in ("k", "v", "alpha", "beta")))
    got = ctx.onela_export_shared_state(0, 0).cpu().double().numpy()
    assert ctx.onela_poll_device_status() == (0, 0)
    want = oracle.prefill(p["k"], p["v"], p["alpha"], p["beta"])
    err = np.linalg.norm(got - want, axis=(1, 2)) / np.linalg.norm(want, axis=(1, 2))
    assert err.max() < bar, (d, dtype, p["k"].shape, err)
    return ctx


def _prompt(d, dtype, H, T, seed=7):
    wl = inputs.WORKLOADS[1].scaled(H=H, dk=d, dv=d, dtype=dtype, prompt_len=T, seed=seed)
    return inputs.prompt_tokens(wl, 0, 0)


@pytest.mark.parametrize("d,dtype", [(32, "fp32"), (32, "bf16"), (64, "fp32"), (64, "bf16"), (128, "fp32"), (128, "bf16")])
@pytest.mark.parametrize("T", [1, 63, 64, 65, 129, 577, 1021])
def test_prefill_lengths_and_head_widths(d, dtype, T):
    _check(_prompt(d, dtype, 3, T), d, dtype)


@pytest.mark.parametrize("H,T", [(1, 4200), (40, 1500), (160, 200)])
def test_prefill_head_counts(H, T):
    """One head on a full cluster; more CTAs than fit at once; more heads than SMs."""
    _check(_prompt(128, "bf16", H, T), 128, "bf16")


@pytest.mark.parametrize("d,dtype", [(64, "fp32"), (128, "bf16"), (128, "fp32")])
def test_prefill_gates_at_their_ends_and_scales(d, dtype):
    T, H = 700, 3
    p = _prompt(d, dtype, H, T, seed=11)
    p["alpha"][::97] = 0.0            # forget everything
    p["alpha"][5:300:7] = 1.0
    p["beta"][3::11] = 0.0
    _check(p, d, dtype)
    p = _prompt(d, dtype, H, T, seed=12)
    p["alpha"][:] = 1.0               # nothing decays: the delta rule alone forgets, over some 2 d tokens
    _check(p, d, dtype, bar=5 * BAR)
    p = _prompt(d, dtype, H, T, seed=13)
    p["v"] = (p["v"].double() * torch.tensor([1e-12, 1.0, 3e9])[None, :, None]).to(p["v"].dtype)
    _check(p, d, dtype)
    p = _prompt(d, dtype, H, T, seed=14)
    scale = torch.tensor([1e-4, 2.0 ** -12, 1.3])           # short keys; keys longer than one, with beta small enough to contract
    p["k"] = (p["k"].double() * scale[None, :, None]).to(p["k"].dtype)
    _check(p, d, dtype, bar=5 * BAR)


@pytest.mark.parametrize("d,dtype", [(32, "fp32"), (32, "bf16"), (64, "fp32"), (64, "bf16"), (128, "fp32"), (128, "bf16")])
@pytest.mark.parametrize("T", [40, 1021])
def test_prefill_is_as_exact_as_the_recurrence_in_fp32(d, dtype, T):
    """Root mean square over the heads of the error against 64 bits, beside that of Eq. 1 token by token in fp32 on the same
    inputs: no larger, but for what a sample of 16 states of d x d elements scatters (a tenth at the smallest head)."""
    H = 16
    p = _prompt(d, dtype, H, T, seed=21)
    ctx = P.Onela(P.make_config(1, 1, H, d, d, 8, 1, dtype, "fp32", 16))
    ctx.onela_prefill_shared_state(0, 0, *(p[n].cuda() for n in ("k", "v", "alpha", "beta")))
    got = ctx.onela_export_shared_state(0, 0).cpu().double().numpy()
    k, v = p["k"].float(), p["v"].float()
    S = torch.zeros((H, d, d))
    for t in range(T):
        a, b = p["alpha"][t][:, None], p["beta"][t][:, None]
        delta = b * (v[t] - a * torch.bmm(S, k[t][:, :, None])[:, :, 0])
        S = a[:, :, None] * S + delta[:, :, None] * k[t][:, None, :]
    want = oracle.prefill(p["k"], p["v"], p["alpha"], p["beta"])
    def error(x):
        return float(np.sqrt(np.mean((np.linalg.norm(x - want, axis=(1, 2)) / np.linalg.norm(want, axis=(1, 2))) ** 2)))
    assert error(got) <= 1.1 * error(S.double().numpy()), (error(got), error(S.double().numpy()))


@pytest.mark.parametrize("d,dtype", [(64, "bf16"), (64, "fp32"), (128, "fp32")])
def test_prefilled_state_decodes_on_the_tiled_kernel(d, dtype):
    H, W = 2, 40
    p = _prompt(d, dtype, H, 333)
    ctx = _check(p, d, dtype)
    wl = inputs.WORKLOADS[1].scaled(H=H, dk=d, dv=d, dtype=dtype, W=8, seed=3)
    tok, q = inputs.decode_token(wl, 0, 0, 0), inputs.decode_query(wl, 0, 0, 0)
    out = torch.empty((1, 8, H, d), device="cuda")
    ctx.onela_reorder_beams(0, 1, None, 8)
    ctx.onela_append_decode_step(0, 1, 0, *(tok[n][None].cuda() for n in ("k", "v", "alpha", "beta")), q[None].cuda(), out)
    S = torch.from_numpy(oracle.prefill(p["k"], p["v"], p["alpha"], p["beta"]).astype(np.float32))
    ref = oracle.decode(S, [tok], [None], q)
    assert rel_l2(out[0].cpu().numpy(), ref).max() <= REL_L2_BAR
