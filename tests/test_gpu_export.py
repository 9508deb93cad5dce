"""onela_export_shared_state: the states come back bit for bit, by the library's own kernel (one step and several of its grid) and,
where the destination is not the device's own memory, by the runtime's copy."""
import ctypes

import pytest
import torch

import paper_2609_12399_b200 as P

pytestmark = pytest.mark.gpu


def _stored(H, d):
    S = torch.randn((1, 2, H, d, d), generator=torch.Generator().manual_seed(H + d)).cuda()
    ctx = P.Onela(P.make_config(1, 2, H, d, d, 8, 1, "bf16", "bf16", 8))
    ctx.onela_init_shared_states(0, 1, S)
    return S, ctx


@pytest.mark.parametrize("H,d", [(1, 32), (3, 64), (75, 128)])       # 256 float4, 3072, 307 200 (more than one step of 1184 x 256)
def test_exported_states(H, d):
    S, ctx = _stored(H, d)
    for layer in range(2):
        assert torch.equal(ctx.onela_export_shared_state(0, layer), S[0, layer])


def test_export_to_managed_memory():
    S, ctx = _stored(3, 64)
    cudart = ctypes.CDLL("libcudart.so.12")
    p, n = ctypes.c_void_p(), S[0, 0].numel()
    assert cudart.cudaMallocManaged(ctypes.byref(p), ctypes.c_size_t(4 * n), ctypes.c_uint(1)) == 0
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    for layer in range(2):
        assert ctx.lib.onela_export_shared_state(ctx.handle, 0, layer, p, stream) == 0
        torch.cuda.synchronize()
        got = torch.frombuffer((ctypes.c_float * n).from_address(p.value), dtype=torch.float32).clone()
        assert torch.equal(got, S[0, layer].cpu().flatten())
    assert cudart.cudaFree(p) == 0
