// Shared-state store and record arena kernels.
//  - append: copy one decode call's (k, v, alpha, beta) into the append-only arena (paper Section 3.3:
//    records are written once to the slots of the current step and never relocated).
//  - store_state: fill the store slot of one (request, layer) with S_0 (Section 3.2: the post-prefill state is
//    stored once per request) from a caller tensor.
#include <cuda_fp16.h>

#include <algorithm>

#include "onela_internal.h"
#include "onela_layout.cuh"

namespace onela {

namespace {

// One warp per (beam, head) row of one request (blockIdx.y).  The arena is head-major ([head][slot][k | v])
// so that the records one decode tile reads - consecutive beams of one head - are contiguous.
__global__ void __launch_bounds__(256) append_kernel(const char* __restrict__ k, const char* __restrict__ v,
                                                     const float* __restrict__ alpha, const float* __restrict__ beta,
                                                     char* __restrict__ kv_plane, float2* __restrict__ gate_plane,
                                                     long long arena_slots, int32_t W, int32_t H, int32_t k_bytes,
                                                     int32_t v_bytes, BatchBases bases) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const int r = blockIdx.y;
    const int row_in_req = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);   // b * H + h
    const int lane = threadIdx.x & 31;
    if (row_in_req >= W * H) return;
    const int b = row_in_req / H, h = row_in_req - b * H;
    const long long row = (long long)r * (W * H) + row_in_req;
    const long long dst_row = (long long)h * arena_slots + (bases.base[r] + b);
    const uint4* ksrc = reinterpret_cast<const uint4*>(k + row * k_bytes);
    const uint4* vsrc = reinterpret_cast<const uint4*>(v + row * v_bytes);
    uint4* dst = reinterpret_cast<uint4*>(kv_plane + dst_row * (k_bytes + v_bytes));
    const int nk = k_bytes >> 4, nv = v_bytes >> 4;
    for (int c = lane; c < nk + nv; c += 32) dst[c] = (c < nk) ? __ldg(ksrc + c) : __ldg(vsrc + (c - nk));
    if (lane == 0) gate_plane[dst_row] = make_float2(__ldg(alpha + row), __ldg(beta + row));
}

// Copy of one (request, layer)'s states out of the store, 16 bytes per thread and step (a prefill has just left them in L2: the
// launch is what it costs, and the code: with a 64-bit index, which the compiler unrolls, 9 prefills of 100 tokens took 220 us, not 213).
// n: at most 2^32 - EXPORT_STEP, so that the index does not wrap in the step beyond the end.
constexpr uint32_t EXPORT_BLOCKS = 1184, EXPORT_STEP = EXPORT_BLOCKS * 256;      // eight CTAs per SM at most
__global__ void __launch_bounds__(256) export_state_kernel(const float4* __restrict__ slot, float4* __restrict__ out, uint32_t n) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (uint32_t i = blockIdx.x * 256 + threadIdx.x; i < n; i += gridDim.x * 256) out[i] = slot[i];
}

// The operand scale of a head (Layout::s0_scale) from the largest magnitude of its state.
__device__ __forceinline__ float operand_scale(float peak) {
    const int eb = (int)(__float_as_uint(peak) >> 23) & 255;          // biased exponent of a non-negative number
    constexpr int target = 11;                                         // scaled peak in [2^11, 2^12)
    const bool ok = eb > target + 1 && eb < 255;
    return ok ? __uint_as_float((uint32_t)(254 + target - eb) << 23) : 1.f;
}
// Copy of the caller's states into the store, with every head's operand scale and - configurations of the tiled
// tensor-core kernel - its operand copy (see Layout::s0_f16) from the same registers.  A CTA holds 16 384 elements (64 KB,
// all of its loads in flight at once); a larger head is a cluster of up to eight CTAs that exchange their largest
// magnitudes through distributed shared memory.  HBM-bound: one read, one write, half a write more with the operand copy.
// (As a CTA of 256 threads per head walking its state, followed by a second kernel that read the store back, 256 heads of
// 256 x 256 took 43 + 27 us; 31 us now.)
// VP: groups of eight elements per thread.
template <int VP, int THREADS>
__global__ void __launch_bounds__(THREADS) store_state_kernel(const float* __restrict__ in, float* __restrict__ out, float* __restrict__ scale_out,
                                                              uint16_t* __restrict__ f16_out, int32_t dk, int32_t dv) {
    __shared__ float part[32];
    __shared__ float cta_peak;
    const int tid = threadIdx.x;
    const uint32_t parts = gridDim.x, head = blockIdx.y, rank = blockIdx.x;      // cluster = the CTAs of one head
    const long long base = (long long)head * dk * dv + (long long)rank * (VP * THREADS * 8);
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    float4 x[VP][2];
#pragma unroll
    for (int j = 0; j < VP; ++j) {
        const float4* p = reinterpret_cast<const float4*>(in + base) + 2 * (j * THREADS + tid);
        x[j][0] = __ldg(p);
        x[j][1] = __ldg(p + 1);
    }
    float peak = 0.f;
#pragma unroll
    for (int j = 0; j < VP; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            reinterpret_cast<float4*>(out + base)[2 * (j * THREADS + tid) + e] = x[j][e];
            peak = fmaxf(fmaxf(peak, fmaxf(fabsf(x[j][e].x), fabsf(x[j][e].y))), fmaxf(fabsf(x[j][e].z), fabsf(x[j][e].w)));
        }
    for (int o = 16; o > 0; o >>= 1) peak = fmaxf(peak, __shfl_xor_sync(0xffffffffu, peak, o));
    if ((tid & 31) == 0) part[tid >> 5] = peak;
    __syncthreads();
    peak = 0.f;
#pragma unroll
    for (int w = 0; w < THREADS / 32; ++w) peak = fmaxf(peak, part[w]);
    if (parts > 1) {
        if (tid == 0) cta_peak = peak;
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
        for (uint32_t p = 0; p < parts; ++p) {
            uint32_t at;
            float other;
            asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(at) : "r"((uint32_t)__cvta_generic_to_shared(&cta_peak)), "r"(p));
            asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(other) : "r"(at) : "memory");
            peak = fmaxf(peak, other);
        }
        asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");      // nobody leaves while its peak is read
    }
    const float sc = operand_scale(peak);
    if (rank == 0 && tid == 0) scale_out[head] = sc;
    if (!f16_out) return;
    // value rows padded to a multiple of 128, tiles of 128 rows x 64 columns, 16-byte chunks swizzled by the row
    const int cpr = dk / 8, kb_n = dk / 64, rows = (dv + 127) / 128 * 128;
    char* dst = reinterpret_cast<char*>(f16_out) + (long long)head * rows * dk * 2;
    auto at = [&](int i, int ch) { return dst + ((long long)((i >> 7) * kb_n + (ch >> 3)) * 128 + (i & 127)) * 128 + (((ch & 7) ^ (i & 7)) << 4); };
    const int first = (int)rank * (VP * THREADS);           // the CTA's first chunk of eight elements
#pragma unroll
    for (int j = 0; j < VP; ++j) {
        const int item = first + j * THREADS + tid, i = item / cpr;
        const __half2 h0 = __floats2half2_rn(x[j][0].x * sc, x[j][0].y * sc), h1 = __floats2half2_rn(x[j][0].z * sc, x[j][0].w * sc);
        const __half2 h2 = __floats2half2_rn(x[j][1].x * sc, x[j][1].y * sc), h3 = __floats2half2_rn(x[j][1].z * sc, x[j][1].w * sc);
        *reinterpret_cast<uint4*>(at(i, item - i * cpr)) =
            make_uint4(*reinterpret_cast<const uint32_t*>(&h0), *reinterpret_cast<const uint32_t*>(&h1), *reinterpret_cast<const uint32_t*>(&h2),
                       *reinterpret_cast<const uint32_t*>(&h3));
    }
    for (int item = dv * cpr + tid; item < rows * cpr; item += THREADS) {        // padding (dv = 64: one CTA per head)
        const int i = item / cpr;
        *reinterpret_cast<uint4*>(at(i, item - i * cpr)) = make_uint4(0u, 0u, 0u, 0u);
    }
}

template <int VP, int THREADS>
cudaError_t launch_store_t(const float* in, float* out, float* scale_out, uint16_t* f16_out, unsigned parts, unsigned n_heads, int32_t dk, int32_t dv,
                           cudaStream_t stream) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(parts, n_heads);
    cfg.blockDim = dim3(THREADS);
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = parts;
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = parts > 1 ? 2 : 1;
    return cudaLaunchKernelEx(&cfg, store_state_kernel<VP, THREADS>, in, out, scale_out, f16_out, dk, dv);
}

}  // namespace

cudaError_t launch_append(const void* k, const void* v, const float* alpha, const float* beta, char* kv_plane,
                          float2* gate_plane, long long arena_slots, int32_t req_count, int32_t W, int32_t H,
                          int32_t dk, int32_t dv, int32_t elem_bytes, const BatchBases& bases,
                          cudaStream_t stream) {
    const int warps_per_block = 8;
    dim3 grid((unsigned)((W * H + warps_per_block - 1) / warps_per_block), (unsigned)req_count);
    return launch_dependent(append_kernel, grid, dim3(warps_per_block * 32), 0, stream, static_cast<const char*>(k), static_cast<const char*>(v), alpha,
                            beta, kv_plane, gate_plane, arena_slots, W, H, dk * elem_bytes, dv * elem_bytes, bases);
}

cudaError_t launch_store_state(const float* S0_in, float* slot, float* scale_out, uint16_t* f16_out, long long n_heads, int32_t dk, int32_t dv,
                               cudaStream_t stream) {
    const int elems = dk * dv;             // every supported head is 1024 or 4096 elements, or a power of two times 16 384
    for (long long h0 = 0; h0 < n_heads; h0 += 65535) {
        const unsigned n = (unsigned)(n_heads - h0 < 65535 ? n_heads - h0 : 65535);
        const float* in = S0_in + h0 * elems;
        float *out = slot + h0 * elems, *sc = scale_out + h0;
        uint16_t* f16 = f16_out ? f16_out + h0 * (long long)(s0_f16_head_bytes(dk, dv) / 2) : nullptr;
        const cudaError_t e = elems == 1024   ? launch_store_t<1, 128>(in, out, sc, f16, 1, n, dk, dv, stream)
                              : elems == 4096 ? launch_store_t<2, 256>(in, out, sc, f16, 1, n, dk, dv, stream)
                              : elems % 16384 == 0 && elems / 16384 <= 8
                                  ? launch_store_t<4, 512>(in, out, sc, f16, (unsigned)(elems / 16384), n, dk, dv, stream)
                                  : cudaErrorInvalidValue;
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_export_state(const float* slot, float* S0_out, int32_t H, int32_t dk, int32_t dv, cudaStream_t stream) {
    // A kernel of our own is a dependent launch, a copy by the runtime is not.  (Together with the prefill's own dependent
    // launch, us a pass of prefill + export: 3 x 100 tokens x 32 heads of 64 x 64 bf16 62 -> 45, 2 x 1021 tokens x 16 heads
    // fp32 82 -> 74.5, 3 x 900 tokens x 16 heads of 128 x 128 160 -> 147, 16 384 tokens 450 -> 445.)  Where the store or the destination
    // is not the current device's own memory (another device's, managed, the host's), which a kernel may not reach, and where the
    // stream is another device's, which takes no kernel from here, the copy is the runtime's.
    cudaPointerAttributes at;
    int dev = 0;
    auto here = [&](const void* p) { return cudaPointerGetAttributes(&at, p) == cudaSuccess && at.type == cudaMemoryTypeDevice && at.device == dev; };
    const long long n = (long long)H * dk * dv / 4;
    if (n <= 0xffffffffll - EXPORT_STEP && cudaGetDevice(&dev) == cudaSuccess && here(S0_out) && here(slot)) {
        const unsigned blocks = (unsigned)std::min<long long>((n + 255) / 256, EXPORT_BLOCKS);
        const cudaError_t e = launch_dependent(export_state_kernel, dim3(blocks), dim3(256), 0, stream, reinterpret_cast<const float4*>(slot),
                                               reinterpret_cast<float4*>(S0_out), (uint32_t)n);
        if (e != cudaErrorInvalidResourceHandle) return e;
        cudaGetLastError();
    }
    return cudaMemcpyAsync(S0_out, slot, (size_t)H * dk * dv * sizeof(float), cudaMemcpyDeviceToDevice, stream);
}

}  // namespace onela
