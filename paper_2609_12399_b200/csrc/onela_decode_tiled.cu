// Tiled tcgen05 decode kernel for B200 (sm_100a): the shapes the warp-specialised kernel does not take - key widths
// 64 and 256, value widths 64 to 512, fp32 records at every width, grouped value heads or not (the operator suite of
// Section 4.1).  The chain walk is the CUDA-core one (see onela_decode_generic.cu); what moves to the tensor cores is
// the contraction with S_0, which dominates these shapes (dv x dk multiply-adds per unit against 3 dk per record).
//
// One CTA = (request, value head, tile of 32 beams - 64 from 128 x 128 up), 8 lanes per (beam, head) unit (4 in large launches of
// 64 x 64 bf16: see four_lanes).
//   1. Every unit folds its query through its records, newest first:  c = k.r ; corr += beta c v ; r -= beta c k,
//      the decay a running scalar.  corr stays in registers.  With the append fused in, the newest record comes from
//      the caller's tensors and the unit also writes it to its arena slot.
//   2. The folded queries go to shared memory as rows of the MMA's B operand: fp16, K-major, 128-byte swizzle, each row
//      times the power of two that brings its largest element into [2^8, 2^9) (exact; undone after the product).
//   3. Per tile of 128 value rows the A operand (the state's stored fp16 copy, by bulk copies) meets the rows: dk / 16 MMAs
//      (M = 128, N = beams, K = 16) accumulate S_0 . r~ in tensor memory; the accumulators go through a shared-memory tile
//      (lane = value row in, a beam's row out) to the units' lanes, which undo the scales, add corr from their registers
//      and store 16-byte vectors.  Where there is room two A operands and two accumulators alternate.
// What bounds it: the phases of a CTA in sequence (inputs from HBM, dependent gathers, MMAs, accumulators through shared
// memory), overlapped only by the other CTAs of the SM - one at the widest shapes.  us per launch on the beam-512 stack
// before / after corr was left in registers, the MMAs issued by an elected lane of a converged warp and the loads moved ahead
// of the first barrier: 64 x 64 bf16 29.8 / 24.0 (depth 1 - 8; 23.4 since with four lanes), 256 x 256 bf16 79.9 / 70.9 (68 since with requests a level ahead), 256 x 512 bf16 (600 beams x 16
// heads) 36.6 / 32.0, 128 x 256 fp32 23.5 / 21.5.  Requests of the next wave's inputs into L2 made it 3 % slower, of all older
// records ahead of the fold at 64 x 64 8 - 13 % (other CTAs hide them, the instructions are paid); a persistent
// loop over the tiles of beams spills (the invariants of every pointer stay live): 64 x 64 40 us.
// The only wait is for the MMAs' completion; it is bounded, and all threads agree on its outcome before going on
// (ONELA_E_TIMEOUT in the status word otherwise).
#include <atomic>
#include <mutex>

#include "onela_internal.h"
#include "onela_layout.cuh"
#include "onela_sm100.cuh"

namespace onela {

namespace {

using sm100::bulk_load;
using sm100::idesc_f16;
using sm100::mbar_expect_tx;
using sm100::mbar_init;
using sm100::mbar_wait;
using sm100::mma_commit;
using sm100::mma_ss;
using sm100::pack_f16x2;
using sm100::pow2_scale;
using sm100::smem_u32;
using sm100::tmem_ld16;
using sm100::umma_desc;

// pitch (floats) of the output tile: conflict-free for both access patterns
template <int VD>
__host__ __device__ constexpr int tile_pitch() { return (VD < 128 ? VD : 128) + 4; }
constexpr int ROW_TARGET = 8;          // a scaled operand row's largest element lies in [2^8, 2^9)

// Beams per CTA (= MMA N; 8 threads each).  Key width 256 takes 64: every CTA turns the whole head's S_0 into its A
// operand, 128 KB of fp32 from L2 per tile of value rows, and at 32 beams per CTA those reads (1 GB per launch at
// 256 x 512 with 65 536 units) were what bounded the kernel; one CTA of 512 threads holds as many warps as two of 256.
template <int KD, int VD>
__host__ __device__ constexpr int tiled_beams() { return KD * VD >= 128 * 128 ? 64 : 32; }
#ifdef ONELA_TEST_HOOKS
// Test-hooks build only (a second library that the product never loads): when set, CTA (0, 0, 0) leaves out its first
// tile's MMAs and their commit, so that the wait for them runs out.
__device__ int g_hook_tiled_skip_issue;
#endif

template <int KD, int VD>
__host__ __device__ constexpr size_t tiled_smem_bytes() {
    // two A operands where there is a next tile to prepare and the key is narrow (at key width 256 the second buffer
    // leaves the fold's record loads 34 KB of L1: 89 -> 106 us at 256 x 256)
    constexpr int NB = tiled_beams<KD, VD>(), ABUF = (VD > 128 && KD <= 128) ? 2 : 1;
    return 1024 + (size_t)ABUF * (KD / 64) * 128 * 128 + (size_t)(KD / 64) * NB * 128 + (size_t)NB * tile_pitch<VD>() * 4 + 64;
}

// CTAs per SM the registers are capped for: small CTAs are latency-bound (a string of dependent loads per level, one MMA
// round trip), so the narrowest shape gets four, with bf16 records - half the registers - five (64 x 64 on the beam-512
// stack: 30 -> 27 us; six: 28.5; fp32 records, five: 16 -> 17 us, three: 4 - 7 % slower at 65 536 units), unless a beam has two
// rows, where five of eight lanes spill (4 x 300 beams x 16 heads, 6 calls, a generation: 185 -> 177 us; four lanes: see four_lanes).  (64 beams of 256 threads at two per
// SM, or 16 lanes per unit, were 5 - 10 % slower at 256 x 256.)
template <int KD, int VD, typename T, bool DELTA, int G>
__host__ __device__ constexpr int tiled_min_ctas() { return KD + VD <= 128 ? (G == 4 ? (DELTA ? 5 : 6) : sizeof(T) == 4 || DELTA ? 4 : 5) : tiled_beams<KD, VD>() == 64 ? 1 : 2; }

// DELTA: the arena keeps (alpha_t, delta_t, k_t) (Section 3.2, Eq. 2-4).  A beam owns TWO rows of the tile - its query
// and its own key, both projected through the parent state: S_{t-1} x = D S_0 x + sum_j d_j (k_j . x) delta_j, the
// replay leaving x unchanged - and after the contraction delta_t = beta_t (v_t - alpha_t S_{t-1} k_t) and
// o_t = alpha_t S_{t-1} q_t + delta_t (k_t . q_t) are formed from the two rows and the record is written; always with
// the append fused in, dk = dv <= 128.
// REQUEST: an older record's lines are requested into L2 a level ahead (see launch_one).  G: lanes per unit, 8 or (64 x 64 bf16 in large launches) 4.  Four lanes add up what eight do, in eight lanes' order: lane g holds
// the chunks of lanes g and g + 4, sums each by itself and adds the two, which is what the first exchange among eight lanes does.  So
// a request's results do not depend on how many others share its launch.
template <int KD, int VD, typename T, typename OutT, bool DELTA, int G, bool REQUEST>
__global__ void __launch_bounds__(tiled_beams<KD, VD>() * G, tiled_min_ctas<KD, VD, T, DELTA, G>()) decode_tiled_kernel(const TiledArgs a) {
    constexpr int NB = tiled_beams<KD, VD>(), CP = tile_pitch<VD>();
    constexpr int THREADS = NB * G, BPT = DELTA ? NB / 2 : NB;          // beams per tile
    static_assert(G == 8 || G == 4, "lanes per unit");
    static_assert(!DELTA || (KD == VD && VD <= 128), "delta records: square heads, one tile of value rows");
    constexpr uint32_t ACC_COLS = 2 * NB;      // two accumulators of NB columns (a power of two >= 32)
    constexpr int VEC = Vec16<T>::N;
    constexpr int CK = KD / (G * VEC), CV = VD / (G * VEC);   // 16-byte chunks per lane
    static_assert(KD % 64 == 0 && VD % 64 == 0 && CK >= 1 && CV >= 1, "whole 64-element K blocks, whole chunks per lane");
    static_assert(128 % (G * VEC) == 0, "a lane's chunk lies inside one tile of 128 value rows");
    constexpr int KB = KD / 64;                   // K blocks of 64 fp16 (one 128-byte swizzled row each)
    constexpr int MT = (VD + 127) / 128;          // tiles of 128 value rows
    constexpr int A_KB = 128 * 128, R_KB = NB * 128;   // bytes of one K block of the two operands

    extern __shared__ uint8_t smem_raw[];
    const uint32_t raw = smem_u32(smem_raw);
    uint8_t* smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);      // swizzle atoms need 1024-byte alignment
    constexpr int ABUF = (MT > 1 && KD <= 128) ? 2 : 1;
    uint8_t* A_s = smem;                                               // [ABUF][KB][128 rows][128 bytes]: tile mt in buffer mt & 1
    uint8_t* R_s = A_s + ABUF * KB * A_KB;                             // [KB][NB rows][128 bytes]
    float* C_s = reinterpret_cast<float*>(R_s + KB * R_KB);            // [NB][CP]
    uint64_t* bar = reinterpret_cast<uint64_t*>(C_s + NB * CP);        // a tile's MMAs complete
    uint64_t* abar = bar + 1;                                          // [2] an A operand has landed
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(abar + 2);

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;   // (warp: uniform for the compiler too)
    if (tid == 0) {
        mbar_init(smem_u32(bar), 1);
        mbar_init(smem_u32(abar), 1);
        mbar_init(smem_u32(abar + 1), 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(ACC_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    // (barriers and tensor memory are first used by others than the threads above after the barrier that ends the fold: no
    // barrier stands between a CTA's start and its first loads)
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    // (programmatic dependent launch: the next launch may set itself up under this one)
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    const int tile = blockIdx.x, hv = blockIdx.y, req = blockIdx.z;
    const int hk = hv / a.g, Hv = a.Hk * a.g;
    const int grp = tid / G, g = tid % G;
    const int b = tile * BPT + (DELTA ? grp >> 1 : grp);
    const bool key_row = DELTA && (grp & 1);          // DELTA: the odd row of a beam projects its key
    const bool active = b < a.W;
    const int bb = active ? b : a.W - 1;  // idle units shadow a live beam so loads and shuffles stay uniform

    const float sc0 = __ldg(a.s0_scale + req * a.s0_scale_req_stride + hv);     // a power of two
    // The A operand of tile mt (S_0 rows [128 mt, 128 mt + 128), rows beyond dv zero): the store keeps every state as
    // this kernel's operand as well - fp16, times the head's scale, in 16 KB tiles of 128 rows x 64 columns laid out
    // as the MMA reads them - so a tile is dk / 64 bulk copies of 16 KB, requested by one thread, landing on a barrier
    // of their own while the CTA does something else (the fold; the previous tile's epilogue).
    const char* A_src = a.s0_f16 + req * a.s0_f16_req_stride + (long long)hv * ((long long)MT * KB * A_KB);
    int a_loads = 0, a_waits = 0;         // thread 0: A operands requested / waited for
    auto load_A = [&](int mt) {           // thread 0 only
        const uint32_t ab = smem_u32(abar + (mt & (ABUF - 1)));
        mbar_expect_tx(ab, KB * A_KB);
#pragma unroll
        for (int kb = 0; kb < KB; ++kb)
            bulk_load(smem_u32(A_s + (mt & (ABUF - 1)) * (KB * A_KB) + kb * A_KB), A_src + ((long long)mt * KB + kb) * A_KB, A_KB, ab);
        ++a_loads;
    };
    // the first warp: once the tile's A operand has landed, its dk / 16 MMAs into accumulator mt & 1 and the commit that
    // completes the barrier's phase (if the operand does not land in time nothing is issued, and the CTA's wait for the
    // MMAs runs out in turn); issued by one elected lane of the converged warp (see mma_ss)
    uint32_t tmem_base = 0;
    auto issue = [&](int mt) {
        const bool landed = mbar_wait(smem_u32(abar + (mt & (ABUF - 1))), (ABUF == 2 ? mt >> 1 : mt) & 1);
        ++a_waits;
        if (!__all_sync(0xffffffffu, landed)) return;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t ad = umma_desc(smem_u32(A_s + (mt & (ABUF - 1)) * (KB * A_KB))), bd = umma_desc(smem_u32(R_s));
        constexpr uint32_t idesc = idesc_f16(NB);
#pragma unroll
        for (int kb = 0; kb < KB; ++kb)
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma_ss(tmem_base + (mt & 1) * NB, ad + (uint64_t)((kb * A_KB + ks * 32) >> 4), bd + (uint64_t)((kb * R_KB + ks * 32) >> 4), idesc,
                       (kb | ks) != 0);
        mma_commit(smem_u32(bar));
    };
    // (the first operand is requested before the wait: see launch_dependent for why the store may be read there)
    if (tid == 0) load_A(0);        // in flight while the chain is walked
    asm volatile("griddepcontrol.wait;" ::: "memory");

    // ---- the fold (Section 3.2's recurrence applied to the query from the newest record back) ----
    const T* q = static_cast<const T*>(a.q) + (((long long)req * a.W + bb) * a.Hk + hk) * KD;
    const int32_t* table = a.table + req * a.table_req_stride;
    T* kplane = reinterpret_cast<T*>(a.kplane) + (long long)hk * a.arena_slots * a.k_stride;
    T* vplane = reinterpret_cast<T*>(a.vplane) + (long long)hv * a.arena_slots * a.v_stride;
    float2* gates = a.gates + (long long)hv * a.arena_slots;
    const bool fused = a.k_in != nullptr;      // append fused in: the newest record comes from the caller's tensors

    float r[CK * VEC], corr[CV * VEC];
#pragma unroll
    for (int c = 0; c < CK; ++c) Vec16<T>::load(q + (c * G + g) * VEC, r + c * VEC);
#pragma unroll
    for (int e = 0; e < CV * VEC; ++e) corr[e] = 0.f;
    float decay = 1.f;  // product of the alphas already passed

    // Lane g of a unit fetches the slots of the unit's ancestors at levels g, g + G, ... (the oldest eight levels: one load latency
    // for the whole chain instead of one per level); deeper levels are looked up when they are reached.
    const int old = a.depth - 1;           // records older than the beam's own: levels old - 1 .. 0
    constexpr int NEAR = 8;
    const int32_t my_slot = g < old ? __ldg(table + (long long)g * a.max_beam + bb) : 0;
    int32_t my_slot2 = 0;
    if constexpr (G < NEAR) my_slot2 = G + g < old ? __ldg(table + (long long)(G + g) * a.max_beam + bb) : 0;
    // (two look-ups, used by two runs of the chain walk: one loop with a branch between them costs every level a
    // dozen instructions, taken or not)
    auto slot_near = [&](int level) -> int32_t {                                                                 // level < NEAR
        if constexpr (G == NEAR) return __shfl_sync(0xffffffffu, my_slot, level, G);
        else return __shfl_sync(0xffffffffu, level >= G ? my_slot2 : my_slot, level & (G - 1), G);
    };
    auto slot_far = [&](int level) -> int32_t { return __ldg(table + (long long)level * a.max_beam + bb); };    // level >= NEAR
    struct Raw { uint4 k[CK], v[CV]; float2 gate; };          // this lane's share of a record, as stored
    auto fetch_slot = [&](long long slot) -> Raw {            // an older record, from the arena
        const uint4* kp = reinterpret_cast<const uint4*>(kplane + slot * a.k_stride) + g;
        const uint4* vp = reinterpret_cast<const uint4*>(vplane + slot * a.v_stride) + g;
        Raw x;
#pragma unroll
        for (int c = 0; c < CK; ++c) x.k[c] = __ldg(kp + c * G);
#pragma unroll
        for (int c = 0; c < CV; ++c) x.v[c] = __ldg(vp + c * G);
        x.gate = __ldg(gates + slot);
        return x;
    };
    auto request_slot = [&](long long slot) {
        const char *kp = reinterpret_cast<const char*>(kplane + slot * a.k_stride), *vp = reinterpret_cast<const char*>(vplane + slot * a.v_stride);
        constexpr int KL = KD * (int)sizeof(T) / 128, VL = VD * (int)sizeof(T) / 128;      // lines
#pragma unroll
        for (int x = 0; x < KL + VL; x += G)
            if (x + g < KL + VL) asm volatile("prefetch.global.L2 [%0];" ::"l"(x + g < KL ? kp + (x + g) * 128 : vp + (x + g - KL) * 128));
    };
    // (narrow heads: packed fp32x2 multiply-adds; wide ones do not have the registers for aligned pairs: 256 x 512 37 -> 50 us)
    constexpr bool PACKED = KD + VD <= 128;
    auto pair_fma = [&](float w, const float* x, float* acc) {
        if constexpr (PACKED) {
            const float2 y = __ffma2_rn(make_float2(w, w), make_float2(x[0], x[1]), make_float2(acc[0], acc[1]));
            acc[0] = y.x;
            acc[1] = y.y;
        } else {
            acc[0] = fmaf(w, x[0], acc[0]);
            acc[1] = fmaf(w, x[1], acc[1]);
        }
    };
    auto fold = [&](const Raw& x) {       // c = k . r~ ;  corr += decay beta c v ;  r~ -= beta c k ;  decay *= alpha
        float kx[CK * VEC];
        float dot = 0.f;
        if constexpr (PACKED) {
            float2 d0 = make_float2(0.f, 0.f), d1 = d0;
#pragma unroll
            for (int c = 0; c < CK; ++c) {
                if (G == 4) d0 = d1 = make_float2(0.f, 0.f);       // chunk by chunk: see the kernel's head
                Vec16<T>::unpack(x.k[c], kx + c * VEC);
#pragma unroll
                for (int e = c * VEC; e < (c + 1) * VEC; e += 4) {
                    d0 = __ffma2_rn(make_float2(kx[e], kx[e + 1]), make_float2(r[e], r[e + 1]), d0);
                    d1 = __ffma2_rn(make_float2(kx[e + 2], kx[e + 3]), make_float2(r[e + 2], r[e + 3]), d1);
                }
                if (G == 4) dot = c == 0 ? (d0.x + d0.y) + (d1.x + d1.y) : dot + ((d0.x + d0.y) + (d1.x + d1.y));
            }
            if (G != 4) dot = (d0.x + d0.y) + (d1.x + d1.y);
        } else {
#pragma unroll
            for (int c = 0; c < CK; ++c) {
                Vec16<T>::unpack(x.k[c], kx + c * VEC);
#pragma unroll
                for (int e = 0; e < VEC; ++e) dot = fmaf(kx[c * VEC + e], r[c * VEC + e], dot);
            }
        }
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
        // (DELTA, Eq. 3: the record's second half is the stored update vector, taken with the weight decay (k . x); the
        // projected vector is not changed)
        const float bc = DELTA ? dot : x.gate.y * dot;
        const float wv = decay * bc;
#pragma unroll
        for (int c = 0; c < CV; ++c) {
            float vx[VEC];
            Vec16<T>::unpack(x.v[c], vx);
#pragma unroll
            for (int e = 0; e < VEC; e += 2) pair_fma(wv, vx + e, corr + c * VEC + e);
        }
        if constexpr (!DELTA) {
#pragma unroll
            for (int e = 0; e < CK * VEC; e += 2) pair_fma(-bc, kx + e, r + e);
        }
        decay *= x.gate.x;
    };
    // The beam's own record: from its arena slot, or - append fused in - from the caller's tensors, in which case this
    // unit also writes it to the slot, bit for bit (16-byte vectors; the key once per key head, by its first value
    // head).  The fold reads the caller's copy, so nothing in this launch reads what another CTA of it writes.
    // 64 x 64 with fp32 records asks for the newest older record before the append's stores, which wait for the own one, and keeps
    // the own fold out of the loop: no spills, 4 x 300 beams x 16 heads 168 -> 159 us a generation, 4 x 512 x 32 1038 -> 988 us.
    // (bf16 records: 1.4 % faster on the stack, 2 - 3 % slower on 60 - 128 beams; 128 x 128: 1 % slower.  They keep the loop.)
    constexpr bool EARLY = !DELTA && KD + VD <= 128 && sizeof(T) == 4;
    Raw cur, first;
    {
        const long long slot = a.bases.base[req] + bb;
        T* kdst = kplane + slot * a.k_stride;
        T* vdst = vplane + slot * a.v_stride;
        const T *ksrc = kdst, *vsrc = vdst;
        if (fused) {
            const long long krow = ((long long)req * a.W + bb) * a.Hk + hk, vrow = ((long long)req * a.W + bb) * Hv + hv;
            ksrc = static_cast<const T*>(a.k_in) + krow * KD;
            vsrc = static_cast<const T*>(a.v_in) + vrow * VD;
            cur.gate = make_float2(__ldg(a.alpha_in + vrow), __ldg(a.beta_in + vrow));
        } else {
            cur.gate = __ldg(gates + slot);
        }
#pragma unroll
        for (int c = 0; c < CK; ++c) cur.k[c] = __ldg(reinterpret_cast<const uint4*>(ksrc) + c * G + g);
#pragma unroll
        for (int c = 0; c < CV; ++c) cur.v[c] = __ldg(reinterpret_cast<const uint4*>(vsrc) + c * G + g);
        if (EARLY && old > 0) first = fetch_slot(old > NEAR ? slot_far(old - 1) : slot_near(old - 1));
        if (fused && active && !key_row) {
            if constexpr (!DELTA) {      // (the delta half of a delta record is written after the contraction)
#pragma unroll
                for (int c = 0; c < CV; ++c) reinterpret_cast<uint4*>(vdst)[c * G + g] = cur.v[c];
            }
            if (hv % a.g == 0) {
#pragma unroll
                for (int c = 0; c < CK; ++c) reinterpret_cast<uint4*>(kdst)[c * G + g] = cur.k[c];
            }
            if (g == 0) gates[slot] = cur.gate;
        }
    }
    float kq = 0.f;          // DELTA: k_t . q_t
    if constexpr (DELTA) {
        float kx[CK * VEC];
#pragma unroll
        for (int c = 0; c < CK; ++c) {
            Vec16<T>::unpack(cur.k[c], kx + c * VEC);
            float part = G == 4 ? 0.f : kq;
#pragma unroll
            for (int e = 0; e < VEC; ++e) part = fmaf(kx[c * VEC + e], r[c * VEC + e], part);
            kq = G == 4 && c > 0 ? kq + part : part;
        }
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) kq += __shfl_xor_sync(0xffffffffu, kq, off);
        if (key_row) {
#pragma unroll
            for (int e = 0; e < CK * VEC; ++e) r[e] = kx[e];
        }
    }
    // Narrow records are fetched one level ahead of their fold (the chain is a string of dependent loads otherwise);
    // wide ones would not fit in the registers twice.
    constexpr bool AHEAD = KD + VD <= 256;
    const int near_top = min(old, NEAR) - 1;        // levels near_top .. 0: slots among the lanes'; old - 1 .. NEAR: in memory
    if constexpr (DELTA) {                       // the replay runs over the older records only
        if (old > 0) {
            Raw x = old > NEAR ? fetch_slot(slot_far(old - 1)) : fetch_slot(slot_near(old - 1));
            for (int level = old - 2; level >= NEAR; --level) {
                const Raw next = fetch_slot(slot_far(level));
                fold(x);
                x = next;
            }
            for (int level = min(old - 2, near_top); level >= 0; --level) {
                const Raw next = fetch_slot(slot_near(level));
                fold(x);
                x = next;
            }
            fold(x);
        }
    } else if constexpr (EARLY) {
        fold(cur);
        if (old > 0) {
            cur = first;
            for (int level = old - 2; level >= NEAR; --level) {
                const Raw next = fetch_slot(slot_far(level));
                fold(cur);
                cur = next;
            }
            for (int level = min(old - 2, near_top); level >= 0; --level) {
                const Raw next = fetch_slot(slot_near(level));
                fold(cur);
                cur = next;
            }
            fold(cur);
        }
    } else if constexpr (AHEAD) {
        for (int level = old - 1; level >= NEAR; --level) {
            const Raw next = fetch_slot(slot_far(level));
            fold(cur);
            cur = next;
        }
        for (int level = near_top; level >= 0; --level) {
            const Raw next = fetch_slot(slot_near(level));
            fold(cur);
            cur = next;
        }
        fold(cur);
    } else {
        if (REQUEST && old > 0 && old <= NEAR) request_slot(slot_near(near_top));
        fold(cur);
        for (int level = old - 1; level >= NEAR; --level) {
            const Raw x = fetch_slot(slot_far(level));
            fold(x);
        }
        for (int level = near_top; level >= 0; --level) {
            const Raw x = fetch_slot(slot_near(level));
            if (REQUEST && level > 0) request_slot(slot_near(level - 1));
            fold(x);
        }
    }

    // ---- the folded query decay * r~ as the unit's operand row ----
    float inv_row;               // what undoes the row's scales
    {
        float m = 0.f;
#pragma unroll
        for (int e = 0; e < CK * VEC; ++e) m = fmaxf(m, fabsf(r[e]));
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, off));
        float sc, inv;
        pow2_scale(m * fabsf(decay), ROW_TARGET, sc, inv);
        const float f = decay * sc;
        inv_row = inv / sc0;                     // both powers of two
#pragma unroll
        for (int c = 0; c < CK; ++c) {
            const int el0 = (c * G + g) * VEC;   // first element of the chunk
            uint8_t* p = R_s + (el0 >> 6) * R_KB + grp * 128 + ((((el0 & 63) >> 3) ^ (grp & 7)) << 4) + (el0 & 7) * 2;
            const float* x = r + c * VEC;
            if constexpr (VEC == 8) {
                *reinterpret_cast<uint4*>(p) = make_uint4(pack_f16x2(x[0] * f, x[1] * f), pack_f16x2(x[2] * f, x[3] * f),
                                                          pack_f16x2(x[4] * f, x[5] * f), pack_f16x2(x[6] * f, x[7] * f));
            } else {
                *reinterpret_cast<uint2*>(p) = make_uint2(pack_f16x2(x[0] * f, x[1] * f), pack_f16x2(x[2] * f, x[3] * f));
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes -> visible to the MMA
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
#ifdef ONELA_TEST_HOOKS
    if (warp == 0 && !(g_hook_tiled_skip_issue && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0)) issue(0);
#else
    if (warp == 0) issue(0);
#endif

    OutT* out = static_cast<OutT*>(a.out) + (((long long)req * a.W + b) * Hv + hv) * VD;
    const int quad = warp & 3, half = warp >> 2;     // tensor-memory lane quadrant of this warp, and which 16 beams it takes (first)
    bool failed = false;
#pragma unroll
    for (int mt = 0; mt < MT; ++mt) {
        if (ABUF == 2 && mt + 1 < MT && tid == 0) {
            // the next tile's A operand, under this tile's MMAs: its buffer was last read by tile mt - 1, whose
            // completion this thread has waited for
            load_A(mt + 1);
        }
        const bool ok = mbar_wait(smem_u32(bar), mt & 1);
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        if (__syncthreads_or(ok ? 0 : 1)) { failed = true; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (ABUF == 2) {
            // ... and its MMAs, under this tile's epilogue: their accumulator was read out before the barrier that
            // ended the previous iteration
            if (mt + 1 < MT && warp == 0) issue(mt + 1);
        } else if (mt + 1 < MT && tid == 0) {        // one A operand: free now; its MMAs go out after the barrier below
            load_A(mt + 1);
        }
        {
            const int i = quad * 32 + lane;          // value row within the tile
#pragma unroll
            for (int pass = 0; pass < NB * 8 / THREADS; ++pass) {
                const int b0 = half * 16 + pass * (THREADS / 8);
                uint32_t v[16];
                tmem_ld16(tmem_base + (mt & 1) * NB + b0 + ((uint32_t)(quad * 32) << 16), v);
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (mt * 128 + i < VD) {
#pragma unroll
                    for (int j = 0; j < 16; ++j) C_s[(b0 + j) * CP + i] = __uint_as_float(v[j]);
                }
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if (ABUF == 1 && mt + 1 < MT && warp == 0) issue(mt + 1);
        // A unit's lanes read their elements of its row back, undo the scales and add corr, which never left their registers.
        // (Corr added in the tile - written there before, read and written again under the accumulator - cost twice the
        // shared-memory accesses.)
        auto output = [&](int c, float* x) {
            // (a chunk of eight elements by two 16-byte reads: lanes 4 - 7 take theirs in the other order, off the banks of lanes 0 - 3)
            const float* src = C_s + grp * CP + (c * G + g) * VEC - mt * 128;
            const int first = VEC == 8 ? (g >> 2) * 4 : 0;       // (four lanes: no such banks)
            const float4 t = *reinterpret_cast<const float4*>(src + first);
            float y[VEC];
            y[0] = t.x; y[1] = t.y; y[2] = t.z; y[3] = t.w;
            if constexpr (VEC == 8) {
                const float4 w = *reinterpret_cast<const float4*>(src + (first ^ 4));
                y[0] = first ? w.x : t.x; y[1] = first ? w.y : t.y; y[2] = first ? w.z : t.z; y[3] = first ? w.w : t.w;
                y[4] = first ? t.x : w.x; y[5] = first ? t.y : w.y; y[6] = first ? t.z : w.z; y[7] = first ? t.w : w.w;
            }
#pragma unroll
            for (int e = 0; e < VEC; ++e) x[e] = fmaf(y[e], inv_row, corr[c * VEC + e]);
        };
        if constexpr (DELTA) {
            // Eq. 2 and 4 on the beam's two rows (even: S_{t-1} q_t, odd: S_{t-1} k_t), by the even row's lanes:
            //   delta_t = beta_t (v_t - alpha_t S_{t-1} k_t) ,  o_t = alpha_t S_{t-1} q_t + delta_t (k_t . q_t)
            float own[CV][VEC];
#pragma unroll
            for (int c = 0; c < CV; ++c) output(c, own[c]);
            __syncwarp();
            if (key_row) {
#pragma unroll
                for (int c = 0; c < CV; ++c)
#pragma unroll
                    for (int e = 0; e < VEC; e += 4)
                        *reinterpret_cast<float4*>(C_s + grp * CP + (c * G + g) * VEC + e) = make_float4(own[c][e], own[c][e + 1], own[c][e + 2], own[c][e + 3]);
            }
            __syncwarp();
            if (active && !key_row) {
                T* ddst = vplane + (long long)(a.bases.base[req] + bb) * a.v_stride;
#pragma unroll
                for (int c = 0; c < CV; ++c) {
                    const float* uk = C_s + (grp + 1) * CP + (c * G + g) * VEC;
                    float vx[VEC], dl[VEC], o[VEC];
                    Vec16<T>::unpack(cur.v[c], vx);
#pragma unroll
                    for (int e = 0; e < VEC; ++e) {
                        dl[e] = cur.gate.y * fmaf(-cur.gate.x, uk[e], vx[e]);
                        o[e] = fmaf(dl[e], kq, cur.gate.x * own[c][e]);
                    }
                    store_out<OutT, VEC>(out + (c * G + g) * VEC, o);
                    store_out<T, VEC>(ddst + (c * G + g) * VEC, dl);
                }
            }
        } else if (active) {
#pragma unroll
            for (int c = 0; c < CV; ++c) {
                if ((c * G * VEC) / 128 != mt) continue;
                float x[VEC];
                output(c, x);
                store_out<OutT, VEC>(out + (c * G + g) * VEC, x);
            }
        }
        if (mt + 1 < MT) __syncthreads();      // the tile is read out before the next accumulators overwrite it
    }
    if (tid == 0) {
        // a CTA must not exit with bulk copies still landing in its shared memory: after a wait ran out nobody may
        // have waited for the A operand requested last (requests use the two barriers in turn, in order)
        for (; a_waits < a_loads; ++a_waits)
            mbar_wait(smem_u32(abar + (a_waits & (ABUF - 1))), (ABUF == 2 ? a_waits >> 1 : a_waits) & 1);
    }
    if (failed && tid == 0) {
        if (atomicCAS(a.status, ONELA_OK, ONELA_E_TIMEOUT) == ONELA_OK) a.status[1] = (int32_t)(blockIdx.x + gridDim.x * (blockIdx.y + gridDim.y * blockIdx.z));
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(ACC_COLS) : "memory");
    }
}

template <int KD, int VD, typename T, typename OutT, bool DELTA, int G, bool REQUEST = false>
cudaError_t launch_lanes(const TiledArgs& a, cudaStream_t stream) {
    auto kern = decode_tiled_kernel<KD, VD, T, OutT, DELTA, G, REQUEST>;
    constexpr int NB = tiled_beams<KD, VD>(), THREADS = NB * G, BPT = DELTA ? NB / 2 : NB;
    constexpr size_t smem = tiled_smem_bytes<KD, VD>();
    static_assert(smem <= 232448, "shared memory per CTA");
    // One-time set-up per instantiation and device (function attributes belong to a device's context).
    constexpr int MAX_DEVICES = 64;
    static std::mutex setup_mutex;
    static bool ready[MAX_DEVICES] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    {
        std::lock_guard<std::mutex> lock(setup_mutex);
        if (!ready[dev]) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
            // shared memory for the CTAs the registers allow and no more: what is left of the SM's 228 KB serves the
            // fold's record loads as L1 (asking for all of it made 128 x 128 fp32 14 % slower)
            constexpr int pct = (int)((tiled_min_ctas<KD, VD, T, DELTA, G>() * (smem + 1024) * 100 + 228 * 1024 - 1) / (228 * 1024));
            if (e == cudaSuccess) e = cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, pct > 100 ? 100 : pct);
            if (e != cudaSuccess) return e;
            ready[dev] = true;
        }
    }
    dim3 grid((a.W + BPT - 1) / BPT, a.Hk * a.g, a.req_count);
    return launch_dependent(kern, grid, dim3(THREADS), smem, stream, a);
}

// SMs of the current device, 0 if there is none to ask.
int sm_count() {
    constexpr int MAX_DEVICES = 64;
    static std::atomic<int> count_of[MAX_DEVICES] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return 0;
    int n = count_of[dev].load(std::memory_order_relaxed);
    if (n == 0 && cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess) count_of[dev].store(n, std::memory_order_relaxed);
    return n;
}

// 64 x 64 bf16: four lanes per unit take a quarter fewer instructions per fold and leave room for six CTAs of 128 threads per SM
// (five with delta records), 192 units in flight instead of 160; but a warp's chain is longer.  Eight / four lanes, us a
// generation on 148 SMs, tiles in brackets.
// Raw records: 1 x 400 beams x 16 heads (208) 27.9 / 27.9, 2 x 320 x 16 (320) 29.0 / 29.4, 4 x 300 x 16 (640) 61.7 / 60.2, 4 x 384 x 16 (768:
// two waves of five CTAs, one of six) 107.2 / 90.4, 3 x 500 x 24 (1152) 58.1 / 56.4, 4 x 512 x 32 (2048) 191.0 / 183.6.  So the line lies at
// one wave of eight lanes' CTAs.  (Seven or eight CTAs spill; 64 beams per CTA 377 against 375, 13 % slower on narrow beams; fp32
// records 5 % slower and more.)
// Delta records: five CTAs of four lanes spill (104 bytes), four of eight do not, and the spills cost what the fold saves: what is
// gained is a wave.  4 x 150 x 16 (640) 67.4 / 60.5, 3 x 224 x 16 (672) 41.6 / 38.5, 4 x 192 x 16 (768) 103.6 / 109.1, 1 x 500 x 32 (1024)
// 55.1 / 56.1, 3 x 250 x 24 (1152) 58.3 / 60.4, 3 x 200 x 32 (1248) 64.8 / 62.4, 4 x 256 x 32 (2048) 195.8 / 190.2, 4 x 512 x 32 (4096) 348.7 /
// 340.6.  So four lanes where their waves are fewer.  (Four CTAs of four lanes, without spills, on the first, third, fourth, fifth and
// seventh: 68.3, 103.2, 53.4, 56.6, 193.1.)
template <int KD, int VD, typename T, bool DELTA>
bool four_lanes(const TiledArgs& a) {
    constexpr int BPT = tiled_beams<KD, VD>() / (DELTA ? 2 : 1);
    const long long tiles = (long long)((a.W + BPT - 1) / BPT) * a.Hk * a.g * a.req_count;
    const long long eight = (long long)sm_count() * tiled_min_ctas<KD, VD, T, DELTA, 8>(), four = (long long)sm_count() * tiled_min_ctas<KD, VD, T, DELTA, 4>();
    if (eight == 0) return false;
    return DELTA ? (tiles + four - 1) / four < (tiles + eight - 1) / eight : tiles > eight;
}

// 256 x 256: an older record does not fit in the registers beside the one at hand, so where it comes from HBM its lines are requested
// into L2 a level ahead (nothing else is in flight under the fold); where it is still in L2 the requests only cost issue slots.
// What decides is what one decode call of all layers touches (TiledArgs::call_bytes): by the next call the L2 of 126 MB has seen that
// much since the record was written.  Without / with requests, us a generation (4 or 8 calls, Zipf or uniform parents), MB a call in
// brackets - bf16: 4 x 100 beams x 16 heads (28) 54.9 / 55.6, 109.6 / 111.9; 2 x 300 x 8 heads, 2 layers (33) 86.2 / 87.1, 185.6 / 188.0; 3
// layers (50) 121.2 / 121.9, 269.7 / 267.1, uniform 124.6 / 122.9; 4 x 100 x 16, 2 layers (56) 100.7 / 99.7, 211.9 / 203.5; 2 x 300 x 8, 4 layers (67)
// 371 / 351, 6 layers (101) 588 / 525.  fp32, two lines a lane: 2 x 300 x 8 (31) 130.9 / 134.5; 4 x 100 x 16 (47) 142.0 / 145.0; 1 x 128 x
// 32, 2 layers (58) 108.6 / 109.9, 236.7 / 238.4; 3 layers (88) 166.5 / 164.9, 375.4 / 364.3; 4 x 100 x 16, 2 layers (95) 290.9 / 280.2.
// (The bf16 instantiation with requests spills 4 bytes.  At 256 x 512, where the fold spills, requests were 11 % slower; 128 x 256 fp32
// the same.)
template <typename T>
constexpr long long REQUEST_FROM = (sizeof(T) == 2 ? 48ll : 80ll) << 20;

template <int KD, int VD, typename T, typename OutT, bool DELTA>
cudaError_t launch_one(const TiledArgs& a, cudaStream_t stream) {
    if constexpr (KD == 256 && VD == 256) {
        if (a.call_bytes > REQUEST_FROM<T>) return launch_lanes<KD, VD, T, OutT, DELTA, 8, true>(a, stream);
    }
    if constexpr (KD + VD <= 128 && sizeof(T) == 2) {
        if (four_lanes<KD, VD, T, DELTA>(a)) return launch_lanes<KD, VD, T, OutT, DELTA, 4>(a, stream);
    }
    return launch_lanes<KD, VD, T, OutT, DELTA, 8>(a, stream);
}

template <int KD, int VD, bool DELTA = false>
cudaError_t launch_dims(const TiledArgs& a, int32_t rec_dtype, int32_t out_dtype, cudaStream_t stream) {
    if (rec_dtype == ONELA_DTYPE_BF16) {
        return out_dtype == ONELA_DTYPE_BF16 ? launch_one<KD, VD, __nv_bfloat16, __nv_bfloat16, DELTA>(a, stream)
                                             : launch_one<KD, VD, __nv_bfloat16, float, DELTA>(a, stream);
    }
    return out_dtype == ONELA_DTYPE_BF16 ? launch_one<KD, VD, float, __nv_bfloat16, DELTA>(a, stream)
                                         : launch_one<KD, VD, float, float, DELTA>(a, stream);
}

}  // namespace

#ifdef ONELA_TEST_HOOKS
extern "C" int onela_testhook_tiled_skip_issue(int on) {
    return (int)cudaMemcpyToSymbol(g_hook_tiled_skip_issue, &on, sizeof(int));
}
#endif

bool decode_tiled_supported(int32_t dk, int32_t dv) {
    return (dk == 64 && dv == 64) || (dk == 128 && (dv == 128 || dv == 256 || dv == 512)) || (dk == 256 && (dv == 256 || dv == 512));
}

cudaError_t launch_decode_tiled(const TiledArgs& a, int32_t dk, int32_t dv, int32_t rec_dtype, int32_t out_dtype,
                                cudaStream_t stream) {
    if (a.delta) {       // (alpha, delta, k) records: square heads, the append fused in
        if (!a.k_in || a.g != 1) return cudaErrorInvalidValue;
        if (dk == 64 && dv == 64) return launch_dims<64, 64, true>(a, rec_dtype, out_dtype, stream);
        if (dk == 128 && dv == 128) return launch_dims<128, 128, true>(a, rec_dtype, out_dtype, stream);
        return cudaErrorInvalidValue;
    }
    if (dk == 64 && dv == 64) return launch_dims<64, 64>(a, rec_dtype, out_dtype, stream);
    if (dk == 128 && dv == 128) return launch_dims<128, 128>(a, rec_dtype, out_dtype, stream);
    if (dk == 128 && dv == 256) return launch_dims<128, 256>(a, rec_dtype, out_dtype, stream);
    if (dk == 128 && dv == 512) return launch_dims<128, 512>(a, rec_dtype, out_dtype, stream);
    if (dk == 256 && dv == 256) return launch_dims<256, 256>(a, rec_dtype, out_dtype, stream);
    if (dk == 256 && dv == 512) return launch_dims<256, 512>(a, rec_dtype, out_dtype, stream);
    return cudaErrorInvalidValue;
}

}  // namespace onela
