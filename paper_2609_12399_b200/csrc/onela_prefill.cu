// Prompt -> shared state on the tensor cores (sm_100a): S_T of Eq. 1 from the zero state, dk = dv in {32, 64, 128}.
//
// Token by token (one CTA per head, the recurrence in fp32) a prompt costs 1.1 us per token on as many SMs as there are
// heads.  Here a chunk of C = 64 tokens is one step, in the chunked form of the delta rule (the WY representation of a product
// of Householder-like factors, Bischof and Van Loan 1987; with gates, Gated DeltaNet, Yang et al. 2024).  With g_i =
// prod_{l <= i} alpha_l inside the chunk, A_ij = beta_i (g_i / g_j) (k_i . k_j) for j < i (strictly lower triangular; the
// ratios are running products, nothing is divided) and T = (I + A)^-1, Eq. 1 over the chunk is
//      S_out = g_C S_in + Delta K ,   Delta = U - S_in W^T ,
//      U^T = diag(g_C / g) T diag(beta) V (C x dv) ,   W = diag(g_C / g) T diag(beta g) K (C x dk) .
// T, U and W depend on the tokens alone, so they are prepared a chunk ahead of the state.  (The other grouping, T applied to
// the keys behind Delta, costs the state the rounding of that product; here what the newest tokens contribute - the greater
// part of the state at the usual gates - is U, in fp32, times the keys as they were given.)
//
// Parallelism along the prompt.  The map of a run of chunks is affine, S -> S M + B, and M obeys the same recurrence as
// S (from the identity, with U = 0).  A head's prompt is cut into segments, one per CTA of a cluster; every segment but
// the first carries M as dk more state rows, and at the end the cluster folds the segments in order, S <- S M_p + B_p,
// handing S from CTA to CTA through distributed shared memory.  Nothing goes through global memory but the inputs and
// the result.
//
// One CTA: two TEAMS of 128 threads that prepare chunks in turn (keys -> operand tile, Gram product, inverse, W, U) and 128
// threads per CHAIN of 128 state rows (dk = 128: S and M are a chain each, and hide each other's latency; dk <= 64: one
// chain holds both), coupled by mbarriers over rings of key, W and U tiles.  A thread keeps one state row in fp32 registers.
// Products run as tcgen05.mma kind::f16 with fp32 accumulation, an operand being one fp16 number where that is exact (bf16
// keys, to 2^-28 of the row's largest), otherwise the sum of two (22 to 23 significant bits) or, fp32 records, three where
// that shows (Delta of the S rows, the keys at dk <= 64); U's operands are bf16, the values as they are or in three parts, T
// diag(beta) in three.  Every fp16 row carries its own power of two, exact to apply and to undo, so the range of the caller's
// data does not matter.
//
// Precision.  The tensor core's accumulator truncates towards zero at every MMA.  So the small products are accumulated
// first, and half a unit of the last place per step that counts (KEEP, below) is given back with an operand's low part.  The
// running products of the gates carry their rounding errors along (two more FMAs each), which was the largest single error of
// the preparation.  Relative error against 64 bits, 24 to 16 384 tokens, gates in [0.9, 1]: 0.7 - 0.9e-7; token by token in
// fp32 0.83 - 0.98e-7 (1.25 - 1.81e-7 in the other grouping, uncompensated).  Without decay 0.7 - 2.0e-7 against 1.0 -
// 3.6e-7; gates spread over [0, 1] 0.5 - 0.75e-7 against 0.5 - 0.6e-7.
//   per chunk and chain:  S W^T               3 x dk / 16 MMAs (M = 128, N = 64), A in tensor memory
//                         Delta K             2 x 4 MMAs (N = dk), A in tensor memory
//   per chunk:            K K^T (dk / 16 MMAs), K^T T'^T (2 x 4), V^T (T diag(beta))^T (3 x 4), A = the tile read MN-major
// (fp32 records: Delta K 5 or 6 products, the lowest part of Delta in shared memory; K K^T three, K^T T'^T three, U six.)
// What bounds it now: the latency of a chain's step and, as long, the two preparations in flight, about 11 000 cycles per
// chunk.  16 384 tokens x 32 heads of 128 x 128 bf16: 18.2 ms token by token, 0.435 ms (0.38 ms in the other grouping, whose
// errors were larger); 1021 tokens x 16 heads of 64 x 64 fp32: 376 -> 35 us.  M's chain retired once M has decayed to zero: 0.44 ->
// 0.50 ms, by spills.  The loops of gates or of Delta unrolled at dk <= 64: within 1 % either way, up to 6 % slower together.
//
// Every wait is bounded: a thread that gives up keeps meeting its team's barriers, whose OR makes the team leave
// together, and the cluster barriers, but hands nothing on; ONELA_E_TIMEOUT goes to the status word.  A team always waits for
// its own MMAs, so none is in flight when its operands are written again or tensor memory is freed.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "onela_internal.h"
#include "onela_layout.cuh"
#include "onela_sm100.cuh"

namespace onela {

namespace {

using sm100::bar_or;
using sm100::idesc_f16;
using sm100::mma_commit;
using sm100::mma_ss;
using sm100::mma_ts;
using sm100::mbar_init;
using sm100::pack_f16x2;
using sm100::pow2_scale;
using sm100::smem_u32;
using sm100::tmem_ld16;
using sm100::tmem_st16;
using sm100::umma_desc;

constexpr int C = 64;              // tokens per chunk
constexpr int TILE = C * 128;      // bytes of one K-major operand block: 64 rows of 64 fp16
constexpr int K_STAGES = 3;
constexpr int CTA_BARRIER = 9;     // named barrier of the whole CTA (1 - 4: the teams')
constexpr int AP = C + 4;          // pitch (floats) of the C x C matrix: 16-byte rows
constexpr int MAX_SEGMENTS = 8;    // portable cluster size
// Largest elements of the scaled operand rows: keys and T' in [2^3, 2^4) (so |W| < 64 * 2^8 = 2^14 stays inside fp16's
// range unscaled), state rows and Delta rows in [2^12, 2^13).
constexpr int NARROW = 3, WIDE = 12;
// What the accumulators' truncation takes on average, given back by the operand that goes into the next product: an MMA drops
// half a unit of the last place of a partial sum, 0.72 x 2^-24 of it, and of the partial sums of a product's last steps (the
// large terms) the final one and a part of those before it count.  Delta: U's and its own product's; W: its own and S W^T's.
constexpr float KEEP_DELTA = 1.5f * 0x1p-24f, KEEP_W = 2.f * 0x1p-24f;

struct PrefillArgs {
    const void *k, *v;
    const float *alpha, *beta;
    float* slot;          // [H][dv][dk]
    float* scale_out;     // [H]
    uint16_t* s0_f16;     // the tiled decode kernel's operand copy (see Layout::s0_f16), or null
    int32_t* status;
    int32_t n_tokens, H;
    int32_t first, rest;  // chunks of the first segment, of each other one (the last may hold fewer)
};

template <int D, typename T>
struct Shape {
    static constexpr int KB = D > 64 ? D / 64 : 1;                  // K blocks of 64 elements
    static constexpr int PK = sizeof(T) == 2 ? 1 : D == 128 ? 2 : 3;      // fp16 parts of a key
    static constexpr int DP = PK == 1 ? 2 : 3;                       // ... of the S rows' Delta
    static constexpr int PREPS = 2, CHAINS = D == 128 ? 2 : 1;      // teams of 128 threads
    static constexpr int THREADS = 128 * (PREPS + CHAINS);
    static constexpr int K_BYTES = PK * KB * TILE;
    static constexpr int W_BYTES = D * 256 > 2 * TILE ? D * 256 : 2 * TILE;    // [hi, lo][dk rows][128 bytes]; before that T' (hi, lo)
    static constexpr int U_BYTES = C * D * 4 > 3 * TILE ? C * D * 4 : 3 * TILE;       // [token][dv]; before that T diag(beta) in three parts
    static constexpr int L_BYTES = DP == 3 ? 128 * 128 : 0;          // lowest part of the Delta operand
    // (fp32 at dk = 128: a tile of each is what there is room for; the preparation waits for the chain once per chunk more)
    static constexpr int W_STAGES = D == 128 && PK == 2 ? 1 : 2, U_STAGES = W_STAGES;
    static constexpr int RING = K_STAGES * K_BYTES + W_STAGES * W_BYTES + U_STAGES * U_BYTES + L_BYTES;
    // per preparing team: the C x C matrix, over it the values as an operand tile, and the scratch of the inversion
    static constexpr int A_BYTES = (C * AP * 4 + 1023) / 1024 * 1024, X_BYTES = 5 * 1024;
    static constexpr int TOK_BYTES = 5 * C * 4;                      // per token: alpha, beta, 1 / key scale, row and column weights in T'
    static constexpr int COEF_BYTES = 1024;                          // per U stage: weight of U[C], what undoes W's scale[C], g_C
    // (the Gram product reads 128 rows from a 64-row block and the MN-major tile a second block: what lies behind the key
    // tile is read and the rows that come of it are ignored)
    static constexpr int SMALL = PREPS * TOK_BYTES + U_STAGES * COEF_BYTES + 128 * 4 + 256;
    static constexpr int SMEM = RING + PREPS * (A_BYTES + X_BYTES) + SMALL + 1024;
    static constexpr uint32_t CHAIN_COLS = D + C;                    // S operand (hi, lo) / Delta K ; S W^T / Delta operand (hi, lo)
    static constexpr uint32_t PREP_COL = CHAINS * CHAIN_COLS;        // per preparing team: Gram product, then W, then U
    static constexpr uint32_t TMEM_COLS = D == 128 ? 512 : 256;
    static_assert(PREP_COL + PREPS * C <= TMEM_COLS && SMEM <= 232448 && RING >= D * 128 * 4 + 2 * KB * D * 128, "tensor and shared memory");
    static_assert(32 * 36 * 4 <= X_BYTES && (A_BYTES + X_BYTES) % 1024 == 0 && 2 * TILE <= A_BYTES, "scratch; a tile's swizzle atoms");
    // registers: 512 threads start with 128 each; the state rows (dk floats per thread) take what the preparation leaves
    static constexpr bool SPLIT_REGS = D == 128;
    static constexpr int PREP_REGS = 80, CHAIN_REGS = 176;
    static_assert(!SPLIT_REGS || PREPS * PREP_REGS + CHAINS * CHAIN_REGS <= 4 * 128, "a split beyond the launch's registers waits for ever");
};

// MN-major operand, 128-byte swizzle: rows (K index) of 64 elements, 8-row groups 1024 bytes apart, blocks of 64
// elements along M or N `block` bytes apart.
__device__ __forceinline__ uint64_t umma_desc_mn(uint32_t smem_addr, uint32_t block) {
    return (uint64_t)((smem_addr & 0x3FFFF) >> 4) | ((uint64_t)(block >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) |
           ((uint64_t)2 << 61);
}
constexpr uint32_t A_MN_MAJOR = 1u << 15, B_MN_MAJOR = 1u << 16;     // instruction descriptor: operand is MN-major
constexpr uint32_t BF16_OPERANDS = (1u << 7) | (1u << 10);           // ... both are bf16

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tc_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void proxy_fence() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void arrive(uint32_t bar) { asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory"); }
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
// Two numbers times a power of two as fp16 numbers hi + lo (+ low), packed.  (Rounding hi to a fixed grid instead would make
// sums of hi x hi products exact, but leaves every lo as large as the row's largest element allows.)
__device__ __forceinline__ void split2(float a, float b, uint32_t& hi, uint32_t& lo) {
    hi = pack_f16x2(a, b);
    const float2 h = __half22float2(*reinterpret_cast<const __half2*>(&hi));
    lo = pack_f16x2(a - h.x, b - h.y);
}
__device__ __forceinline__ void split3(float a, float b, uint32_t& hi, uint32_t& lo, uint32_t& low) {
    hi = pack_f16x2(a, b);
    const float2 h = __half22float2(*reinterpret_cast<const __half2*>(&hi));
    const float ra = a - h.x, rb = b - h.y;
    lo = pack_f16x2(ra, rb);
    const float2 l = __half22float2(*reinterpret_cast<const __half2*>(&lo));
    low = pack_f16x2(ra - l.x, rb - l.y);
}
// Sixteen numbers times `scale` in two parts or (low not null) three; `keep`: what the low part gives on top (see KEEP_DELTA).
__device__ __forceinline__ void split16(const float* x, float scale, uint32_t* hi, uint32_t* lo, float keep = 0.f, uint32_t* low = nullptr) {
    const float2 sc = make_float2(scale, scale), kp = make_float2(keep, keep);
#pragma unroll
    for (int e = 0; e < 8; ++e) {
        const float2 y = __fmul2_rn(make_float2(x[2 * e], x[2 * e + 1]), sc);
        hi[e] = pack_f16x2(y.x, y.y);
        const float2 h = __half22float2(*reinterpret_cast<const __half2*>(&hi[e]));
        float2 l = __fadd2_rn(y, make_float2(-h.x, -h.y));
        if (keep != 0.f) l = __ffma2_rn(y, kp, l);
        lo[e] = pack_f16x2(l.x, l.y);
        if (low) {
            const float2 q = __half22float2(*reinterpret_cast<const __half2*>(&lo[e]));
            const float2 r = __fadd2_rn(l, make_float2(-q.x, -q.y));
            low[e] = pack_f16x2(r.x, r.y);
        }
    }
}
// Two fp32 numbers as the sum of three bf16 ones each, packed: eight bits at a time, exact.  (The first is cut off, so that the
// largest numbers stay finite, the second rounded, so that the third has either sign and products left out have no bias.)
__device__ __forceinline__ void split_bf16(float a, float b, uint32_t (&part)[3]) {
    const uint32_t ua = __float_as_uint(a), ub = __float_as_uint(b);
    part[0] = __byte_perm(ua, ub, 0x7632);
    const float ra = a - __uint_as_float(ua & 0xffff0000u), rb = b - __uint_as_float(ub & 0xffff0000u);
    part[1] = sm100::pack_bf16x2(ra, rb);
    float ma, mb;
    unpack_bf16x2(part[1], ma, mb);
    part[2] = sm100::pack_bf16x2(ra - ma, rb - mb);
}
// ... as one K step of a tensor-memory A operand: columns [0, 8) hi, [8, 16) lo
__device__ __forceinline__ void split_to_tmem(uint32_t taddr, const float* x, float scale) {
    uint32_t w[16];
    split16(x, scale, w, w + 8);
    tmem_st16(taddr, w);
}

// acc[r] = sum over l < N of rows[r][l] cols[l]: eight rows (pitch AP, read as broadcast vectors) times this lane's column, the
// even and the odd l in the two halves of packed multiply-adds.  UNROLL steps of four l at a time: all of them at dk <= 64 (5000
// tokens x 16 heads of 32 x 32 fp32 83.2 -> 79.5 us, 6000 x 32 heads of 64 x 64 bf16 124.0 -> 119.5, although that one then spills 12
// bytes: four steps, which do not, 1 - 2 % slower from 1021 to 16 384 tokens), two at dk = 128, whose roles miss the instruction cache
// (16 384 tokens 434.7 -> 429.5; four 439.6, eight 454.2).  Error against 64
// bits: 0.3 % smaller on the mean of fourteen shapes, none more than 0.5 % larger.
template <int N, int UNROLL>
__device__ __forceinline__ void rows8(float* acc, const float* rows, const float* cols, int pitch) {
    float2 sum[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) sum[r] = make_float2(0.f, 0.f);
#pragma unroll UNROLL
    for (int l = 0; l < N; l += 4) {
        const float2 t0 = make_float2(cols[l * pitch], cols[(l + 1) * pitch]), t1 = make_float2(cols[(l + 2) * pitch], cols[(l + 3) * pitch]);
#pragma unroll
        for (int r = 0; r < 8; ++r) {
            const float4 q = *reinterpret_cast<const float4*>(rows + r * AP + l);
            sum[r] = __ffma2_rn(make_float2(q.x, q.y), t0, __ffma2_rn(make_float2(q.z, q.w), t1, sum[r]));
        }
    }
#pragma unroll
    for (int r = 0; r < 8; ++r) acc[r] = sum[r].x + sum[r].y;
}

#ifdef ONELA_TEST_HOOKS
// Test-hooks build only (a second library that the product never loads): when set, one thread of the first head's last segment
// leaves out its arrival for the first chunk's W, so that the chains' wait for it runs out.
__device__ int g_hook_prefill_drop;
#endif

template <int D, typename T>
__global__ void __launch_bounds__(Shape<D, T>::THREADS, 1) prefill_chunk_kernel(const PrefillArgs a) {
    using Z = Shape<D, T>;
    constexpr int JOIN = D == 128 ? 2 : 8;           // see rows8
    constexpr int KB = Z::KB, PK = Z::PK, KS = (D < 64 ? D : 64) / 16;        // K steps of 16 per block of 64
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    uint8_t* w_ring = smem + K_STAGES * Z::K_BYTES;
    float* u_ring = reinterpret_cast<float*>(w_ring + Z::W_STAGES * Z::W_BYTES);
    uint8_t* low_s = reinterpret_cast<uint8_t*>(u_ring) + Z::U_STAGES * Z::U_BYTES;      // the Delta operand's lowest part
    uint8_t* prep_s = smem + Z::RING;                                         // per preparing team: matrix / values, scratch
    float* tok_s = reinterpret_cast<float*>(prep_s + Z::PREPS * (Z::A_BYTES + Z::X_BYTES));
    float* coef_s = tok_s + Z::PREPS * (Z::TOK_BYTES / 4);
    float* hinv_s = coef_s + Z::U_STAGES * (Z::COEF_BYTES / 4);               // [128] what undoes the scales of the rows handed on
    uint64_t* bars = reinterpret_cast<uint64_t*>(hinv_s + 128);
    // W and U: the barriers of even and odd chunks, however many tiles there are (a wait by parity does not tell a chunk's turn
    // from the one after next, and a team that comes late may find both past)
    auto bar_w = [&](int i) { return smem_u32(bars + (i & 1)); };             // W prepared
    auto bar_u = [&](int i) { return smem_u32(bars + 2 + (i & 1)); };         // U (and its coefficients)
    auto bar_wfree = [&](int i) { return smem_u32(bars + 4 + (i & 1)); };     // W, U read out
    auto bar_ufree = [&](int i) { return smem_u32(bars + 6 + (i & 1)); };
    auto bar_kfree = [&](int s) { return smem_u32(bars + 8 + s); };           // key stage s read out
    auto bar_prep = [&](int w) { return smem_u32(bars + 11 + w); };           // a preparing team's MMAs complete
    auto bar_chain = [&](int c) { return smem_u32(bars + 13 + c); };          // a chain's
    auto turn = [](int i) { return (uint32_t)(i >> 1) & 1; };                 // chunk i's parity on its pair of barriers
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 15);
    volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);

    const int tid = threadIdx.x, warp = __shfl_sync(0xffffffffu, tid >> 5, 0), lane = tid & 31;
    const int rank = blockIdx.x, P = gridDim.x, h = blockIdx.y;               // segment of the prompt, segments, head
    const int total = (a.n_tokens + C - 1) / C;
    const int c_begin = rank == 0 ? 0 : a.first + (rank - 1) * a.rest;
    const int n = max(0, min(total, rank == 0 ? a.first : c_begin + a.rest) - c_begin);   // chunks of this CTA
    const bool has_m = rank > 0;

    if (tid == 0) {
        const int chains = D == 128 && has_m ? 2 : 1;
        for (int s = 0; s < 2; ++s) {
            mbar_init(bar_w(s), 128);                                         // the preparing threads
            mbar_init(bar_u(s), 128);
            mbar_init(bar_wfree(s), chains);                                  // the chains' commits
            mbar_init(bar_ufree(s), chains);                                  // ... their leaders
        }
        for (int s = 0; s < K_STAGES; ++s) mbar_init(bar_kfree(s), chains);
        for (int w = 0; w < Z::PREPS; ++w) mbar_init(bar_prep(w), 1);
        for (int c = 0; c < Z::CHAINS; ++c) mbar_init(bar_chain(c), 1);
        *abort_flag = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)), "r"(Z::TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem_base = __shfl_sync(0xffffffffu, *tmem_slot, 0);
    // (programmatic dependent launch: set up beside the previous launch; nothing is read before it has completed)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

    bool fail = false;
    // a team's own MMAs: they complete by themselves, so nobody gives up early and leaves them behind
    auto wait_mma = [&](uint32_t bar, uint32_t parity) {
        if (!sm100::mbar_wait(bar, parity)) {
            fail = true;
            *abort_flag = 1;
        }
    };
    // what another role has to do: bounded, and given up as soon as a role has
    auto wait = [&](uint32_t bar, uint32_t parity) {
        for (int i = 0; i < sm100::WAIT_LIMIT; ++i) {
            if (sm100::mbar_try_wait(bar, parity)) return;
            if ((i & 63) == 63 && *abort_flag) break;
        }
        fail = true;
        *abort_flag = 1;
    };

    if (warp < 4 * Z::PREPS) {
        // =============================== PREPARATION ===============================
        // (two teams take the chunks in turn: each step of a chunk is bounded by the latency of its own dependent chain)
        if constexpr (Z::SPLIT_REGS) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(Z::PREP_REGS));
        const int team = warp >> 2, w4 = warp & 3, pt = tid & 127;
        float* A_s = reinterpret_cast<float*>(prep_s + team * (Z::A_BYTES + Z::X_BYTES));       // [C][AP], later the values
        uint8_t* V_s = reinterpret_cast<uint8_t*>(A_s);
        float* X_s = A_s + Z::A_BYTES / 4;                                                      // [32][36]
        float* alpha_s = tok_s + team * (Z::TOK_BYTES / 4);
        float *beta_s = alpha_s + C, *kinv_s = beta_s + C, *row_s = kinv_s + C, *col_s = row_s + C;
        constexpr int VR = sizeof(T) == 2 ? 1 : 3;                            // bf16 parts of a value
        const uint32_t acc_at = tmem_base + Z::PREP_COL + team * C;
        constexpr int VEC = Vec16<T>::N, CPR = D / VEC, LR = CPR < 8 ? CPR : 8;      // 16-byte chunks and lanes per key row
        constexpr int ROWS = 128 / LR, PASSES = C / ROWS, NC = CPR / LR;
        constexpr int BATCH = PASSES * NC > 8 ? 8 / NC : PASSES;                      // passes whose loads are in flight together
        const T* kp = static_cast<const T*>(a.k) + (long long)h * D;
        const T* vp = static_cast<const T*>(a.v) + (long long)h * D;
        const long long row_stride = (long long)a.H * D;
        auto gate_of = [&](const float* g, int t, float pad) { return t < a.n_tokens ? __ldg(g + (long long)t * a.H + h) : pad; };
        float alpha_next = 1.f, beta_next = 0.f;
        if (team < n && pt < C) {
            alpha_next = gate_of(a.alpha, (c_begin + team) * C + pt, 1.f);
            beta_next = gate_of(a.beta, (c_begin + team) * C + pt, 0.f);
        }
        uint32_t phase = 0;
        for (int i = team; i < n; i += Z::PREPS) {
            const int ks_n = i % K_STAGES, ws = i % Z::W_STAGES, us = i % Z::U_STAGES, t0 = (c_begin + i) * C;
            uint8_t *K_s = smem + ks_n * Z::K_BYTES, *W_s = w_ring + ws * Z::W_BYTES;
            float *U_s = u_ring + us * (Z::U_BYTES / 4), *co = coef_s + us * (Z::COEF_BYTES / 4);
            uint8_t* T_s = reinterpret_cast<uint8_t*>(U_s);                  // T diag(beta), later U
            if (i >= K_STAGES) wait(bar_kfree(ks_n), (i / K_STAGES - 1) & 1);
            // keys as the K-major operand tile, every row with its own power of two; tokens beyond the prompt are zeros with
            // alpha = 1, beta = 0: they change nothing.  (First loads on their way since the chunk before, the state's update on
            // packed pairs: dk = 128 bf16 438 -> 485 us at 16 384 tokens, by spills.)
            const int lr = pt % LR, row0 = pt / LR;
#pragma unroll
            for (int p0 = 0; p0 < PASSES; p0 += BATCH) {
                uint4 raw[BATCH][NC];
#pragma unroll
                for (int p = 0; p < BATCH; ++p) {
                    const int t = t0 + (p0 + p) * ROWS + row0;
#pragma unroll
                    for (int c = 0; c < NC; ++c)
                        raw[p][c] = t < a.n_tokens ? __ldg(reinterpret_cast<const uint4*>(kp + t * row_stride) + c * LR + lr) : make_uint4(0, 0, 0, 0);
                }
#pragma unroll
                for (int p = 0; p < BATCH; ++p) {
                    const int row = (p0 + p) * ROWS + row0;
                    float x[NC * VEC], m = 0.f;
#pragma unroll
                    for (int c = 0; c < NC; ++c) Vec16<T>::unpack(raw[p][c], x + c * VEC);
#pragma unroll
                    for (int e = 0; e < NC * VEC; ++e) m = fmaxf(m, fabsf(x[e]));
#pragma unroll
                    for (int o = LR / 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
                    float sc, inv;
                    pow2_scale(m, NARROW, sc, inv);
                    if (lr == 0) kinv_s[row] = inv;
#pragma unroll
                    for (int c = 0; c < NC; ++c) {
                        const int el = (c * LR + lr) * VEC;
                        uint8_t* dst = K_s + (el >> 6) * TILE + row * 128 + ((((el & 63) >> 3) ^ (row & 7)) << 4) + (el & 7) * 2;
                        const float* y = x + c * VEC;
                        if constexpr (VEC == 8) {        // bf16 keys: exact in one fp16 number
                            *reinterpret_cast<uint4*>(dst) = make_uint4(pack_f16x2(y[0] * sc, y[1] * sc), pack_f16x2(y[2] * sc, y[3] * sc),
                                                                        pack_f16x2(y[4] * sc, y[5] * sc), pack_f16x2(y[6] * sc, y[7] * sc));
                        } else {
                            uint32_t hi[2], lo[2], low[2];
#pragma unroll
                            for (int e = 0; e < 2; ++e)
                                split3(y[2 * e] * sc, y[2 * e + 1] * sc, hi[e], lo[e], low[e]);
                            *reinterpret_cast<uint2*>(dst) = make_uint2(hi[0], hi[1]);
                            *reinterpret_cast<uint2*>(dst + KB * TILE) = make_uint2(lo[0], lo[1]);
                            if constexpr (PK == 3) *reinterpret_cast<uint2*>(dst + 2 * KB * TILE) = make_uint2(low[0], low[1]);
                        }
                    }
                }
            }
            const float alpha = alpha_next, beta = beta_next;
            if (pt < C) {
                alpha_s[pt] = alpha;
                beta_s[pt] = beta;
                if (i + Z::PREPS < n) {
                    alpha_next = gate_of(a.alpha, t0 + Z::PREPS * C + pt, 1.f);
                    beta_next = gate_of(a.beta, t0 + Z::PREPS * C + pt, 0.f);
                }
            }
            proxy_fence();
            tc_fence_before();
            if (bar_or(1 + team, 128, fail ? 1 : 0)) { fail = true; break; }
            if (w4 == 0) {          // Gram product of the (scaled) keys: rows 0 - 63 are wanted, 128 are computed
                tc_fence_after();
                const uint64_t kd = umma_desc(smem_u32(K_s));
#pragma unroll 1
                for (int t = PK > 1 ? 2 : 0; t >= 0; --t)                   // small terms first: (lo hi, hi lo,) hi hi
#pragma unroll 1
                    for (int kb = 0; kb < KB; ++kb)
#pragma unroll
                        for (int ks = 0; ks < KS; ++ks) {
                            const int at = (kb * TILE + ks * 32) >> 4;
                            mma_ss(acc_at, kd + (at + (t == 2 ? (KB * TILE) >> 4 : 0)), kd + (at + (t == 1 ? (KB * TILE) >> 4 : 0)), idesc_f16(C),
                                   t != (PK > 1 ? 2 : 0) || kb || ks);
                        }
                mma_commit(bar_prep(team));
            }
            if (i + Z::PREPS < n) { // the lines of the team's next chunk into L2
                constexpr int LINES = D * (int)sizeof(T) / 128 > 0 ? D * (int)sizeof(T) / 128 : 1;
                for (int x = pt; x < 2 * C * LINES; x += 128) {
                    const int row = (x >> 1) / LINES, ln = (x >> 1) % LINES, t = min(t0 + Z::PREPS * C + row, a.n_tokens - 1);
                    const char* p = reinterpret_cast<const char*>(((x & 1) ? vp : kp) + t * row_stride) + ln * 128;
                    asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
                }
            }
            wait_mma(bar_prep(team), phase);
            phase ^= 1;
            tc_fence_after();
            // A = beta_i (g_i / g_j) (k_i . k_j), row i by thread i; the gate products run from the right, each as a sum of two
            // numbers (the product and what its roundings have left out).  g = alpha_0 ... alpha_i; the other half of the
            // threads takes the products of the gates behind the token.
            float g = 1.f, g_rest = 0.f;
            auto times = [&](float x) {
                const float p = g * x;
                g_rest = fmaf(g_rest, x, fmaf(g, x, -p));
                g = p;
            };
            if (w4 >= 2) {
#pragma unroll 2
                for (int l = C - 4; l >= 0; l -= 4) {
                    const float4 al = *reinterpret_cast<const float4*>(alpha_s + l);
                    const int me = pt - C;
                    times(l + 3 > me ? al.w : 1.f);
                    times(l + 2 > me ? al.z : 1.f);
                    times(l + 1 > me ? al.y : 1.f);
                    times(l > me ? al.x : 1.f);
                }
                row_s[pt - C] = (g + g_rest) * kinv_s[pt - C];
            } else {
                const float coef = beta * kinv_s[pt];
#pragma unroll 1
                for (int cb = 3; cb >= 0; --cb) {
                    uint32_t v[16];
                    tmem_ld16(acc_at + cb * 16 + ((uint32_t)(w4 * 32) << 16), v);
                    tc_wait_ld();
#pragma unroll
                    for (int e = 12; e >= 0; e -= 4) {
                        const float4 al = *reinterpret_cast<const float4*>(alpha_s + cb * 16 + e), ki = *reinterpret_cast<const float4*>(kinv_s + cb * 16 + e);
                        const float alv[4] = {al.x, al.y, al.z, al.w}, kiv[4] = {ki.x, ki.y, ki.z, ki.w};
                        float row[4];
#pragma unroll
                        for (int f = 3; f >= 0; --f) {
                            const int l = cb * 16 + e + f;
                            row[f] = l < pt ? (coef * (g + g_rest)) * (__uint_as_float(v[e + f]) * kiv[f]) : 0.f;
                            times(l <= pt ? alv[f] : 1.f);
                        }
                        *reinterpret_cast<float4*>(A_s + pt * AP + cb * 16 + e) = make_float4(row[0], row[1], row[2], row[3]);
                    }
                }
                col_s[pt] = (g + g_rest) * kinv_s[pt];
                __syncwarp();
                // T = (I + A)^-1 in place, from the diagonal out.  Blocks of 16, two per warp, one column per lane by forward
                // substitution; then a warp's two blocks are joined, then the two warps': - T22 A21 T11 below the diagonal.
                float* L = A_s + (w4 * 32) * (AP + 1) + (lane >> 4) * (16 * AP + 16);
                const int col = lane & 15;
                float x[16];
#pragma unroll
                for (int r = 0; r < 16; ++r) {
                    float s0 = r == col ? 1.f : 0.f, s1 = 0.f;
#pragma unroll
                    for (int l = 0; l < r; l += 4) {
                        const float4 q = *reinterpret_cast<const float4*>(L + r * AP + l);
                        s0 = fmaf(-q.x, x[l], s0);
                        if (l + 1 < r) s1 = fmaf(-q.y, x[l + 1], s1);
                        if (l + 2 < r) s0 = fmaf(-q.z, x[l + 2], s0);
                        if (l + 3 < r) s1 = fmaf(-q.w, x[l + 3], s1);
                    }
                    x[r] = s0 + s1;
                }
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 16; ++r) L[r * AP + col] = x[r];
                __syncwarp();
                float* B21 = A_s + (w4 * 32) * (AP + 1) + (16 + (lane >> 4) * 8) * AP;       // eight rows of the lower block per half warp
                float acc[8];
                rows8<16, JOIN>(acc, B21, A_s + (w4 * 32) * (AP + 1) + col, AP);
#pragma unroll
                for (int r = 0; r < 8; ++r) X_s[w4 * (16 * 20) + ((lane >> 4) * 8 + r) * 20 + col] = acc[r];
                __syncwarp();
                rows8<16, JOIN>(acc, B21 + 16, X_s + w4 * (16 * 20) + col, 20);
                __syncwarp();
#pragma unroll
                for (int r = 0; r < 8; ++r) B21[r * AP + col] = -acc[r];
            }
            tc_fence_before();
            bar_or(1 + team, 128, 0);
            {
                float acc[8];
                rows8<32, JOIN>(acc, A_s + (32 + 8 * w4) * AP, A_s + lane, AP);
#pragma unroll
                for (int r = 0; r < 8; ++r) X_s[(8 * w4 + r) * 36 + lane] = acc[r];
                bar_or(1 + team, 128, 0);
                rows8<32, JOIN>(acc, A_s + (32 + 8 * w4) * AP + 32, X_s + lane, 36);
#pragma unroll
                for (int r = 0; r < 8; ++r) A_s[(32 + 8 * w4 + r) * AP + lane] = -acc[r];
            }
            bar_or(1 + team, 128, 0);
            // T' = diag(g_C / g) T diag(beta g), the keys' scales undone on both sides, as an operand tile (fp16 hi, lo) where W
            // will be, and T diag(beta) as one (bf16, three parts) where U will be.  Row pt / 2 by threads pt and pt + 1, columns
            // 16 h .. and 32 + 16 h .. (conflict-free reads)
            if (i >= Z::W_STAGES) wait(bar_wfree(i - Z::W_STAGES), turn(i - Z::W_STAGES));
            if (i >= Z::U_STAGES) wait(bar_ufree(i - Z::U_STAGES), turn(i - Z::U_STAGES));
            {
                const int ti = pt >> 1, hf = pt & 1;
                const float weight = row_s[ti];
                float t[32], m = 0.f;
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const int at = 16 * hf + (q >> 2) * 32 + (q & 3) * 4;
                    const float4 x = *reinterpret_cast<const float4*>(A_s + ti * AP + at), be = *reinterpret_cast<const float4*>(beta_s + at);
                    const float4 c4 = *reinterpret_cast<const float4*>(col_s + at);
                    t[4 * q] = x.x * be.x;
                    t[4 * q + 1] = x.y * be.y;
                    t[4 * q + 2] = x.z * be.z;
                    t[4 * q + 3] = x.w * be.w;
                    m = fmaxf(fmaxf(m, fabsf((t[4 * q] * c4.x) * weight)), fabsf((t[4 * q + 1] * c4.y) * weight));
                    m = fmaxf(fmaxf(m, fabsf((t[4 * q + 2] * c4.z) * weight)), fabsf((t[4 * q + 3] * c4.w) * weight));
                }
                m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 1));
                float sc, inv;
                pow2_scale(m, NARROW, sc, inv);
#pragma unroll
                for (int c = 0; c < 4; ++c) {                               // chunks of eight columns
                    const int ch = 4 * (c >> 1) + 2 * hf + (c & 1), at = ti * 128 + ((ch ^ (ti & 7)) << 4);
                    uint32_t hi[4], lo[4], part[4][3];
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
                        const float a0 = t[8 * c + 2 * e], a1 = t[8 * c + 2 * e + 1];
                        const float2 c2 = *reinterpret_cast<const float2*>(col_s + 8 * ch + 2 * e);
                        split_bf16(a0, a1, part[e]);
                        split2(((a0 * c2.x) * weight) * sc, ((a1 * c2.y) * weight) * sc, hi[e], lo[e]);
                    }
                    *reinterpret_cast<uint4*>(W_s + at) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
                    *reinterpret_cast<uint4*>(W_s + TILE + at) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
#pragma unroll
                    for (int p = 0; p < 3; ++p) *reinterpret_cast<uint4*>(T_s + p * TILE + at) = make_uint4(part[0][p], part[1][p], part[2][p], part[3][p]);
                }
                if (hf == 0) {
                    co[ti] = weight;
                    co[C + ti] = inv;
                }
                if (pt == C - 1) co[2 * C] = g + g_rest;
            }
            proxy_fence();
            if (bar_or(1 + team, 128, fail ? 1 : 0)) { fail = true; break; }
            if (w4 == 0) {          // W^T = K^T T'^T: lanes = dk, columns = tokens
                tc_fence_after();
                const uint64_t kd = umma_desc_mn(smem_u32(K_s), TILE), td = umma_desc(smem_u32(W_s));
                constexpr int FIRST = PK > 1 ? 2 : 1;
#pragma unroll 1
                for (int t = FIRST; t >= 0; --t)                            // small terms first: (lo hi,) hi lo, hi hi
#pragma unroll
                    for (int ks = 0; ks < C / 16; ++ks)
                        mma_ss(acc_at, kd + (t == 2 ? (KB * TILE) >> 4 : 0) + ((ks * 2048) >> 4), td + (t == 1 ? TILE >> 4 : 0) + ((ks * 32) >> 4),
                               idesc_f16(C) | A_MN_MAJOR, t != FIRST || ks);
                mma_commit(bar_prep(team));
            }
            // the values ([token][dv]), part `round` of them, as an operand tile over the matrix (which nobody needs any more), in
            // groups whose loads are in flight together
            constexpr int CH = D / 8, EACH = C * CH / 128, GROUP = EACH > 4 ? 4 : EACH;
            uint4 val[GROUP][sizeof(T) / 2];
            auto load_values = [&](int x0) {
#pragma unroll
                for (int x = 0; x < GROUP; ++x) {
                    const int item = (x0 + x) * 128 + pt, t = t0 + item / CH;
#pragma unroll
                    for (int c = 0; c < (int)sizeof(T) / 2; ++c)
                        val[x][c] = t < a.n_tokens ? __ldg(reinterpret_cast<const uint4*>(vp + t * row_stride + item % CH * 8) + c) : make_uint4(0, 0, 0, 0);
                }
            };
            auto store_values = [&](int x0, int round) {
#pragma unroll
                for (int x = 0; x < GROUP; ++x) {
                    const int item = (x0 + x) * 128 + pt, row = item / CH, ch = item % CH;
                    uint4 w = val[x][0];
                    if constexpr (sizeof(T) == 4) {
                        const uint32_t f[8] = {val[x][0].x, val[x][0].y, val[x][0].z, val[x][0].w, val[x][1].x, val[x][1].y, val[x][1].z, val[x][1].w};
                        uint32_t part[4][3];
#pragma unroll
                        for (int e = 0; e < 4; ++e) split_bf16(__uint_as_float(f[2 * e]), __uint_as_float(f[2 * e + 1]), part[e]);
                        w = round == 0   ? make_uint4(part[0][0], part[1][0], part[2][0], part[3][0])
                            : round == 1 ? make_uint4(part[0][1], part[1][1], part[2][1], part[3][1])
                                         : make_uint4(part[0][2], part[1][2], part[2][2], part[3][2]);
                    }
                    *reinterpret_cast<uint4*>(V_s + (ch >> 3) * TILE + row * 128 + (((ch & 7) ^ (row & 7)) << 4)) = w;
                }
            };
            load_values(0);
            if constexpr (VR == 1) {
#pragma unroll
                for (int x0 = 0; x0 < EACH; x0 += GROUP) {
                    if (x0 > 0) load_values(x0);
                    store_values(x0, 0);
                }
            }
            wait_mma(bar_prep(team), phase);
            phase ^= 1;
            tc_fence_after();
#pragma unroll
            for (int cb = 0; cb < 4; ++cb) {                                // over T', which has been read
                uint32_t v[16], hi[8], lo[8];
                tmem_ld16(acc_at + cb * 16 + ((uint32_t)(w4 * 32) << 16), v);
                tc_wait_ld();
                float x[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) x[e] = __uint_as_float(v[e]);
                split16(x, 1.f, hi, lo, KEEP_W);
                if (pt < D) {
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        uint8_t* dst = W_s + pt * 128 + (((2 * cb + e) ^ (pt & 7)) << 4);
                        *reinterpret_cast<uint4*>(dst) = make_uint4(hi[4 * e], hi[4 * e + 1], hi[4 * e + 2], hi[4 * e + 3]);
                        *reinterpret_cast<uint4*>(dst + D * 128) = make_uint4(lo[4 * e], lo[4 * e + 1], lo[4 * e + 2], lo[4 * e + 3]);
                    }
                }
            }
            proxy_fence();
            tc_fence_before();
#ifdef ONELA_TEST_HOOKS
            if (!(g_hook_prefill_drop && blockIdx.x == gridDim.x - 1 && blockIdx.y == 0 && i == 0 && pt == 0)) arrive(bar_w(i));
#else
            arrive(bar_w(i));
#endif
            // U^T (but for g_C / g) = V^T (T diag(beta))^T: lanes = dv, columns = tokens; bf16 values as they are, fp32 ones in
            // three rounds of a bf16 part each, the smallest first
#pragma unroll 1
            for (int round = VR - 1; round >= 0; --round) {
                if constexpr (VR > 1) {
                    if (round < VR - 1) {
                        if (EACH > GROUP) load_values(0);
                        wait_mma(bar_prep(team), phase);                        // the tile has been read
                        phase ^= 1;
                    }
#pragma unroll
                    for (int x0 = 0; x0 < EACH; x0 += GROUP) {
                        if (x0 > 0) load_values(x0);
                        store_values(x0, round);
                    }
                }
                proxy_fence();
                tc_fence_before();
                bar_or(1 + team, 128, 0);
                if (w4 == 0) {
                    tc_fence_after();
                    const uint64_t vd = umma_desc_mn(smem_u32(V_s), TILE), td = umma_desc(smem_u32(T_s));
#pragma unroll 1
                    for (int t = 2 - round; t >= 0; --t)
#pragma unroll
                        for (int ks = 0; ks < C / 16; ++ks)
                            mma_ss(acc_at, vd + ((ks * 2048) >> 4), td + ((t * TILE) >> 4) + ((ks * 32) >> 4), idesc_f16(C) | A_MN_MAJOR | BF16_OPERANDS,
                                   round != VR - 1 || t != 2 - round || ks);
                    mma_commit(bar_prep(team));
                }
            }
            wait_mma(bar_prep(team), phase);
            phase ^= 1;
            tc_fence_after();
#pragma unroll
            for (int cb = 0; cb < 4; ++cb) {                                // over T diag(beta), which has been read
                uint32_t v[16];
                tmem_ld16(acc_at + cb * 16 + ((uint32_t)(w4 * 32) << 16), v);
                tc_wait_ld();
                if (pt < D) {
#pragma unroll
                    for (int e = 0; e < 16; ++e) U_s[(cb * 16 + e) * D + pt] = __uint_as_float(v[e]);
                }
            }
            tc_fence_before();
            arrive(bar_u(i));
        }
        bar_or(CTA_BARRIER, Z::THREADS, fail ? 1 : 0);        // the chains take the rings' memory over
        if (P > 1)
            for (int p = 0; p < P; ++p) cluster_sync();       // (every thread of the cluster meets every one)
    } else {

    // =============================== STATE ROWS ===============================
    // thread = one row: of S, of M (segments that do not start the prompt), or idle (dk <= 64)
    if constexpr (Z::SPLIT_REGS) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(Z::CHAIN_REGS));
    const int chain = (warp >> 2) - Z::PREPS, team = 1 + (warp >> 2);
    const int r = (warp & 3) * 32 + lane;
    const bool is_s = (D == 128 ? chain == 0 : r < D);
    const bool is_m = has_m && (D == 128 ? chain == 1 : r >= D && r < 2 * D);
    const int mrow = D == 128 ? r : r - D;
    const uint32_t taddr = tmem_base + chain * Z::CHAIN_COLS + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t s_at = taddr, d_at = taddr + D;            // S operand / Delta K ; S W^T / Delta operand
    const uint32_t s_col = tmem_base + chain * Z::CHAIN_COLS, d_col = s_col + D;      // ... without the warp's lanes
    const bool issuer = (warp & 3) == 0, leader = issuer && lane == 0;
    uint32_t phase = 0;                                       // of the chain's barrier
    float S[D];
    float inv_row = 1.f;
    auto store_operand = [&](float m) {                       // the row as the next product's A operand; m: its largest magnitude
        float sc;
        pow2_scale(m, WIDE, sc, inv_row);
#pragma unroll
        for (int b = 0; b < D / 16; ++b) split_to_tmem(s_at + 16 * b, S + 16 * b, sc);
        tc_wait_st();
        tc_fence_before();
    };
#pragma unroll
    for (int d = 0; d < D; ++d) S[d] = is_m && d == mrow ? 1.f : 0.f;
    if ((D < 128 || chain == 0 || has_m) && n > 0) {
        float largest = is_m ? 1.f : 0.f;                     // of the row
#pragma unroll 1
        for (int i = 0; i < n; ++i) {
            store_operand(largest);
            if (bar_or(team, 128, fail ? 1 : 0)) { fail = true; break; }
            const int ks_n = i % K_STAGES, ws = i % Z::W_STAGES, us = i % Z::U_STAGES;
            const uint8_t *K_s = smem + ks_n * Z::K_BYTES, *W_s = w_ring + ws * Z::W_BYTES;
            const float *U_s = u_ring + us * (Z::U_BYTES / 4), *co = coef_s + us * (Z::COEF_BYTES / 4);
            wait(bar_w(i), turn(i));
            if (issuer) {                                     // S W^T, small terms first: hi lo, lo hi, hi hi
                tc_fence_after();
                const uint64_t wd = umma_desc_mn(smem_u32(W_s), D * 128);
#pragma unroll 1
                for (int t = 2; t >= 0; --t)
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks)
                        mma_ts(d_col, s_col + ks * 16 + (t == 1 ? 8 : 0), wd + (t == 2 ? (D * 128) >> 4 : 0) + ((ks * 2048) >> 4),
                               idesc_f16(C) | B_MN_MAJOR, t != 2 || ks);
                mma_commit(bar_chain(chain));
                mma_commit(bar_wfree(i));
            }
            wait_mma(bar_chain(chain), phase);
            phase ^= 1;
            tc_fence_after();
            wait(bar_u(i), turn(i));
            // Delta (times what undoes the keys' scales) in place; U is the S rows'
            const float neg = -inv_row, g_chunk = co[2 * C];
            float m = 0.f;
            auto delta = [&](auto with_u) {
#pragma unroll 1
                for (int b = 0; b < 4; ++b) {
                    uint32_t v[16];
                    tmem_ld16(d_at + 16 * b, v);
                    float x[16];
                    if constexpr (decltype(with_u)::value) {
#pragma unroll
                        for (int e = 0; e < 16; ++e) x[e] = U_s[(16 * b + e) * D + r];
                    }
                    tc_wait_ld();
#pragma unroll
                    for (int e = 0; e < 16; e += 4) {
                        const float4 cc = *reinterpret_cast<const float4*>(co + C + 16 * b + e);
                        const float c4[4] = {cc.x, cc.y, cc.z, cc.w};
                        float b4[4];
                        if constexpr (decltype(with_u)::value) {
                            const float4 bb = *reinterpret_cast<const float4*>(co + 16 * b + e);
                            b4[0] = bb.x; b4[1] = bb.y; b4[2] = bb.z; b4[3] = bb.w;
                        }
#pragma unroll
                        for (int f = 0; f < 4; f += 2) {      // (neg and c are powers of two)
                            float2 y = __fmul2_rn(__fmul2_rn(make_float2(__uint_as_float(v[e + f]), __uint_as_float(v[e + f + 1])), make_float2(neg, neg)),
                                                  make_float2(c4[f], c4[f + 1]));
                            if constexpr (decltype(with_u)::value) y = __ffma2_rn(make_float2(b4[f], b4[f + 1]), make_float2(x[e + f], x[e + f + 1]), y);
                            m = fmaxf(fmaxf(m, fabsf(y.x)), fabsf(y.y));
                            v[e + f] = __float_as_uint(y.x);
                            v[e + f + 1] = __float_as_uint(y.y);
                        }
                    }
                    tmem_st16(d_at + 16 * b, v);
                }
            };
            if (is_s) delta(std::true_type{});
            else delta(std::false_type{});
            tc_wait_st();
            float sc, inv_d;
            pow2_scale(m, WIDE, sc, inv_d);
            // ... and as the next product's A operand: hi and lo in tensor memory; fp32 records: what is left in shared memory (not
            // for M's chain at dk = 128: S takes M's error times what is left of it after a segment)
            const bool three = Z::DP == 3 && (D < 128 || chain == 0);
#pragma unroll 1
            for (int b = 0; b < 4; ++b) {
                uint32_t v[16], w[16], low[8];
                tmem_ld16(d_at + 16 * b, v);
                tc_wait_ld();
                float x[16];
#pragma unroll
                for (int e = 0; e < 16; ++e) x[e] = __uint_as_float(v[e]);
                split16(x, sc, w, w + 8, KEEP_DELTA, Z::DP == 3 ? low : nullptr);
                tmem_st16(d_at + 16 * b, w);
                if (three) {
#pragma unroll
                    for (int e = 0; e < 2; ++e)
                        *reinterpret_cast<uint4*>(low_s + r * 128 + (((2 * b + e) ^ (r & 7)) << 4)) = make_uint4(low[4 * e], low[4 * e + 1], low[4 * e + 2], low[4 * e + 3]);
                }
            }
            tc_wait_st();
            if (Z::DP == 3) proxy_fence();
            tc_fence_before();
            if (bar_or(team, 128, fail ? 1 : 0)) { fail = true; break; }
            if (leader) arrive(bar_ufree(i));
            if (issuer) {                                     // Delta K over the S operand (read by now), small terms first
                tc_fence_after();
                const uint64_t kd = umma_desc_mn(smem_u32(K_s), TILE), ld = umma_desc(smem_u32(low_s));
                bool first = true;
                auto product = [&](int dp, int kp) {          // part dp of Delta, part kp of the keys
#pragma unroll
                    for (int ks = 0; ks < C / 16; ++ks) {
                        const uint64_t bd = kd + ((kp * KB * TILE) >> 4) + ((ks * 2048) >> 4);
                        if (dp == 2) mma_ss(s_col, ld + ((ks * 32) >> 4), bd, idesc_f16(D) | B_MN_MAJOR, !first);
                        else mma_ts(s_col, d_col + ks * 16 + dp * 8, bd, idesc_f16(D) | B_MN_MAJOR, !first);
                        first = false;
                    }
                };
                if (three) product(2, 0);
                if constexpr (PK > 1) {
                    product(1, 1);
                    if constexpr (PK > 2) product(0, 2);
                    product(0, 1);
                }
                product(1, 0);
                product(0, 0);
                mma_commit(bar_chain(chain));
                mma_commit(bar_kfree(ks_n));
            }
            wait_mma(bar_chain(chain), phase);
            phase ^= 1;
            tc_fence_after();
            largest = 0.f;
#pragma unroll
            for (int b = 0; b < D / 16; ++b) {
                uint32_t v[16];
                tmem_ld16(s_at + 16 * b, v);
                tc_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) {
                    S[16 * b + e] = fmaf(g_chunk, S[16 * b + e], __uint_as_float(v[e]) * inv_d);
                    largest = fmaxf(largest, fabsf(S[16 * b + e]));
                }
            }
        }
    }
    // (a CTA in which somebody gave up has nothing to hand on: it only keeps meeting the cluster)
    const bool lost = bar_or(CTA_BARRIER, Z::THREADS, fail ? 1 : 0);

    // =============================== SEGMENTS IN ORDER ===============================
    // S of the segments so far passes from CTA to CTA as the receiver's A operand (per row dk words in the order of the K
    // steps, and what undoes the row's scale), written to the receiver's shared memory over the cluster: what it then waits for
    // is the barrier and local reads.  (Read over the cluster by the receiver, a hop had their latency four to eight times over:
    // 2000 tokens x 8 heads of 128 x 128 bf16 69.1 -> 65.7 us, 400 tokens 38.7 -> 37.5, 3000 tokens x 8 heads of 64 x 64
    // 49.0 -> 47.4.)
    uint4* hand_s = reinterpret_cast<uint4*>(smem);           // [dk / 4][128 rows]
    uint8_t* M_s = smem + D * 128 * 4;                        // M_p as an MN-major B operand: [hi, lo][blocks of 64][dk rows][128 bytes]
    auto hand_over = [&]() {
        float m = 0.f, sc, inv;
#pragma unroll
        for (int d = 0; d < D; d += 2) m = fmaxf(fmaxf(m, fabsf(S[d])), fabsf(S[d + 1]));
        pow2_scale(m, WIDE, sc, inv);
        uint32_t peer, peer_inv;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(smem_u32(hand_s + r)), "r"(rank + 1));
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer_inv) : "r"(smem_u32(hinv_s + r)), "r"(rank + 1));
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(peer_inv), "f"(inv) : "memory");
#pragma unroll
        for (int b = 0; b < D / 16; ++b) {
            uint32_t w[16];
            split16(S + 16 * b, sc, w, w + 8);
#pragma unroll
            for (int q = 0; q < 4; ++q)
                asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(peer + (4 * b + q) * (128 * 16)), "r"(w[4 * q]), "r"(w[4 * q + 1]),
                             "r"(w[4 * q + 2]), "r"(w[4 * q + 3])
                             : "memory");
        }
    };
    if (P > 1) {
        if (!lost && has_m && (D < 128 || chain == 1)) {      // M with one scale for all its rows (every warp of the team comes along)
            float m = 0.f, sc, inv;
            if (is_m) {
#pragma unroll
                for (int d = 0; d < D; d += 2) m = fmaxf(fmaxf(m, fabsf(S[d])), fabsf(S[d + 1]));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (lane == 0) tok_s[warp & 3] = m;
            bar_or(team, 128, 0);
            m = fmaxf(fmaxf(tok_s[0], tok_s[1]), fmaxf(tok_s[2], tok_s[3]));
            pow2_scale(m, WIDE, sc, inv);
            if (leader) tok_s[4] = inv;
            if (is_m) {
#pragma unroll
                for (int b = 0; b < D / 16; ++b) {
                    uint32_t hi[8], lo[8];
                    split16(S + 16 * b, sc, hi, lo);
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int ch = 2 * b + e;
                        uint8_t* dst = M_s + (ch >> 3) * (D * 128) + mrow * 128 + (((ch & 7) ^ (mrow & 7)) << 4);
                        *reinterpret_cast<uint4*>(dst) = make_uint4(hi[4 * e], hi[4 * e + 1], hi[4 * e + 2], hi[4 * e + 3]);
                        *reinterpret_cast<uint4*>(dst + KB * D * 128) = make_uint4(lo[4 * e], lo[4 * e + 1], lo[4 * e + 2], lo[4 * e + 3]);
                    }
                }
            }
            proxy_fence();
        }
        cluster_sync();                                       // every CTA is through its chunks: its rings may be written
        if (!lost && rank == 0 && is_s) hand_over();
        // (one chain holds the S operand; its product lands in the other chain's columns, or beside it)
        const uint32_t o_at = D == 128 ? taddr + Z::CHAIN_COLS : d_at, o_col = D == 128 ? s_col + Z::CHAIN_COLS : d_col;
        for (int p = 1; p < P; ++p) {
            cluster_sync();
            if (lost || rank != p || chain != 0) continue;
            const int row = is_s ? r : 0;                     // (rows that are none come along with row 0's data)
            float inv = hinv_s[row];
#pragma unroll 2
            for (int b = 0; b < D / 16; ++b) {
                uint32_t w[16];
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const uint4 x = hand_s[(4 * b + q) * 128 + row];
                    w[4 * q] = x.x; w[4 * q + 1] = x.y; w[4 * q + 2] = x.z; w[4 * q + 3] = x.w;
                }
                tmem_st16(s_at + 16 * b, w);
            }
            tc_wait_st();
            tc_fence_before();
            bar_or(team, 128, 0);
            inv *= tok_s[4];
            if (issuer) {
                tc_fence_after();
                const uint64_t md = umma_desc_mn(smem_u32(M_s), D * 128);
#pragma unroll 1
                for (int t = 2; t >= 0; --t)                  // lo hi, hi lo, hi hi
#pragma unroll
                    for (int ks = 0; ks < D / 16; ++ks)
                        mma_ts(o_col, s_col + ks * 16 + (t == 2 ? 8 : 0), md + (t == 1 ? (KB * D * 128) >> 4 : 0) + ((ks * 2048) >> 4),
                               idesc_f16(D) | B_MN_MAJOR, t != 2 || ks);
                mma_commit(bar_chain(0));
            }
            wait_mma(bar_chain(0), phase);
            phase ^= 1;
            tc_fence_after();
#pragma unroll
            for (int b = 0; b < D / 16; ++b) {
                uint32_t v[16];
                tmem_ld16(o_at + 16 * b, v);
                tc_wait_ld();
#pragma unroll
                for (int e = 0; e < 16; ++e) S[16 * b + e] = fmaf(__uint_as_float(v[e]), inv, S[16 * b + e]);
            }
            tc_fence_before();
            if (p + 1 < P && is_s) hand_over();
        }
    }

    // =============================== RESULT ===============================
    if (!lost && rank == P - 1 && chain == 0) {
        float m = 0.f;
        if (is_s) {
            float4* dst = reinterpret_cast<float4*>(a.slot + ((long long)h * D + r) * D);
#pragma unroll
            for (int d = 0; d < D; d += 4) dst[d / 4] = make_float4(S[d], S[d + 1], S[d + 2], S[d + 3]);
#pragma unroll
            for (int d = 0; d < D; ++d) m = fmaxf(m, fabsf(S[d]));
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) tok_s[warp & 3] = m;
        bar_or(team, 128, 0);
        m = fmaxf(fmaxf(tok_s[0], tok_s[1]), fmaxf(tok_s[2], tok_s[3]));
        float sc, inv;
        pow2_scale(m, 11, sc, inv);                           // the head's operand scale (see Layout::s0_scale)
        if (leader) a.scale_out[h] = sc;
        if (a.s0_f16) {                                       // the tiled kernel's operand: value rows padded to 128
            char* dst = reinterpret_cast<char*>(a.s0_f16) + (long long)h * (128 * D * 2) + r * 128;
#pragma unroll
            for (int ch = 0; ch < D / 8; ++ch) {
                uint4 w = make_uint4(0u, 0u, 0u, 0u);
                if (is_s) {
                    const float* x = S + 8 * ch;
                    w = make_uint4(pack_f16x2(x[0] * sc, x[1] * sc), pack_f16x2(x[2] * sc, x[3] * sc), pack_f16x2(x[4] * sc, x[5] * sc),
                                   pack_f16x2(x[6] * sc, x[7] * sc));
                }
                *reinterpret_cast<uint4*>(dst + (ch >> 3) * (128 * 128) + (((ch & 7) ^ (r & 7)) << 4)) = w;
            }
        }
    }
    }   // chains
    if (fail && atomicCAS(a.status, ONELA_OK, ONELA_E_TIMEOUT) == ONELA_OK) a.status[1] = (int32_t)(blockIdx.x + gridDim.x * blockIdx.y);
    tc_fence_before();
    __syncthreads();
    if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(Z::TMEM_COLS) : "memory");
}

// How a prompt of `chunks` chunks is cut: P segments (a cluster of P CTAs per head), the first of `first` chunks, the
// others of `rest`.  Cost model, in chunk steps of a segment that carries M: a chunk of the first segment counts FIRST, one
// fold at the end FOLD, and `resident[P]` clusters of P run at a time.  FOLD, measured around the cuts it decides: 128 x 128 bf16,
// 250 tokens 29.8 us at 0.8, 31.4 at 0.4, 800 tokens 45.4 / 49.0; 64 x 64 fp32, 700 tokens 32.7 / 29.8, 2 x 1021 tokens 73.5 / 72.7;
// 32 x 32, 200 tokens 17.1 / 14.6.  One chain is cut no finer for that: every fold takes the whole state through two fp16 parts.
// Relative error against 64 bits at 0.8 / at 0.4, 64 x 64 without decay: 200 tokens 1.6e-7 / 2.4e-7, 300 1.6e-7 / 2.3e-7, 969
// 1.6e-7 / 1.9e-7; gates in [0.9, 1], 200 tokens 0.8e-7 / 1.1e-7.
struct Cut {
    int P, first, rest;
};
Cut cut_prompt(int chunks, int H, bool two_chains, const int* resident) {
    const double first_cost = two_chains ? 0.95 : 1.0, fold = 0.8;
    Cut best{1, chunks, 0};
    double best_cost = 1e30;
    for (int P = 1; P <= MAX_SEGMENTS && P <= chunks; ++P) {
        if (resident[P] < 1) continue;
        int rest = 0, first = chunks;
        if (P > 1) {
            rest = std::max(1, (int)(chunks / (P - 1 + 1.0 / first_cost) + 0.5));
            while (rest > 1 && (P - 1) * rest >= chunks) --rest;
            first = chunks - (P - 1) * rest;
            if (first < 1) continue;
        }
        const double waves = (double)((H + resident[P] - 1) / resident[P]);
        const double cost = waves * (std::max(first * first_cost, (double)rest) + (P - 1) * fold + 2.0);
        if (cost < best_cost) {
            best_cost = cost;
            best = Cut{P, first, rest};
        }
    }
    return best;
}

template <int D, typename T>
cudaError_t launch_dt(const PrefillArgs& args, cudaStream_t stream) {
    using Z = Shape<D, T>;
    auto kern = prefill_chunk_kernel<D, T>;
    // One-time set-up per instantiation and device: the shared-memory limit, and how many clusters of each size fit.
    constexpr int MAX_DEVICES = 64;
    static std::mutex setup_mutex;
    static int resident_of[MAX_DEVICES][MAX_SEGMENTS + 1] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX_DEVICES) return cudaErrorInvalidDevice;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(Z::THREADS);
    cfg.dynamicSmemBytes = Z::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int* resident = resident_of[dev];
    {
        std::lock_guard<std::mutex> lock(setup_mutex);
        if (resident[0] == 0) {
            cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, Z::SMEM);
            if (e != cudaSuccess) return e;
            for (int P = 1; P <= MAX_SEGMENTS; ++P) {
                attr[0].val.clusterDim.x = P;
                cfg.gridDim = dim3(P, 1);
                int clusters = 0;
                e = cudaOccupancyMaxActiveClusters(&clusters, kern, &cfg);
                if (e != cudaSuccess) return e;
                resident[P] = clusters;
            }
            resident[0] = 1;
        }
    }
    PrefillArgs a = args;
    const Cut cut = cut_prompt((a.n_tokens + C - 1) / C, a.H, Z::CHAINS == 2, resident);
    a.first = cut.first;
    a.rest = cut.rest;
    attr[0].val.clusterDim.x = cut.P;
    cfg.gridDim = dim3(cut.P, a.H);
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int D>
cudaError_t launch_d(const PrefillArgs& a, int32_t rec_dtype, cudaStream_t stream) {
    return rec_dtype == ONELA_DTYPE_BF16 ? launch_dt<D, __nv_bfloat16>(a, stream) : launch_dt<D, float>(a, stream);
}

}  // namespace

cudaError_t launch_prefill(const void* k, const void* v, const float* alpha, const float* beta, float* slot, float* scale_out,
                           uint16_t* s0_f16, int32_t* status, int32_t n_tokens, int32_t H, int32_t dk, int32_t dv, int32_t rec_dtype,
                           bool* supported, cudaStream_t stream) {
    const PrefillArgs a{k, v, alpha, beta, slot, scale_out, s0_f16, status, n_tokens, H, 0, 0};
    *supported = true;
    if (dk == 32 && dv == 32) return launch_d<32>(a, rec_dtype, stream);
    if (dk == 64 && dv == 64) return launch_d<64>(a, rec_dtype, stream);
    if (dk == 128 && dv == 128) return launch_d<128>(a, rec_dtype, stream);
    *supported = false;
    return cudaErrorInvalidValue;
}

}  // namespace onela

#ifdef ONELA_TEST_HOOKS
extern "C" int onela_testhook_prefill_drop(int on) { return (int)cudaMemcpyToSymbol(onela::g_hook_prefill_drop, &on, sizeof(int)); }
#endif
