// Ancestry index kernels (paper Section 3.3, Eq. 5).  Integer work only: beam selection prunes,
// reorders and fans out beams by rewriting slot ids; no transition record is moved or copied.
//
// Table layout per request: two buffers [max_steps][max_beam] of int32 global slot ids, level-major
// (row `level` holds, for every live beam, the slot of its ancestor's record written at decode call
// `level`; the last live row is the beam's own record).  Buffer (depth-1)&1 is current at depth `depth`.
#include "onela_internal.h"

namespace onela {

namespace {

// One CTA per request: Eq. 5 for every (level, beam) of the new table, and - `want_index`, for the decode kernel's staging
// of shared ancestors - the distinct-record index of the levels older than the beams' own records: which slots of a level
// some live chain refers to, in increasing order, and every beam's position in the request's concatenated list.
// The slots of one level of one request are consecutive (level_base keeps the first), so a level's records are a bitmap of
// max_beam bits: marks are atomic ORs into shared memory, a warp per level turns them into running counts, and a position
// is a count plus the bits below - three barriers for all levels.  (As two kernels, with one prefix sum over max_beam marks
// and seven barriers per level, the pair took 5.5 us at depth 2 and 19 us at depth 8 for 4 x 512 beams; 2.9 - 4.1 us here.)
// What is left is latency: parents, then the old table's slots beside their levels' first slots, two barriers, the stores.  The
// parents are asked for before anything else, nothing stands between them and the table, a thread has its beam's slots in
// registers for the positions, and there are no more threads than beams: 0.9 us less per launch at 128 beams and depth 2 - 4,
// 2.1 us less at 4 x 512 beams and depth 2 - 8 than with a barrier before the parents, slots read back and 1024 threads.
// Levels beyond `chunk` are taken in further rounds of the same three steps.
struct IndexArgs {
    int32_t* tables;            // [request][2][max_steps][max_beam]
    const int32_t* parents;     // [request][W_new], null at depth 0
    int32_t *level_base, *sidx, *ulist, *urep, *uoff;
    uint8_t *sg8, *unode;       // shared-chains kernel only, else null
    int32_t* status;
    long long table_req_stride, sidx_req_stride, uoff_req_stride, sg8_req_stride;
    int32_t sg_stride, W_new, W_prev, depth_old, max_beam, max_steps, chunk, want_index;
    BatchBases bases;
};

__global__ void __launch_bounds__(1024) index_kernel(const __grid_constant__ IndexArgs a) {
    extern __shared__ uint32_t bits[];                     // [chunk][words] marks, then [chunk][words] running counts
    __shared__ int32_t s_count[32], s_base[32], s_off;
    const int r = blockIdx.x, tid = threadIdx.x, threads = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int words = (a.max_beam + 31) / 32, levels = a.depth_old, chunk = a.chunk;
    uint32_t* counts = bits + chunk * words;
    const long long buf = (long long)a.max_steps * a.max_beam;
    int32_t* newt = a.tables + r * a.table_req_stride + (a.depth_old & 1) * buf;
    const int32_t* oldt = a.tables + r * a.table_req_stride + ((a.depth_old - 1) & 1) * buf;
    int32_t* lbase = a.level_base + (long long)r * a.max_steps;
    int32_t *sidx = a.sidx + r * a.sidx_req_stride, *ulist = a.ulist + r * a.sidx_req_stride, *urep = a.urep + r * a.sidx_req_stride;
    int32_t* uoff = a.uoff + r * a.uoff_req_stride;
    if (a.want_index)
        for (int i = tid; i < min(chunk, levels) * words; i += threads) bits[i] = 0u;
    if (tid == 0) s_off = 0;
    __syncthreads();
    // the caller's parents, the old table and every array written here belong to earlier launches of the stream
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // h_t(b, t): the record a beam is about to append lives at base(req, t) + b
    const int p_first = levels > 0 && tid < a.W_new ? a.parents[(long long)r * a.W_new + tid] : 0;
    for (int b = tid; b < a.W_new; b += threads) newt[(long long)a.depth_old * a.max_beam + b] = a.bases.base[r] + b;
    if (tid == 0) {
        lbase[a.depth_old] = a.bases.base[r];
        if (a.want_index) uoff[0] = 0;
    }
    for (int l0 = 0; l0 < levels; l0 += chunk) {
        const int n = min(chunk, levels - l0);
        if (a.want_index && l0 > 0) {
            __syncthreads();
            for (int i = tid; i < n * words; i += threads) bits[i] = 0u;
            __syncthreads();
        }
        if (tid < n) s_base[tid] = lbase[l0 + tid];            // (for the positions; the marks read it beside the old table)
        int32_t slot[8];
        // Eq. 5: the child inherits its parent's row (levels < t-1) and, at level t-1, the parent's own slot, which is the
        // last entry of the parent's row - one gather covers both cases.
        for (int b = tid; b < a.W_new; b += threads) {
            int p = b == tid ? p_first : a.parents[(long long)r * a.W_new + b];
            if ((unsigned)p >= (unsigned)a.W_prev) {
                if (atomicCAS(a.status, ONELA_OK, ONELA_E_DEVICE_CHECK) == ONELA_OK) a.status[1] = p;
                p = 0;
            }
            for (int l1 = 0; l1 < n; l1 += 8) {             // eight gathers in flight
                int32_t first[8];
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (l1 + e < n) {
                        slot[e] = oldt[(long long)(l0 + l1 + e) * a.max_beam + p];
                        first[e] = lbase[l0 + l1 + e];
                    }
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int l = l1 + e;
                    if (l >= n) break;
                    newt[(long long)(l0 + l) * a.max_beam + b] = slot[e];
                    if (a.want_index) {
                        const int key = slot[e] - first[e];
                        atomicOr(&bits[l * words + (key >> 5)], 1u << (key & 31));
                    }
                }
            }
        }
        if (!a.want_index) continue;
        __syncthreads();
        // counts of the records before each word, level by level (one warp each); then the levels' offsets in the list
        for (int l = warp; l < n; l += threads / 32) {
            int32_t run = 0;
            for (int w0 = 0; w0 < words; w0 += 32) {
                const int w = w0 + lane;
                const int32_t mine = w < words ? __popc(bits[l * words + w]) : 0;
                int32_t incl = mine;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int32_t t = __shfl_up_sync(0xffffffffu, incl, o);
                    if (lane >= o) incl += t;
                }
                if (w < words) counts[l * words + w] = run + incl - mine;
                run += __shfl_sync(0xffffffffu, incl, 31);
            }
            if (lane == 0) s_count[l] = run;
        }
        __syncthreads();
        int32_t off = s_off;                               // of the chunk's first level
        const int32_t c_mine = lane < n ? s_count[lane] : 0;
        int32_t c_incl = c_mine;                           // every warp scans the (at most 32) levels for itself
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t t = __shfl_up_sync(0xffffffffu, c_incl, o);
            if (lane >= o) c_incl += t;
        }
        if (warp == 0 && lane < n) uoff[l0 + lane + 1] = off + c_incl;
        const bool kept = a.W_new <= threads && n <= 8;   // this thread's slots are still in its registers
        for (int b0 = 0; b0 < a.W_new; b0 += threads) {       // (whole warps stay in the loop for the shuffles)
            const int b = b0 + tid;
            for (int l1 = 0; l1 < n; l1 += 8) {
#pragma unroll
                for (int e = 0; e < 8; ++e)                // (written by this thread)
                    if (!kept) slot[e] = l1 + e < n && b < a.W_new ? newt[(long long)(l0 + l1 + e) * a.max_beam + b] : 0;
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                    const int l = l1 + e;
                    if (l >= n) break;
                    const int32_t first = off + __shfl_sync(0xffffffffu, c_incl - c_mine, l);
                    if (b < a.W_new) {
                        const int key = slot[e] - s_base[l];
                        const uint32_t word = bits[l * words + (key >> 5)];
                        const int32_t pos = first + counts[l * words + (key >> 5)] + __popc(word & ((1u << (key & 31)) - 1u));
                        sidx[(long long)(l0 + l) * a.max_beam + b] = pos;
                        ulist[pos] = slot[e];              // (the beams that share a record write the same slot,
                        urep[pos] = b;                     //  and any of them will do as its representative)
                    }
                }
            }
        }
        off += __shfl_sync(0xffffffffu, c_incl, 31);
        __syncthreads();
        if (tid == 0) s_off = off;
    }
    if (!a.want_index || !a.sg8) return;
    // Compact copies for the shared-chains decode kernel (meaningful while the request has at most 255 distinct
    // records; the kernel checks the count): every beam's list position per level as one byte, rows padded with the
    // last live beam's; and per distinct record its level and its ancestors' list positions (through one of the
    // beams that hold it).
    __syncthreads();
    const int32_t total = s_off;
    uint8_t* sg8 = a.sg8 + r * a.sg8_req_stride;
    for (int i = tid; i < levels * a.sg_stride; i += threads) {
        const int level = i / a.sg_stride, b = i - level * a.sg_stride;
        sg8[i] = (uint8_t)sidx[(long long)level * a.max_beam + min(b, a.W_new - 1)];
    }
    uint8_t* unode = a.unode + (long long)r * (ONELA_UNODE_CAP * 16);
    for (int j = tid; j < min(total, ONELA_UNODE_CAP); j += threads) {
        int lv = 0;
        for (int l = 1; l < levels; ++l) lv += (j >= uoff[l]) ? 1 : 0;
        const int rp = urep[j];
        uint32_t w[4] = {0u, 0u, (uint32_t)lv, 0u};
        for (int l = 0; l < min(lv, 8); ++l)
            w[l >> 2] |= ((uint32_t)sidx[(long long)l * a.max_beam + rp] & 0xffu) << (8 * (l & 3));
        reinterpret_cast<uint4*>(unode)[j] = make_uint4(w[0], w[1], w[2], w[3]);
    }
}

__global__ void __launch_bounds__(256) export_chains_kernel(const int32_t* __restrict__ table, int32_t W, int32_t depth,
                                                            int32_t max_beam, int32_t* __restrict__ out) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= W * depth) return;
    const int b = i / depth, level = i % depth;
    out[i] = table[(long long)level * max_beam + b];
}

}  // namespace

cudaError_t launch_index(const Layout& lay, int32_t req_begin, int32_t req_count, const int32_t* parents, int32_t W_new, int32_t W_prev,
                         int32_t depth_old, int32_t max_beam, int32_t max_steps, const BatchBases& bases, bool want_index, bool want_compact,
                         cudaStream_t stream) {
    IndexArgs a{};
    a.table_req_stride = 2LL * max_steps * max_beam;
    a.sidx_req_stride = (long long)max_steps * max_beam;
    a.uoff_req_stride = max_steps + 1;
    a.sg_stride = sg_row_stride(max_beam);
    a.sg8_req_stride = (long long)max_steps * a.sg_stride;
    a.tables = lay.tables + req_begin * a.table_req_stride;
    a.parents = parents;
    a.level_base = lay.level_base + (long long)req_begin * max_steps;
    a.sidx = lay.sidx + req_begin * a.sidx_req_stride;
    a.ulist = lay.ulist + req_begin * a.sidx_req_stride;
    a.urep = lay.urep + req_begin * a.sidx_req_stride;
    a.uoff = lay.uoff + req_begin * a.uoff_req_stride;
    if (want_compact) {
        a.sg8 = lay.sg8 + req_begin * a.sg8_req_stride;
        a.unode = lay.unode + (size_t)req_begin * ONELA_UNODE_CAP * 16;
    }
    a.status = lay.status;
    a.W_new = W_new;
    a.W_prev = W_prev;
    a.depth_old = depth_old;
    a.max_beam = max_beam;
    a.max_steps = max_steps;
    a.want_index = want_index && depth_old >= 1;
    a.bases = bases;
    // levels per round: two words per 32 beams and level, at most 32 levels (one per lane) and what a launch gets without
    // asking, 48 KB less the kernel's static shared memory - one level's bitmap fits up to 192 000 beams
    constexpr size_t ROOM = 47 * 1024;
    const size_t per_level = 2 * sizeof(uint32_t) * (size_t)((max_beam + 31) / 32);
    int chunk = (int)(ROOM / per_level);
    chunk = chunk < 1 ? 1 : chunk > 32 ? 32 : chunk;
    if (chunk > depth_old) chunk = depth_old > 0 ? depth_old : 1;
    a.chunk = chunk;
    const size_t smem = a.want_index ? per_level * chunk : 0;
    if (smem > ROOM) {
        cudaError_t e = cudaFuncSetAttribute(index_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    // a thread per beam; at least eight warps (one counts a level)
    const int threads = W_new > 1024 ? 1024 : W_new < 256 ? 256 : (W_new + 31) / 32 * 32;
    return launch_dependent(index_kernel, dim3(req_count), dim3(threads), smem, stream, a);
}

cudaError_t launch_export_chains(const int32_t* table_cur, int32_t W, int32_t depth, int32_t max_beam,
                                 int32_t* slots_out, cudaStream_t stream) {
    const int n = W * depth;
    export_chains_kernel<<<(n + 255) / 256, 256, 0, stream>>>(table_cur, W, depth, max_beam, slots_out);
    return cudaGetLastError();
}

}  // namespace onela
