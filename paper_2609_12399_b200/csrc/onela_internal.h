// Internal declarations shared by the host-side context (onela_api.cu) and the kernel files.
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "onela.h"

namespace onela {

// Device addresses of the sub-buffers carved out of the caller's workspace.
struct Layout {
    int32_t* status;   // [4]: code, detail, spare, spare
    unsigned long long* select_claims;   // [request], behind the status, zero from the start: whose select_scratch is (see onela_select.cu)
    int32_t* tables;   // [request][2][max_steps][max_beam] global slot ids (double-buffered per request)
    int32_t* sidx;     // [request][max_steps][max_beam] per (level, beam): index into the request's distinct-record list
    int32_t* ulist;    // [request][max_steps*max_beam] distinct record slots of the live chains, oldest level first
    int32_t* level_base;   // [request][max_steps] first slot of the request's records of each decode call
    int32_t* uoff;     // [request][max_steps+1] start of each level inside ulist (uoff[level+1] = end)
    int32_t* urep;     // [request][max_steps*max_beam] per distinct record: one live beam whose chain holds it
    uint8_t* sg8;      // [request][max_steps][sg_stride] sidx as bytes, rows padded with the last live beam's entry
    uint8_t* unode;    // [request][ONELA_UNODE_CAP][16] per distinct record: ancestors' list positions (bytes 0-7), level (byte 8)
    float* s0;         // [request][layer][head][dv*dk] fp32
    float2* gates;     // [layer][head][arena_slots] (alpha, beta)
    char* kv;          // [layer][head][arena_slots][dk + dv] in rec_dtype: one row = k | v of one record
                       // (grouped value heads: keys only, [layer][key head][arena_slots][dk])
    char* vv;          // grouped value heads only: values [layer][value head][arena_slots][dv]
    unsigned long long* select_scratch;   // [request][ONELA_SELECT_PARTS * ONELA_SELECT_CAP]: beam selection, the largest of shares of
                                          // the candidates; behind them candidates beyond its shared memory
    float* s0_scale;   // [request][layer][head]: the power of two that brings the head's largest |S_0| element into
                       // [2^11, 2^12) (1 for an all-zero or non-finite state); written with the state, read by the
                       // tensor-core kernel, whose fp16 operand it keeps in range
    uint16_t* s0_f16;  // configurations of the tiled tensor-core kernel only: [request][layer][head] the state as that
                       // kernel's MMA operand - fp16, times the head's operand scale, value rows padded to a multiple
                       // of 128, in tiles of 128 rows x 64 columns (16 KB, rows of 128 bytes, 16-byte chunks swizzled
                       // by the row) in the order [tile of rows][tile of columns]; written with the state
    size_t total_bytes;
};
// bytes of one head's operand copy (see Layout::s0_f16)
inline size_t s0_f16_head_bytes(int32_t dk, int32_t dv) { return (size_t)((dv + 127) / 128) * 128 * (size_t)dk * 2; }

struct BatchBases {
    int32_t base[ONELA_MAX_BATCH];  // first slot of this call's records, per request of the batch
};

// Everything a decode kernel needs, passed by value as the kernel parameter.
struct DecodeArgs {
    const void* q;          // [req_count][W][H][dk]
    void* out;              // [req_count][W][H][dv]
    const void* k_in;       // fused append: this call's records [req_count][W][H][dk], [..][dv], gates [..][H];
    const void* v_in;       //   null for a plain decode (the newest record is then read from the arena)
    const float* alpha_in;
    const float* beta_in;
    char* kv_out;           // fused append: arena plane to write (same plane as kv)
    float2* gates_out;
    const float* s0;        // store slot of (req_begin, layer)
    const char* kv;         // arena plane of this layer
    const float2* gates;    // gate plane of this layer
    const int32_t* table;   // current ancestry buffer of req_begin: [level][max_beam]
    int32_t* status;
    long long s0_req_stride;     // floats between consecutive requests' store slots (same layer)
    long long table_req_stride;  // ints between consecutive requests' tables
    long long arena_slots;
    const int32_t* sidx;    // distinct-record index of req_begin (see Layout)
    const int32_t* ulist;
    const int32_t* uoff;
    const uint8_t* sg8;     // byte copies of sidx and the per-record table (see Layout), of req_begin
    const uint8_t* unode;
    long long sg8_req_stride;
    int32_t sg_stride;
    long long sidx_req_stride, ulist_req_stride, uoff_req_stride;
    int32_t req_count, W, H, depth, max_beam;
    BatchBases bases;
    // grouped value heads (tensor-core kernel only; H above is then the number of VALUE heads): kv / kv_out are the
    // layer's key plane [Hk][arena_slots][dk], vv / vv_out its value plane [H][arena_slots][dv]; q and k_in have Hk heads
    const char* vv;
    char* vv_out;
    int32_t Hk, g, Hv;      // key heads, value tiles per key head, value heads (before they are cut into tiles)
    // ... and value widths of 256 / 512 (grouped or not): every value head is cut into `tiles` heads of 128 outputs, so
    // H = tiles * (value heads) and g = tiles * (value heads per key head); k_stride / v_stride: bytes between
    // consecutive slots of a key head's keys and of a value head's values (from kv and vv: one interleaved plane or two)
    int32_t tiles;
    long long k_stride, v_stride;
    // tensor-core kernel: per-head operand scale of S_0 (see Layout), entry of (req_begin, layer, head 0)
    const float* s0_scale;
    long long s0_scale_req_stride;
};

// Grouped value heads (Hv = g * Hk): what the grouped decode kernel needs.
struct GroupedArgs {
    const void* q;          // [req_count][W][Hk][dk]
    void* out;              // [req_count][W][Hv][dv]
    const float* s0;        // store slot of (req_begin, layer): [Hv][dv][dk]
    const char* kplane;     // this layer's keys   [Hk][arena_slots][dk]
    const char* vplane;     // this layer's values [Hv][arena_slots][dv]
    const float2* gates;    // this layer's gates  [Hv][arena_slots]
    const int32_t* table;   // current ancestry buffer of req_begin
    long long s0_req_stride, table_req_stride, arena_slots;
    int32_t req_count, W, Hk, g, depth, max_beam;
    BatchBases bases;
};
bool decode_grouped_supported(int32_t dk, int32_t dv);
cudaError_t launch_decode_grouped(const GroupedArgs& a, int32_t dk, int32_t dv, int32_t rec_dtype, int32_t out_dtype,
                                  cudaStream_t stream);
cudaError_t launch_append_grouped(const void* k, const void* v, const float* alpha, const float* beta, char* kplane,
                                  char* vplane, float2* gates, long long arena_slots, int32_t req_count, int32_t W,
                                  int32_t Hk, int32_t g, int32_t dk, int32_t dv, int32_t elem_bytes, const BatchBases& bases,
                                  cudaStream_t stream);

// Tiled tcgen05 decode kernel (onela_decode_tiled.cu): every supported shape from 64 x 64 up in either record dtype,
// grouped value heads or not.  Keys and values are addressed through planes and per-slot strides, so one struct serves
// the interleaved arena (kplane = the layer's k | v rows, vplane = kplane + dk elements, both strides dk + dv) and the
// split one (grouped value heads: two planes, strides dk and dv).
struct TiledArgs {
    const void* q;          // [req_count][W][Hk][dk]
    void* out;              // [req_count][W][Hv][dv]
    const void* k_in;       // fused append: this call's records [req_count][W][Hk][dk], [..][Hv][dv], gates [..][Hv], which
    const void* v_in;       //   the launch also writes to their arena slots; null for a plain decode (the newest record
    const float* alpha_in;  //   is then read from the arena)
    const float* beta_in;
    const float* s0;        // store slot of (req_begin, layer): [Hv][dv][dk]
    const float* s0_scale;  // operand scale of (req_begin, layer, value head 0) (see Layout)
    const char* s0_f16;     // operand copy of (req_begin, layer, value head 0) (see Layout::s0_f16)
    long long s0_f16_req_stride;   // bytes between consecutive requests' copies (same layer)
    char* kplane;           // key of (key head hk, slot) at kplane + ((hk * arena_slots + slot) * k_stride) elements
    char* vplane;           // value of (value head hv, slot) at vplane + ((hv * arena_slots + slot) * v_stride) elements
    float2* gates;          // [Hv][arena_slots]
    const int32_t* table;   // current ancestry buffer of req_begin
    int32_t* status;
    long long s0_req_stride, s0_scale_req_stride, table_req_stride, arena_slots, k_stride, v_stride;
    int32_t req_count, W, Hk, g, depth, max_beam;
    int32_t delta;          // 1: the arena keeps (alpha, delta, k) records and the launch replays both projections forward
    long long call_bytes;   // what a decode call of these requests touches in all layers: operand copies, tokens, records written, outputs
    BatchBases bases;
};
bool decode_tiled_supported(int32_t dk, int32_t dv);
cudaError_t launch_decode_tiled(const TiledArgs& a, int32_t dk, int32_t dv, int32_t rec_dtype, int32_t out_dtype,
                                cudaStream_t stream);

// Launch with programmatic stream serialisation: the kernel may start once every CTA of the previous kernel of the stream has
// let it (griddepcontrol.launch_dependents), and griddepcontrol.wait returns when that kernel has completed.
//   * Every CTA of a kernel launched this way waits.  So a kernel that has completed has seen its predecessor complete, and
//     past its own wait a kernel sees everything that earlier launches of the stream have written.
//   * Before its wait a kernel may count on nothing: the decode kernels let their dependents start before they have waited
//     themselves, and all others do so behind their wait but before they have written anything.  "Two launches ago" is no
//     guarantee either.
//   * The one thing read before the wait is the stored states (with their scales and operand copies), by the decode kernels.
//     They are written by the state calls alone; the host admits a decode only when a reorder of its request lies between
//     (finish_state_write restarts the request), and the index kernel of that reorder lets nothing start before its own wait,
//     so the states were complete when any kernel behind it started.
// The CUDA-core kernels for delta records and grouped heads, and export_chains are ordinary launches: they start when
// everything before them has completed, and what follows them starts when they have.
template <class... Params, class... Args>
cudaError_t launch_dependent(void (*kern)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, const Args&... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, kern, args...);
}

// Ancestry index update of one decode call (Eq. 5) and, on request, the distinct-record index of the new table's levels
// 0 .. depth-2 (the newest level is the beams' own records, all distinct): per level the sorted distinct slots, per beam
// where its ancestor sits in the request's concatenated list, per distinct record one of the live beams whose chain holds
// it (all such beams share its older ancestors); want_compact: byte-sized copies for the shared-chains kernel (see Layout).
// Integer work only.
cudaError_t launch_index(const Layout& lay, int32_t req_begin, int32_t req_count, const int32_t* parents, int32_t W_new, int32_t W_prev,
                         int32_t depth_old, int32_t max_beam, int32_t max_steps, const BatchBases& bases, bool want_index, bool want_compact,
                         cudaStream_t stream);
#define ONELA_UNODE_CAP 256
inline int32_t sg_row_stride(int32_t max_beam) { return (max_beam + 64 + 15) & ~15; }
cudaError_t launch_export_chains(const int32_t* table_cur, int32_t W, int32_t depth, int32_t max_beam,
                                 int32_t* slots_out, cudaStream_t stream);

// global beam selection: the W_new best (parent, code) pairs per request, best first (see onela_select.cu).
// At most ONELA_SELECT_PARTS * 4096 candidates per request.  `scratch` ([request][ONELA_SELECT_PARTS * ONELA_SELECT_CAP] 64-bit
// words, or null) takes the largest of shares of the candidates and, behind them, the candidates that the selection bound leaves where
// shared memory cannot hold them; `claims` ([request], see Layout): whose it is.
#define ONELA_SELECT_CAP 1024
#define ONELA_SELECT_PARTS 256
cudaError_t launch_select(const float* beam_scores, const float* cand_logp, int32_t req_count, int32_t W_prev, int32_t C,
                          int32_t W_new, unsigned long long* scratch, unsigned long long* claims, int32_t* parents, int32_t* codes,
                          float* scores, cudaStream_t stream);
int select_launches(long long candidates, int32_t W_new);      // kernels a call with a scratch launches

// record / state kernels
cudaError_t launch_append(const void* k, const void* v, const float* alpha, const float* beta, char* kv_plane,
                          float2* gate_plane, long long arena_slots, int32_t req_count, int32_t W, int32_t H,
                          int32_t dk, int32_t dv, int32_t elem_bytes, const BatchBases& bases,
                          cudaStream_t stream);
// copies n_heads states of dv x dk floats and leaves each head's operand scale (see Layout::s0_scale) in scale_out and,
// f16_out not null, the tiled kernel's operand copy (see Layout::s0_f16) there
cudaError_t launch_store_state(const float* S0_in, float* slot, float* scale_out, uint16_t* f16_out, long long n_heads, int32_t dk, int32_t dv,
                               cudaStream_t stream);
cudaError_t launch_export_state(const float* slot, float* S0_out, int32_t H, int32_t dk, int32_t dv, cudaStream_t stream);
// Eq. 1 from the zero state over a prompt, into the store slot of one (request, layer), with the heads' operand scales and
// (s0_f16 not null) the tiled kernel's operand copies (onela_prefill.cu).  Returns cudaErrorInvalidValue with *supported =
// false when (dk, dv) has no instantiation.
cudaError_t launch_prefill(const void* k, const void* v, const float* alpha, const float* beta, float* slot, float* scale_out,
                           uint16_t* s0_f16, int32_t* status, int32_t n_tokens, int32_t H, int32_t dk, int32_t dv, int32_t rec_dtype,
                           bool* supported, cudaStream_t stream);

// decode kernels
cudaError_t launch_decode_generic(const DecodeArgs& a, int32_t dk, int32_t dv, int32_t rec_dtype,
                                  int32_t out_dtype, bool* supported, cudaStream_t stream);
bool decode_generic_supported(int32_t dk, int32_t dv, int32_t rec_dtype);
// tcgen05 tensor-core kernel (sm_100a): dk = dv = 128, bf16 records
// forward projection replay over (alpha, delta, k) records (ONELA_FLAG_GTR_DELTA): append + decode of one layer
cudaError_t launch_decode_gtr(const DecodeArgs& a, int32_t dk, int32_t dv, int32_t rec_dtype, int32_t out_dtype,
                              bool* supported, cudaStream_t stream);
bool decode_sm100_supported(int32_t dk, int32_t dv, int32_t rec_dtype);
// delta_records: the arena keeps (alpha, delta, k) and the launch replays both projections forward (fused append only)
cudaError_t launch_decode_sm100_ws(const DecodeArgs& a, int32_t out_dtype, bool grouped, bool delta_records, cudaStream_t stream);

// Contiguous ranges of beam groups, one per CTA of a persistent decode kernel (host-side partitioner in
// onela_decode_sm100.cu): CTA c works on groups [begin[c], begin[c + 1]).
constexpr int DECODE_MAX_CTAS = 160;
struct DecodePartition {
    int32_t begin[DECODE_MAX_CTAS + 1];
};
// group_cost / seg_cost: relative cost of one group and of starting a (request, head) segment.  Returns the CTA count.
int make_decode_partition(int total_groups, int groups_per_pair, int sms, int group_cost, int seg_cost, DecodePartition* part);
int decode_sm_count();

// tcgen05 kernel for chains with heavily shared ancestors (dk = dv = 128, bf16 records, one key head per value head):
// the older levels of all chains are applied in compact form on the tensor cores (see onela_decode_wy.cu).
// Usable when every request of the call has at most WY_MAX_NODES distinct older records, at most WY_MAX_DEEP of them
// older than the beams' parents, and 2 <= depth <= WY_MAX_LEVELS + 1; the kernel checks the first two on the device.
constexpr int WY_MAX_NODES = 160, WY_MAX_DEEP = 64, WY_MAX_LEVELS = 8;
cudaError_t launch_decode_wy(const DecodeArgs& a, int32_t out_dtype, cudaStream_t stream);

}  // namespace onela
