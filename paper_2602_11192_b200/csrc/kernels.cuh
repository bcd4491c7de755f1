// Launch interfaces of the library's kernels (all sm_100a, all launched by api.cu).
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/melinoe_moe.h"
#include "moe_types.cuh"

namespace melinoe {

void count_launch();
// Programmatic stream serialisation for the decode kernels (on unless MELINOE_MOE_NO_PDL is set in the environment).
bool pdl_enabled();

// ---- router (Eq. 1): logits, top-k, gates, and per block how many of its tokens chose each expert
struct RouterShape {
    int tokens_per_warp, n_eg;       // tokens and expert groups of a warp's tile
    int tokens_per_block, n_blocks;
};
RouterShape router_shape(int T, int E, int n_sms);
// block_counts [n_blocks][kMaxExperts]
cudaError_t router_configure();
cudaError_t launch_router(cudaStream_t stream, const RouterShape &shape, const uint16_t *x, const uint16_t *w_r,
                          const float *bias, const int32_t *token_seq, int T, int d, int E, int k,
                          int32_t *idx, float *gate, float *logits_out, int32_t *block_counts);

// Calls of at most so many tokens, of bf16 slots, have their rows fetched by index in the grouped GEMM (and the lists for it made with
// the plan), others' are copied into the experts' order first.  A fetch by index takes TMA some 28 cycles per four rows: beyond 32
// rows of a CTA it is slower than the weights' (d 2048, d_ff 1024, 64 experts, 8 per token, 4 layers, us a pass, copied and
// by index: 16 tokens 254 and 240, 64 tokens 278 and 270, 128 tokens 293 and 300, 290 tokens 370 and 435).  Expansion of 4-bit
// codes hides what the copy takes (16 tokens 57 and 58).
constexpr int kIndexedTokens = 64;

// ---- planning: gather lists, LRU slot lookup, miss queue, statistics
struct PlanParams {
    const int32_t *idx;
    int T, k, E, C, n_shared;
    DevCache *cache;
    DevPlan *plan;
    const char *slots;        // device cache (slot s at slots + s * slot_stride)
    size_t slot_stride;
    const char *const *shared_blobs;
    const char *const *host_blobs;   // device array [E]: every expert's blob in the host store as the device
                                     // sees it (null entries, or a null array: the store cannot be read from kernels)
    int32_t *perm, *inv_pos, *tok_of_sorted;
    HostPlan *hplan;          // page-locked host memory (device-visible address)
    uint32_t gmax;            // compute groups the caller has room for
    uint32_t call_seq;        // written to the miss queue's seq word when the record is complete
    int fast;                 // fused planner: 1 = the call is served by one decode launch that fetches the missed experts itself,
                              // 2 = by one launch per compute group, the first of which is queued already
    int policy;               // MELINOE_POLICY_LRU or MELINOE_POLICY_COUNT
    float gamma;              // decay of the count policy
    melinoe_moe_stats *stats; // may be null
    size_t expert_bytes;
    // request trace (melinoe_moe_set_trace): this call's record, or null; see trace_layout()
    char *trace_rec;
    int trace_max_tokens;
    const float *gate;        // [T][k], for the trace record of calls planned by the general kernel
    // general kernel: the router's counts per block; become the pairs of each expert in the blocks before
    int32_t *block_counts;
    int n_blocks;
};
// What the general kernels want to know besides.
struct PromptParams {
    int tokens_per_block;     // of the router
    int lists;                // the planning kernel makes the token lists, too (each of the router's blocks had one token)
    float *row_gate;          // null, or the gate of the pair at every sorted position, 1 for a shared expert's rows
    GemmCounters *counters;   // null, or the grouped GEMM's
    int *err;                 // device error word (0 = ok)
};
// Layout of one request-trace record for a layer of n_experts experts and top_k, max_tokens tokens.
struct TraceLayout {
    size_t req_off, idx_off, gate_off, bytes;
};
__host__ __device__ inline TraceLayout trace_layout(int n_experts, int top_k, int max_tokens)
{
    TraceLayout t;
    t.req_off = sizeof(melinoe_moe_trace_header);
    t.idx_off = t.req_off + (size_t)n_experts * sizeof(melinoe_moe_request);
    t.gate_off = t.idx_off + (size_t)max_tokens * top_k * sizeof(int32_t);
    t.bytes = (t.gate_off + (size_t)max_tokens * top_k * sizeof(float) + 15) / 16 * 16;
    return t;
}
cudaError_t launch_plan(cudaStream_t stream, const PlanParams &p, const PromptParams &q);

// ---- router and planning in one kernel (one thread-block cluster), for calls of at most 8 tokens
// Loads the kernels' code.  Called ahead of ffn_decode_configure: with the two kernels of a decode call in memory side by side, and not
// the grouped GEMM's between them, their instructions stay out of one another's way (a call of a tiny layer 12.75 -> 12.55 us).
cudaError_t route_plan_small_configure();
bool route_plan_small_supported(int T, int k, int d);
cudaError_t launch_route_plan_small(cudaStream_t stream, const uint16_t *x, const uint16_t *w_r, const float *bias,
                                    const int32_t *token_seq, int n_seq, int d, int32_t *idx, float *gate, float *logits_out,
                                    const PlanParams &p);

// ---- decode expert FFN (Eq. 3) with the gate-weighted combine (Eq. 2) fused in, for up to 8 tokens per launch
struct DecParams {
    const DevPlan *plan;
    const uint16_t *x;               // hidden [T][d] bf16
    const int32_t *idx;              // [T][k]
    const float *gate;               // [T][k]
    long long *yacc;                 // [8][d] output accumulator words of the launch; all zero between launches
    float *ybuf;                     // [T][d] fp32: sum over the earlier launches of the same tokens (group mode)
    uint16_t *out;                   // [T][d] bf16
    unsigned *sync;                  // counters: of every consumer warp's columns, and of the launch (all zero between launches)
    uint32_t call_seq;               // the call's sequence number: the plan is ready when the low half of plan->ready equals it
    int *err;                        // device error word (0 = ok)
    unsigned long long *trace;       // null, or 8 clock stamps per CTA of the most recent launch
    int d, F, E, k, T, n_shared;
    int group;                       // -1: every request of the call in this one launch, the missed experts read
                                     // straight from the host store; g >= 0: compute group g only, from the slots
    int chunk, n_chunks;             // tokens [8 * chunk, 8 * chunk + 8) of the call; launches the call is made in
    int write_back;                  // group -1: store the fetched experts that stay resident into their slots
    int wait_prior;                  // the kernel ahead in the stream is another launch of the same call (it uses the
                                     // same accumulator): wait for that grid to finish before anything else
    int fmt;                         // 0: bf16 blobs, 1: 4-bit blobs
    int fast;                        // directly behind the fused planner: the launch's requests are plan->fast or plan->one; those of
                                     // group 0 only if the plan's word says so, or plan->one does
};
// The counters of DecParams::sync, a cache line each: where the CTAs end together, sixteen counters in one line cost a
// short launch about a microsecond.
constexpr int kSyncPitch = 32, kSyncCounters = 17;
struct DecLaunchCfg {
    int grid;                        // one CTA per SM
    size_t max_smem;                 // dynamic shared memory the kernel may use
    bool pdl;                        // launch with programmatic stream serialisation
};
// Shape of the shared-memory ring for one launch.
struct DecGeometry {
    int n_warps;                     // consumer warps (16)
    int tile_rows;                   // f rows per tile = ring stage: at most 8
    int n_stages;
    int row_bytes;                   // bytes of one f row of the blob (its W_g, W_u and W_d^T rows)
    int stage_bytes;
    int x_pitch;                     // bytes between token rows of the staged hidden states
    int tokens;                      // tokens of the launch (1..8)
    int x_tmem;                      // 1: the hidden states' operand fragments live in tensor memory, not in shared memory
    int groups;                      // groups of consumer warps, each with tiles (and so stages) of its own
    size_t smem_bytes;
};
cudaError_t ffn_decode_configure(int n_sms, size_t max_smem, DecLaunchCfg *cfg);
bool ffn_decode_supported(int d, int F);
bool ffn_decode_supported_q4(int d, int F);
// min_req: requests that the call has for certain (its top_k and the shared experts; a launch of one compute group may have fewer)
cudaError_t ffn_decode_geometry(const DecLaunchCfg &cfg, int d, int F, int tokens, int fmt, int min_req, DecGeometry *geo);
cudaError_t launch_ffn_decode(cudaStream_t stream, const DecLaunchCfg &cfg, const DecGeometry &geo,
                              const DecParams &p);

// ---- grouped GEMM expert FFN on tcgen05 for calls with many tokens per expert (prefill)
// Tensor maps in device memory, in this order:
enum {
    kMapXs0 = 0, kMapHs0 = 3,                                        // activations: boxes of 32, 64, 128 rows x 64 columns
    kMapSlots0 = 6,                                                  // weights of all slots for GEMM 1 and for GEMM 2 (see ffn_gemm.cu)
    kMapShared0 = 8,                                                 // per shared expert: the same two views
    kMapCount = kMapShared0 + 2 * kMaxShared
};
struct GemmParams {
    // by index: the call's hidden states, boxes of one row x 64 columns, and the token of every sorted row; otherwise the gather
    // kernel has made Xs
    CUtensorMap x_map;
    const int32_t *tok_of_sorted;
    int by_index;
    uint32_t call_seq;               // the plan is ready when the low half of plan->ready equals it
    const DevPlan *plan;
    GemmCounters *counters;
    const CUtensorMap *maps;         // device array of kMapCount tensor maps
    uint16_t *hs;                    // h, [sorted rows][F] bf16; with 4-bit slots times the row's gate
    const float *row_gate;           // 4-bit slots: gate of every sorted row (PromptParams::row_gate)
    float *zs;                       // expert outputs, [sorted rows][d] fp32
    int *err;
    int group, d, F, E;
    // 4-bit slots: the blobs themselves (their scales are read directly) and the bytes of one hidden unit
    const char *slots;
    size_t slot_stride;
    const char *const *shared_blobs;
    int unit_bytes;
};
bool ffn_gemm_supported(int d, int F);
cudaError_t ffn_gemm_configure();
// Token lists (perm, inv_pos, tok_of_sorted, row_gate) of a call planned by the general kernel that did not make them
// itself, and, unless xs is null, the gathered activations, in the blocks the router worked in.  permute: elements j
// and j + 4 of every eight side by side (the order in which 4-bit codes expand).
cudaError_t launch_gather_rows(cudaStream_t stream, int n_sms, const PlanParams &p, const PromptParams &q, const uint16_t *x, uint16_t *xs, int d,
                               bool permute);
// Both GEMMs of a compute group, in one launch or two, by CTA pairs or single CTAs (single_only: bf16 slots, too).  fmt: what the slots
// hold, 0 = bf16 blobs, 1 = 4-bit blobs; T, k: of the call
cudaError_t launch_ffn_gemm(cudaStream_t stream, int n_sms, int fmt, bool single_only, const GemmParams &p, int T, int k);
// gate null: the rows are weighted already
cudaError_t launch_combine_rows(cudaStream_t stream, const DevPlan *plan, const float *gate, const int32_t *inv_pos,
                                const float *zs, uint16_t *out, int T, int d, int k, int n_shared, int n_sms);

// ---- preload (Eq. 5): cache requests of a list of experts, and the copy of the missing ones into their slots
struct PreloadParams {
    DevCache *cache;
    PreloadList *list;               // device
    PreloadList *host_list;          // page-locked host memory as the device sees it, or null
    int32_t ids[kMaxExperts];
    int n, C, policy;
    uint32_t seq;
};
struct FetchParams {
    const PreloadList *list;
    const char *const *host_blobs;   // device array: the host store as the device sees it
    char *slots;
    size_t slot_stride;
    int rows, row_bytes;             // rows of one expert blob (d_ff) and their size
    int rows_per_piece, piece_bytes; // rows copied at a time (at most 48 KB)
    int *err;
};
cudaError_t launch_preload_plan(cudaStream_t stream, const PreloadParams &p);
cudaError_t launch_fetch_experts(cudaStream_t stream, int n_sms, const FetchParams &p);

// ---- cache-miss proxies of a recorded routing trace (Section 3.1, Definition C.1)
cudaError_t launch_miss_proxies(cudaStream_t stream, const int32_t *idx, int n_layers, int T, int K, int E,
                                const melinoe_proxy_config *cfgs, int n_cfg, int n_sms, double *soft_mean, long long *hard_total);

// ---- 4-bit host store: expand one 4-bit expert (layout in dequant.cu) into a bf16 slot
// ---- decode-sized input from device-mapped host memory into device memory (bytes % 16 == 0)
cudaError_t launch_stage_in(cudaStream_t stream, const void *src_mapped, void *dst, size_t bytes);
cudaError_t launch_dequant_q4(cudaStream_t stream, const void *q4_blob, void *slot, int d, int F, int n_sms);

}  // namespace melinoe
