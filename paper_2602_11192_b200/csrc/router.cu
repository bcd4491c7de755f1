// Router: logits, top-k with lowest-index tie-breaking, renormalised gates (Eq. 1), for calls that the fused decode
// planner does not take; and how often each block's tokens chose each expert, from which the planning kernel makes
// the token lists.
//
// The selected indices are an integer result that must agree bit for bit with a CPU
// evaluation, so the fp32 logit is summed in one fixed order: element j belongs to lane
// (j mod 256) / 8; every lane adds its elements in increasing j into one accumulator
// (products of two bf16 values are exact in fp32, so fused or unfused multiply-add give the
// same bits); the 32 lane sums are folded by xor-butterflies with strides 16, 8, 4, 2, 1; the
// bias is added last.  That is exactly one 16-byte load per lane per 256 columns.
//
// A warp holds TT tokens x EE experts in registers; a block is n_eg expert groups x TG token groups of warps, so
// every block reads the whole router matrix once.  What bounds it: for a few hundred tokens the latency of those
// reads (TT = 1 or 2, EE = 4: many warps, CH pieces of 256 columns in flight), for thousands the FMA pipe and the issue
// slots: 4 x 8 gives 256 multiply-adds per 12 loads and 128 conversions, and fma.rn.f32x2 (two experts at a time, each rounded
// on its own: the same bits) halves what the multiply-adds take of the issue slots; an SM holds only 16 such warps,
// so their operands go through a ring in shared memory (cp.async) instead of waiting for the loads.  The butterfly folds
// TT * EE values at once by exchanging halves: 31 shuffles for 32 values instead of 160.  The bias is added by
// the warp that selects, a lane per expert.  Measured (d 2048, 64 experts): 128 tokens 16.7 -> 8 us, 512 tokens
// 38 -> 17 us, 8192 tokens 193 -> 93 us (FMA pipe half busy); 4096 tokens, d 4096, 16 experts 119 -> 26 us.
#include "kernels.cuh"

namespace melinoe {

namespace {

__device__ __forceinline__ float bf16lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

__device__ __forceinline__ uint64_t pack2(float lo, float hi)
{
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void fma2(uint64_t &acc, uint64_t a, uint64_t b)
{
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// Unsigned numbers (none of them 0) in the order of floats, both zeros alike, and back.  A NaN (the sum
// makes every one the same) is above all: the order is total, whatever the logits are.
__device__ __forceinline__ unsigned order_key(float v)
{
    const unsigned b = __float_as_uint(v + 0.0f);
    return b & 0x80000000u ? ~b : b | 0x80000000u;
}
__device__ __forceinline__ float key_value(unsigned key)
{
    return __uint_as_float(key & 0x80000000u ? key & 0x7fffffffu : ~key);
}

constexpr int kStages = 4;                 // staged form: pieces of 256 columns in the ring
__device__ __forceinline__ void copy16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}

// TT tokens x EE experts per warp, CH pieces of 256 columns loaded ahead of their arithmetic; CH = 0: the block's rows of
// both operands go through a ring in shared memory.
template <int TT, int EE, int CH>
__global__ void __launch_bounds__(512)
router_topk_kernel(const uint16_t *__restrict__ x, const uint16_t *__restrict__ w_r,
                   const float *__restrict__ bias, const int32_t *__restrict__ token_seq,
                   int T, int d, int E, int k, int n_eg, int tokens_per_block, int32_t *__restrict__ idx,
                   float *__restrict__ gate, float *__restrict__ logits_out, int32_t *__restrict__ block_counts)
{
    extern __shared__ __align__(16) float s_logit[];        // [tokens_per_block][kMaxExperts]
    __shared__ int32_t s_count[kMaxExperts];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, n_warps = blockDim.x >> 5;
    const int b0 = blockIdx.x * tokens_per_block;            // the block's first token
    const int n_tok = min(tokens_per_block, T - b0);
    const int e0 = warp % n_eg * EE, tl = warp / n_eg * TT;  // this warp's first expert, first token within the block
    for (int i = threadIdx.x; i < kMaxExperts; i += blockDim.x)
        s_count[i] = 0;

    const int n_chunks = d >> 8;
    const uint4 *xrow[TT], *wrow[EE];
#pragma unroll
    for (int t = 0; t < TT; ++t)
        xrow[t] = reinterpret_cast<const uint4 *>(x + (size_t)min(b0 + tl + t, T - 1) * d) + lane;
#pragma unroll
    for (int e = 0; e < EE; ++e)
        wrow[e] = reinterpret_cast<const uint4 *>(w_r + (size_t)min(e0 + e, E - 1) * d) + lane;
    uint64_t acc[TT][EE / 2];
#pragma unroll
    for (int t = 0; t < TT; ++t)
#pragma unroll
        for (int e = 0; e < EE / 2; ++e)
            acc[t][e] = 0ull;
    // staged form: this warp's rows of a piece, those of the router matrix or those of the tokens
    const int w_rows = n_eg * EE, stage_bytes = (w_rows + tokens_per_block) * 512;
    const uint32_t ring = (uint32_t)__cvta_generic_to_shared(s_logit + tokens_per_block * kMaxExperts);
    auto fetch = [&](int c, bool tokens) {
        const uint32_t dst = ring + (c % kStages) * stage_bytes + lane * 16;
        const int at = c * 256 + lane * 8;
        if (tokens)
            for (int r = warp; r < tokens_per_block; r += n_warps)
                copy16(dst + (w_rows + r) * 512, x + (size_t)min(b0 + r, T - 1) * d + at);
        else
            for (int r = warp; r < w_rows; r += n_warps)
                copy16(dst + r * 512, w_r + (min(r, E - 1) * d + at));
    };
    // (all operands, the router matrix too, may be the work of the kernel ahead)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (CH == 0)
        for (int c = 0; c < kStages - 1; ++c) {
            if (c < n_chunks) {
                fetch(c, false);
                fetch(c, true);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
    // top-k below: warp w serves token w of the block first; its bias is on the way meanwhile
    float bias0 = 0.0f, bias1 = 0.0f;
    auto load_bias = [&](int t) {
        const int q = token_seq ? token_seq[b0 + t] : 0;
        bias0 = lane < E ? bias[(size_t)q * E + lane] : 0.0f;
        bias1 = lane + 32 < E ? bias[(size_t)q * E + lane + 32] : 0.0f;
    };
    if (bias && warp < n_tok)
        load_bias(warp);

    auto multiply = [&](const uint4(&xv)[TT], const uint4(&wv)[EE]) {
#pragma unroll
        for (int r = 0; r < 4; ++r) {
            auto word = [r](const uint4 &v) { return r == 0 ? v.x : r == 1 ? v.y : r == 2 ? v.z : v.w; };
            uint64_t wl[EE / 2], wh[EE / 2];
#pragma unroll
            for (int e = 0; e < EE / 2; ++e) {
                const uint32_t a = word(wv[2 * e]), b = word(wv[2 * e + 1]);
                wl[e] = pack2(bf16lo(a), bf16lo(b));
                wh[e] = pack2(bf16hi(a), bf16hi(b));
            }
#pragma unroll
            for (int t = 0; t < TT; ++t) {
                const uint32_t v = word(xv[t]);
                const uint64_t xl = pack2(bf16lo(v), bf16lo(v)), xh = pack2(bf16hi(v), bf16hi(v));
#pragma unroll
                for (int e = 0; e < EE / 2; ++e)
                    fma2(acc[t][e], xl, wl[e]);
#pragma unroll
                for (int e = 0; e < EE / 2; ++e)
                    fma2(acc[t][e], xh, wh[e]);
            }
        }
    };
    if (CH == 0) {
#pragma unroll 1
        for (int c = 0; c < n_chunks; ++c) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
            __syncthreads();
            // (every warp has read the stage that is filled now)
            if (c + kStages - 1 < n_chunks) {
                fetch(c + kStages - 1, false);
                fetch(c + kStages - 1, true);
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
            const uint32_t src = ring + (c % kStages) * stage_bytes + lane * 16;
            uint4 xv[TT], wv[EE];
#pragma unroll
            for (int t = 0; t < TT; ++t)
                xv[t] = lds128(src + (w_rows + tl + t) * 512);
#pragma unroll
            for (int e = 0; e < EE; ++e)
                wv[e] = lds128(src + (e0 + e) * 512);
            multiply(xv, wv);
        }
    }
    if (tl < n_tok) {
        constexpr int kAhead = CH ? CH : 1;
#pragma unroll 1
        for (int c0 = 0; CH != 0 && c0 < n_chunks; c0 += kAhead) {
            uint4 xv[kAhead][TT], wv[kAhead][EE];
#pragma unroll
            for (int c = 0; c < kAhead; ++c)
                if (c0 + c < n_chunks) {
#pragma unroll
                    for (int t = 0; t < TT; ++t)
                        xv[c][t] = __ldca(xrow[t] + (c0 + c) * 32);
#pragma unroll
                    for (int e = 0; e < EE; ++e)
                        wv[c][e] = __ldg(wrow[e] + (c0 + c) * 32);
                }
#pragma unroll
            for (int c = 0; c < kAhead; ++c)
                if (c0 + c < n_chunks)
                    multiply(xv[c], wv[c]);
        }
        // the butterfly over the lanes: while more than one value is left, the lower lanes of a stride take the first half
        // of them and the upper lanes the second
        constexpr int N = TT * EE;
        float v[N];
#pragma unroll
        for (int t = 0; t < TT; ++t)
#pragma unroll
            for (int e = 0; e < EE / 2; ++e)
                asm("mov.b64 {%0, %1}, %2;" : "=f"(v[t * EE + 2 * e]), "=f"(v[t * EE + 2 * e + 1]) : "l"(acc[t][e]));
        int left = N;
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1) {
            if (left > 1) {
                left >>= 1;
                const bool up = (lane & m) != 0;
#pragma unroll
                for (int i = 0; i < N / 2; ++i)
                    if (i < left) {
                        const float o = __shfl_xor_sync(0xffffffffu, up ? v[i] : v[i + left], m);
                        v[i] = __fadd_rn(up ? v[i + left] : v[i], o);
                    }
            } else {
                v[0] = __fadd_rn(v[0], __shfl_xor_sync(0xffffffffu, v[0], m));
            }
        }
        constexpr int kLanesPer = 32 / N;
        const int i = lane / kLanesPer, e = e0 + i % EE;
        if (lane % kLanesPer == 0 && e < E)
            s_logit[(tl + i / EE) * kMaxExperts + e] = v[0];
    }
    __syncthreads();

    // top-k: a warp per token.  Lane l holds experts l and l + 32.
    for (int t = warp; t < n_tok; t += n_warps) {
        const float *row = s_logit + t * kMaxExperts;
        if (bias && t != warp)
            load_bias(t);
        float v0 = 0.0f, v1 = 0.0f;
        if (lane < E)
            v0 = bias ? __fadd_rn(row[lane], bias0) : row[lane];
        if (lane + 32 < E)
            v1 = bias ? __fadd_rn(row[lane + 32], bias1) : row[lane + 32];
        if (lane < E)
            logits_out[(size_t)(b0 + t) * E + lane] = v0;
        if (lane + 32 < E)
            logits_out[(size_t)(b0 + t) * E + lane + 32] = v1;
        // k times the greatest of what is left, the lowest index among equals.  (Counting for every element those that
        // beat it took 770 instructions a token whatever k; this takes about 12 per selected expert.)
        unsigned key0 = lane < E ? order_key(v0) : 0u, key1 = lane + 32 < E ? order_key(v1) : 0u;
        float my_sel = 0.0f, top = 0.0f;
        int my_idx = 0;
        for (int j = 0; j < k; ++j) {
            const unsigned best = __reduce_max_sync(0xffffffffu, max(key0, key1));
            const unsigned at0 = __ballot_sync(0xffffffffu, key0 == best), at1 = __ballot_sync(0xffffffffu, key1 == best);
            const int e = at0 ? __ffs(at0) - 1 : 31 + __ffs(at1);
            const float value = key_value(best);
            top = j ? top : value;
            my_sel = lane == j ? value : my_sel;
            my_idx = lane == j ? e : my_idx;
            key0 = e == lane ? 0u : key0;
            key1 = e == lane + 32 ? 0u : key1;
        }
        if (lane < k)
            atomicAdd(&s_count[my_idx], 1);
        float ev = lane < k ? expf(my_sel - top) : 0.0f;
        float sum = ev;
#pragma unroll
        for (int m = 16; m >= 1; m >>= 1)
            sum += __shfl_xor_sync(0xffffffffu, sum, m);
        if (lane < k) {
            idx[(size_t)(b0 + t) * k + lane] = my_idx;
            gate[(size_t)(b0 + t) * k + lane] = ev / sum;
        }
    }
    __syncthreads();
    for (int i = threadIdx.x; i < kMaxExperts; i += blockDim.x)
        block_counts[(size_t)blockIdx.x * kMaxExperts + i] = s_count[i];
}

template <int TT, int EE, int CH>
cudaError_t router_launch(cudaStream_t stream, const RouterShape &sh, const uint16_t *x, const uint16_t *w_r, const float *bias,
                          const int32_t *token_seq, int T, int d, int E, int k, int32_t *idx, float *gate, float *logits_out,
                          int32_t *block_counts)
{
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(sh.n_blocks);
    lc.blockDim = dim3(32 * sh.n_eg * (sh.tokens_per_block / TT));
    lc.dynamicSmemBytes = (size_t)sh.tokens_per_block * kMaxExperts * sizeof(float) +
                          (CH == 0 ? (size_t)kStages * (sh.n_eg * EE + sh.tokens_per_block) * 512 : 0);
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = pdl_enabled() ? 1 : 0;
    return cudaLaunchKernelEx(&lc, router_topk_kernel<TT, EE, CH>, x, w_r, bias, token_seq, T, d, E, k, sh.n_eg, sh.tokens_per_block,
                              idx, gate, logits_out, block_counts);
}

}  // namespace

// One token per warp while that gives no more than two blocks per SM, two up to four, else four (the staged form); more
// token groups per block (at most 16 warps) once there are blocks for every SM, and of the staged form, of which an SM
// holds one, so many that the blocks fit in one round.
RouterShape router_shape(int T, int E, int n_sms)
{
    RouterShape s;
    s.tokens_per_warp = T <= 2 * n_sms ? 1 : T <= 4 * n_sms ? 2 : 4;
    const int ee = s.tokens_per_warp == 4 ? 8 : 4;
    s.n_eg = (E + ee - 1) / ee;
    int tg = (T + (s.tokens_per_warp == 4 ? 4 * n_sms - 1 : 0)) / (s.tokens_per_warp * n_sms);
    tg = tg < 1 ? 1 : tg > 16 / s.n_eg ? 16 / s.n_eg : tg;
    s.tokens_per_block = tg * s.tokens_per_warp;
    s.n_blocks = (T + s.tokens_per_block - 1) / s.tokens_per_block;
    return s;
}

// the staged form's ring: at most 8 expert groups of 8 rows beside 2 groups of 4 tokens, or one beside 16
cudaError_t router_configure()
{
    return cudaFuncSetAttribute(router_topk_kernel<4, 8, 0>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                64 * kMaxExperts * (int)sizeof(float) + kStages * 72 * 512);
}

cudaError_t launch_router(cudaStream_t stream, const RouterShape &sh, const uint16_t *x, const uint16_t *w_r,
                          const float *bias, const int32_t *token_seq, int T, int d, int E, int k,
                          int32_t *idx, float *gate, float *logits_out, int32_t *block_counts)
{
    cudaError_t e;
    if (sh.tokens_per_warp == 1)
        e = router_launch<1, 4, 4>(stream, sh, x, w_r, bias, token_seq, T, d, E, k, idx, gate, logits_out, block_counts);
    else if (sh.tokens_per_warp == 2)
        e = router_launch<2, 4, 2>(stream, sh, x, w_r, bias, token_seq, T, d, E, k, idx, gate, logits_out, block_counts);
    else
        e = router_launch<4, 8, 0>(stream, sh, x, w_r, bias, token_seq, T, d, E, k, idx, gate, logits_out, block_counts);
    count_launch();
    return e;
}

}  // namespace melinoe
