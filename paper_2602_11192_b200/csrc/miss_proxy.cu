// Forward-only evaluation of the paper's cache-miss proxies over a recorded routing trace
// (Section 3.1: the soft cache state of the cache simulation loss L_cs; Definition C.1: the hard
// gamma-discounted Top-C cache, whose misses are the transfers of Appendix C.1).  fp64 throughout;
// the hard misses (an integer result) are exact, the soft proxy differs from a straightforward
// evaluation by fp64 rounding only.
//
//   soft:  c starts at 0 and follows c <- gamma c + r while its L1 norm stays below C; the first
//          update that reaches C is rescaled to norm C and starts the normaliser Z = 1; from then
//          on c <- (gamma Z c + r) / Z', Z' = gamma Z + K / C.  proxy_t = sum_i r_i (1 - c_i).
//   hard:  count starts at 0, count <- gamma count + r; the cache holds the up to C experts of
//          largest non-zero count (lower index first among equals); miss_t = requested experts
//          outside it.
//
// One block per configuration (layer, cache size, gamma).  What bounds it is the walk along the trace,
// a chain of dependent fp64 operations per token, so the chain is kept as short as the definitions
// allow and everything else is moved off it:
//   - the requests of a token are one bit mask, made once per block by all threads and transposed, so that
//     a lane has 32 tokens' requests of its expert in one word;
//   - soft (two warps): u = Z c follows u <- gamma u + r with no division and no normaliser in it, and
//     c = u / Z.  Z does not depend on the requests: lane i holds gamma^i and 1 + gamma + .. + gamma^(i-1),
//     so 32 tokens' normalisers are one multiply-add and one division per lane.  Every lane sums its own
//     expert's u / Z; the lanes meet once, at the end.
//   - hard (one warp, or two): the counts do not depend on C.  The configurations of one layer and gamma
//     therefore share the ranking: each block ranks a part of the tokens (the counts up to there are
//     replayed, two operations per token), keeps a histogram of the requested experts' ranks, and adds to
//     each of those configurations the requests whose rank is C or more.  Only requested experts are
//     ranked, one per lane.
// 912 configurations (57 sizes of 16 layers) over 512 tokens of 8 requests: 1128 us when every
// configuration ranked all 64 experts of every token and met in a warp-wide sum per token, 43 us like this (46.2 with every block
// ranking a part and the totals cleared by a memset ahead; a single layer's 57 configurations 18.8, 20.4 with the memset, of which the
// chain is about 8).  One walk for four configurations, linear in N, and the rest a token per thread, took 34 us but 29 instead of
// 23 for four layers.
#include "kernels.cuh"

namespace melinoe {

namespace {

constexpr int kProxyThreads = 128;
constexpr int kProxyChunk = 512;       // tokens whose masks are held at a time (7 blocks of an SM fit its shared memory)
constexpr int kProxyGroup = 4;         // tokens a warp ranks at a time
constexpr int kProxyWindow = 1024;     // configurations among which equal (layer, gamma) pairs share their ranking

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1)
        v += __shfl_xor_sync(0xffffffffu, v, m);
    return v;
}

// 32 x 32 bits across the warp: bit j of lane l becomes bit l of lane j.
__device__ __forceinline__ unsigned transpose32(unsigned x, int lane)
{
    const unsigned keep[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
        const int o = 16 >> i;
        const unsigned m = keep[i], y = __shfl_xor_sync(0xffffffffu, x, o);
        x = lane & o ? ((y >> o) & m) | (x & ~m) : (x & m) | ((y & m) << o);
    }
    return x;
}

__device__ __forceinline__ bool proxy_config_valid(const melinoe_proxy_config &c, int n_layers, int E)
{
    return c.layer >= 0 && c.layer < n_layers && c.cache_slots >= 1 && c.cache_slots <= E && c.gamma >= 0.0 && c.gamma <= 1.0;
}

// The totals that the blocks of the kernel behind this one add to.
__global__ void clear_totals_kernel(unsigned long long *total, int n)
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
        total[i] = 0ull;
}

__global__ void __launch_bounds__(kProxyThreads, 7) miss_proxy_kernel(const int32_t *__restrict__ idx, int n_layers, int T, int K, int E,
                                                                      const melinoe_proxy_config *__restrict__ cfgs, int n_cfg, int n_sms, int share,
                                                                      double *__restrict__ soft_mean, unsigned long long *hard_total)
{
    __shared__ unsigned s_mask[2][kProxyChunk];      // requests of a token: experts 0..31, 32..63
    __shared__ double s_iz[2][32];
    __shared__ double s_part[2][32][33];             // fill phase: the lanes' states after each of 32 tokens
    __shared__ double s_snap[2][kProxyGroup][kMaxExperts + 1];   // ranking: the counts before each of some tokens
    __shared__ int s_group[4][2];                    // per warp: configurations with this layer and gamma, before this one and in all
    __shared__ unsigned long long s_asked[4];
    __shared__ double s_hit[2];
    __shared__ unsigned s_hist[kMaxExperts + 1];     // requests by rank; the last entry: experts with a zero count
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int ci = blockIdx.x;
    // Warps 0 and 1 of the roles walk the soft state, 2 and 3 rank.  A block's warp w sits on scheduler w of its SM, so
    // the roles rotate from one block of an SM to the next.
    const int role = (warp + ci / n_sms) & 3;
    const melinoe_proxy_config cfg = cfgs[ci];
    if (!proxy_config_valid(cfg, n_layers, E)) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        if (tid == 0) {       // a configuration that names nothing: marked, not evaluated
            soft_mean[ci] = __longlong_as_double(0x7ff8000000000000ll);
            hard_total[ci] = ~0ull;
        }
        return;
    }
    const int C = cfg.cache_slots;
    const double gamma = cfg.gamma;
    for (int i = tid; i <= kMaxExperts; i += kProxyThreads)
        s_hist[i] = 0u;
    const int w0 = ci / kProxyWindow * kProxyWindow, w1 = min(w0 + kProxyWindow, n_cfg);
    auto same = [&](int j) {
        const melinoe_proxy_config o = cfgs[j];
        return o.layer == cfg.layer && o.gamma == gamma && o.cache_slots >= 1 && o.cache_slots <= E;
    };
    int before = 0, all = 0;
#pragma unroll 8
    for (int j = w0 + tid; j < w1; j += kProxyThreads) {
        const bool s = same(j);
        all += s;
        before += s && j < ci;
    }
    before = __reduce_add_sync(0xffffffffu, before);
    all = __reduce_add_sync(0xffffffffu, all);
    if (lane == 0) {
        s_group[warp][0] = before;
        s_group[warp][1] = all;
    }
    // (the histogram has to be clear before it is read, also where there are no tokens and so none of the barriers below; for
    // every trace this would cost 0.9 us of 45)
    if (T == 0)
        __syncthreads();

    const int32_t *trace = idx + (size_t)cfg.layer * T * K;
    const bool vec = (K & 3) == 0 && (reinterpret_cast<uintptr_t>(trace) & 15u) == 0;
    const int e0 = lane, e1 = lane + 32;
    const unsigned bit = 1u << lane;
    // soft warps: the state of this lane's expert (warp `half` has experts 32 half ..), and what the lane needs to
    // form the normalisers
    const int half = role & 1;
    double u = 0.0, acc = 0.0, Zb = 1.0;
    double gi = 1.0, si = 0.0, g32 = 1.0, s32 = 0.0;
    if (role < 2) {
#pragma unroll 1
        for (int i = 0; i < 32; ++i) {
            if (i == lane) {
                gi = g32;
                si = s32;
            }
            s32 = fma(gamma, s32, 1.0);
            g32 *= gamma;
        }
    }
    const double KC = (double)K / (double)C;
    bool filled = false;
    // ranking warps: the counts of this lane's experts
    const int group_tokens = K <= 32 ? min(32 / K, kProxyGroup) : 1;
    double n0 = 0.0, n1 = 0.0;
    int rank_lo = 0, rank_hi = 0;
    // 1 or 0 as a double without a conversion (the low word is zero)
    auto one_if = [](bool r) { return __hiloint2double(r ? 0x3ff00000 : 0, 0); };
    unsigned long long asked = 0ull;

    for (int t0 = 0; t0 < T; t0 += kProxyChunk) {
        const int nt = min(kProxyChunk, T - t0);
#pragma unroll 2
        for (int t = tid; t < nt; t += kProxyThreads) {
            const int32_t *row = trace + (size_t)(t0 + t) * K;
            unsigned lo = 0u, hi = 0u;
            auto add = [&](int e) {
                const unsigned b = (unsigned)e < (unsigned)E ? 1u << (e & 31) : 0u;
                if (e < 32)
                    lo |= b;
                else
                    hi |= b;
            };
            if (vec) {
#pragma unroll 2
                for (int j = 0; j < K; j += 4) {
                    const int4 v = __ldg(reinterpret_cast<const int4 *>(row + j));
                    add(v.x);
                    add(v.y);
                    add(v.z);
                    add(v.w);
                }
            } else {
#pragma unroll 4
                for (int j = 0; j < K; ++j)
                    add(__ldg(row + j));
            }
            s_mask[0][t] = lo;
            s_mask[1][t] = hi;
            asked += (unsigned)(__popc(lo) + __popc(hi));
        }
        __syncthreads();
        if (t0 == 0) {
            // The tokens this block ranks, and the warps that do it: one where many configurations share the work.  Every n-th
            // block ranks only where that leaves 16 or more of the group (512 tokens, us, every third or fourth block of any group
            // and this: 400 groups of 3 sizes 174 and 154, 160 of 4 105 and 72, 64 of 14 53.3 and 50.4).
            const int G = s_group[0][1] + s_group[1][1] + s_group[2][1] + s_group[3][1];
            const int o = s_group[0][0] + s_group[1][0] + s_group[2][0] + s_group[3][0];
            const int n_rank_warps = G >= 16 ? 1 : 2, every = max(1, min(share, G / 16));
            if (role - 2 < n_rank_warps && o % every == 0) {
                const long long parts = (long long)((G + every - 1) / every) * n_rank_warps, part = (long long)(o / every) * n_rank_warps + (role - 2);
                rank_lo = (int)(part * T / parts);
                rank_hi = (int)((part + 1) * T / parts);
            }
        }
        if (role < 2) {
            // r: the lane's expert is requested
            // (predicated by hand: five instructions)
            auto step = [&](unsigned r, double iz) {
                asm("{\n\t.reg .pred p;\n\t.reg .b32 h, l;\n\t.reg .f64 q;\n\t"
                    "setp.ne.u32 p, %2, 0;\n\t"
                    "@p fma.rn.f64 %0, %1, %3, %0;\n\t"
                    "selp.b32 h, 0x3ff00000, 0, p;\n\t"
                    "mov.b32 l, 0;\n\t"
                    "mov.b64 q, {l, h};\n\t"
                    "fma.rn.f64 %1, %4, %1, q;\n\t}"
                    : "+d"(acc), "+d"(u)
                    : "r"(r), "d"(iz), "d"(gamma));
            };
            int t = 0;
            // fill phase: 32 tokens ahead as if none of them filled the cache, then their norms, one per lane (each the
            // sum over the lanes in a fixed tree order); the first that reaches C, if any, is gone back to
            while (t < nt && !filled) {
                const int cnt = min(32, nt - t);
                // bit j: the lane's expert is requested by token t + j
                const unsigned asks = transpose32(lane < cnt ? s_mask[half][t + lane] : 0u, lane);
                const double b = u, c = acc;
#pragma unroll 4
                for (int j = 0; j < cnt; ++j) {
                    step(asks & (1u << j), 1.0);
                    s_part[half][j][lane] = u;
                }
                asm volatile("bar.sync 1, 64;" ::: "memory");
                double v[16];
#pragma unroll
                for (int i = 0; i < 16; ++i)
                    v[i] = (s_part[0][lane][i] + s_part[1][lane][i]) + (s_part[0][lane][i + 16] + s_part[1][lane][i + 16]);
#pragma unroll
                for (int w = 8; w >= 1; w >>= 1)
#pragma unroll
                    for (int i = 0; i < w; ++i)
                        v[i] += v[i + w];
                const unsigned full = __ballot_sync(0xffffffffu, lane < cnt && v[0] >= (double)C);
                if (full) {
                    const int run = __ffs((int)full);
                    const double norm = __shfl_sync(0xffffffffu, v[0], run - 1);
                    u = b, acc = c;
#pragma unroll 1
                    for (int j = 0; j < run; ++j)
                        step(asks & (1u << j), 1.0);
                    u *= (double)C / norm;
                    filled = true;
                    t += run;
                } else {
                    t += cnt;
                }
                asm volatile("bar.sync 1, 64;" ::: "memory");
            }
            while (t < nt) {
                // Z of the next 32 tokens, one per lane
                const int cnt = min(32, nt - t);
                const unsigned asks = transpose32(lane < cnt ? s_mask[half][t + lane] : 0u, lane);
                const double z = fma(gi, Zb, KC * si);
                s_iz[half][lane] = 1.0 / z;
                __syncwarp();
                if (cnt == 32) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        step(asks & (1u << j), s_iz[half][j]);
                    Zb = fma(g32, Zb, KC * s32);
                } else {
#pragma unroll 1
                    for (int j = 0; j < cnt; ++j)
                        step(asks & (1u << j), s_iz[half][j]);
                    Zb = __shfl_sync(0xffffffffu, z, cnt);
                }
                __syncwarp();
                t += cnt;
            }
        } else if (rank_hi > t0) {
            // product rounded before the sum (no contraction): the hard cache's decisions hang on these bits
            auto advance = [&](bool r0, bool r1) {
                n0 = __dadd_rn(__dmul_rn(gamma, n0), one_if(r0));
                n1 = __dadd_rn(__dmul_rn(gamma, n1), one_if(r1));
            };
            const int lo = min(max(rank_lo - t0, 0), nt), hi = min(max(rank_hi - t0, 0), nt);
            for (int t = 0; t < lo; t += 32) {
                const int cnt = min(32, lo - t);
                const unsigned a0 = transpose32(lane < cnt ? s_mask[0][t + lane] : 0u, lane);
                const unsigned a1 = transpose32(lane < cnt ? s_mask[1][t + lane] : 0u, lane);
                if (cnt == 32) {
#pragma unroll
                    for (int j = 0; j < 32; ++j)
                        advance((a0 >> j) & 1u, (a1 >> j) & 1u);
                } else {
#pragma unroll 1
                    for (int j = 0; j < cnt; ++j)
                        advance((a0 >> j) & 1u, (a1 >> j) & 1u);
                }
            }
            // as many tokens at a time as have their requests in one warp: the counts before each of them, then one
            // request per lane against all of its token's counts
            double(*snap)[kMaxExperts + 1] = s_snap[role - 2];
            for (int t = lo; t < hi; t += group_tokens) {
                const int g = min(group_tokens, hi - t);
                for (int i = 0; i < g; ++i) {
                    snap[i][e0] = n0;
                    snap[i][e1] = n1;
                    advance(s_mask[0][t + i] & bit, s_mask[1][t + i] & bit);
                }
                __syncwarp();
                uint64_t seen = 0;      // more than 32 requests per token: those of the token's earlier passes
                for (int i0 = 0; i0 < g * K; i0 += 32) {
                    const int i = i0 + lane, tok = i / K;
                    int r = i < g * K ? __ldg(trace + (size_t)(t0 + t) * K + i) : -1;
                    if ((unsigned)r >= (unsigned)E || ((seen >> r) & 1ull))
                        r = -1;
                    // an expert that a token names twice is one request
                    const unsigned twins = __match_any_sync(0xffffffffu, r < 0 ? -1 - lane : tok * kMaxExperts + r);
                    if (g * K > 32)
                        seen |= (uint64_t)__reduce_or_sync(0xffffffffu, r >= 0 && r < 32 ? 1u << r : 0u) |
                                (uint64_t)__reduce_or_sync(0xffffffffu, r >= 32 ? 1u << (r - 32) : 0u) << 32;
                    const double *row = snap[r < 0 ? 0 : tok];
                    const double nr = row[max(r, 0)];
                    int k = 0;
                    for (int b = 0; b < E; b += 16)      // (what is not an expert has no count)
#pragma unroll
                        for (int e = b; e < b + 16; ++e) {
                            const double n = row[e];
                            k += n > nr || (n == nr && e < r);
                        }
                    if (r >= 0 && (twins & (bit - 1u)) == 0u)
                        atomicAdd(&s_hist[nr > 0.0 ? k : kMaxExperts], 1u);
                }
                __syncwarp();
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int m = 16; m >= 1; m >>= 1)
        asked += __shfl_xor_sync(0xffffffffu, asked, m);
    if (lane == 0)
        s_asked[warp] = asked;
    if (role < 2) {
        const double hit = warp_sum(acc);
        if (lane == 0)
            s_hit[half] = hit;
    } else if (role == 2) {
        // requests of rank r or more
        unsigned above = s_hist[kMaxExperts];
#pragma unroll
        for (int h = 1; h >= 0; --h) {
            unsigned v = s_hist[32 * h + lane];
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned w = __shfl_down_sync(0xffffffffu, v, o);
                v += lane + o < 32 ? w : 0u;
            }
            v += above;
            s_hist[32 * h + lane] = v;
            above = __shfl_sync(0xffffffffu, v, 0);
        }
    }
    __syncthreads();
    // (programmatic launch: the totals are clear only now; whatever came before the kernel that clears them was complete when it began)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    if (tid == 0) {
        const double n = (double)(s_asked[0] + s_asked[1] + s_asked[2] + s_asked[3]);
        soft_mean[ci] = T > 0 ? (n - (s_hit[0] + s_hit[1])) / (double)T : 0.0;
    }
#pragma unroll 8
    for (int j = w0 + tid; j < w1; j += kProxyThreads)
        if (same(j)) {
            const unsigned n = s_hist[cfgs[j].cache_slots];
            if (n)
                atomicAdd(hard_total + j, (unsigned long long)n);
        }
}

}  // namespace

cudaError_t launch_miss_proxies(cudaStream_t stream, const int32_t *idx, int n_layers, int T, int K, int E,
                                const melinoe_proxy_config *cfgs, int n_cfg, int n_sms, double *soft_mean, long long *hard_total)
{
    // the blocks add their parts up
    const int n_clear = (n_cfg + 255) / 256;
    clear_totals_kernel<<<n_clear < 64 ? n_clear : 64, 256, 0, stream>>>(reinterpret_cast<unsigned long long *>(hard_total), n_cfg);
    count_launch();
    // Every block ranks while the GPU is not full; beyond two blocks per SM the replays that this takes cost more than the ranking
    // of more tokens by fewer blocks (912 configurations in groups of 57: 46.2 us with every block, 43.4 with every third), as long as
    // enough blocks of a group are left to rank (see the kernel).
    const int want = n_cfg / (2 * n_sms), share = want < 1 ? 1 : want < 4 ? want : 4;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(n_cfg);
    lc.blockDim = dim3(kProxyThreads);
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = pdl_enabled() ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&lc, miss_proxy_kernel, idx, n_layers, T, K, E, cfgs, n_cfg, n_sms, share, soft_mean,
                                             reinterpret_cast<unsigned long long *>(hard_total));
    count_launch();
    return e != cudaSuccess ? e : cudaGetLastError();
}

}  // namespace melinoe
