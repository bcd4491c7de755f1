// Expert FFN (Eq. 3) for calls with many tokens per expert (prefill): a grouped GEMM on the
// fifth-generation tensor cores (tcgen05.mma, accumulators in tensor memory, operands staged
// in shared memory by TMA), plus the combine (Eq. 2) behind.
//
//   gather    (plan.cu) Xs[pos] = hidden[token of sorted position pos]: the tokens of one expert become
//             consecutive rows, so an expert's activations are one 2-D box for TMA.  Short calls do without:
//             TMA fetches the rows by index (kIndexedTokens).
//   GEMM 1    per expert: [G ; U] = [W_g ; W_u] * Xs_e^T (K = d); the epilogue forms h = SiLU(g) * u and
//             stores it as bf16.
//   GEMM 2    per expert: Z^T = W_d * H_e^T (K = d_ff), fp32.
//   combine   y_t = sum_j gate[t][j] * Z[pos(t, j)] (+ shared experts), rank order, one rounding.
// With 4-bit slots the gate goes into h before its rounding, as in the decode kernel, and the combine adds the rows up: a token
// gets the same result from a long call as from a short one, but for the order of fp32 sums (3.2e-3 apart otherwise).
//
// The weights are the M side of the tensor-core operation and the tokens its N side.  An expert's weights
// come in whole tiles of 128 rows (64 hidden units of W_g and W_u, or 128 output columns), but its
// tokens do not come in any multiple: N follows them in steps of 16 (32 for a CTA pair), so that no
// arithmetic is spent on rows that do not exist.  (With the tokens on the M side a last tile of 256 rows was
// half empty on average: one fifth of the arithmetic of 4096 tokens over 16 experts.)
//
// The expert blob (see melinoe_moe_pack_expert) holds, per hidden unit f, the rows W_g[f], W_u[f]
// and W_d[:, f], each d elements, with the 16-byte pieces of every 128-byte group stored at
// (piece xor (f mod 8)).  That permutation is exactly what a TMA load with 128-byte swizzle would
// have produced in shared memory from plain rows, as long as a row lands at a shared-memory row equal to f
// modulo 8; so the weight tiles are fetched by TMA WITHOUT swizzle and the MMA descriptors name the
// 128-byte-swizzled layout.
//   GEMM 1    a stage's weight tile is ONE box of a 4-D view (column, f mod 8, W_g | W_u, f / 8): eight rows
//             of W_g, eight of W_u, and so on, K-major.  g and u of a hidden unit are then accumulator
//             rows eight apart, and the epilogue brings them together with one shuffle per two tokens.
//   GEMM 2    rows of W_d^T are "K x M, M contiguous": the operand is M-major, two boxes of 64 columns
//             x 64 rows f per stage, fetched as one box of the view (column, f, column group, slot); f beyond
//             d_ff is out of bounds there and reads as zero, so d_ff may end inside a stage.
// The slots' experts are addressed through one tensor map per view, because the slots are contiguous.
//
// 4-bit slots (template parameter FMT = 1): TMA brings the codes into a ring of its own, and sixteen warps expand
// them into the weight tile of a stage (the arithmetic of the decode kernel: 15 instructions per 8
// weights) in front of the tensor cores, so that HBM carries 4-bit data only and no bf16 copy of an expert
// exists.  In GEMM 1 the expansion leaves elements j and j + 4 of eight side by side; a sum over K does not
// care, so Xs is gathered with the same order.
//
// One persistent CTA per SM, warp-specialised: warp 0 issues TMA loads of weights into a ring of stages, warp 1
// issues the MMAs (one elected thread) and commits them to mbarriers, warps 2..9 drain
// the accumulator (tcgen05.ld, 32 rows per warp) and write the tile, warp 10 loads activations; with 4-bit slots warp 0 loads those,
// warps 10..25 expand and warp 26 fetches codes.  Two accumulators alternate so the epilogue of a tile overlaps the MMAs of the next.
// Work items are (GEMM, request, weight tile, token chunk).  One launch does both GEMMs of a compute group and hands its items out to
// the CTA pairs as they run out of work, or each GEMM has a launch of its own, whose items are dealt out beforehand (GemmWalk,
// ffn_gemm_kernel; which: launch_ffn_gemm).
//
// Ragged N: a chunk's box may run past its expert's last row; those columns are computed on whatever
// the next rows hold (or zeros past the end of the buffer) and never stored.
//
// CTA pairs (template parameter CG = 2; CG = 1 serves short calls of 4-bit slots and stays selectable for bf16 slots): two CTAs of a
// cluster on neighbouring SMs take two adjacent weight tiles of the same expert and chunk and run them
// as ONE tensor-core operation of M = 256 (tcgen05.mma.cta_group::2, issued by the even CTA).  Each
// CTA stages its own 128 weight rows but only HALF of the tokens; the tensor cores of both SMs read both
// halves.  Per CTA and k-block that is 32 KB for a chunk of 256 tokens instead of 48 KB.  Both CTAs' loads
// complete on the even CTA's barrier; its MMA thread frees a stage, and hands over an accumulator, in both
// CTAs at once (commit with cluster multicast); the odd CTA's epilogue warps report to the even CTA's
// barrier.  Each CTA drains its own accumulator rows.
//
// What bounds it: the tensor cores under the power cap from some 250 tokens per expert on (1.1 to 1.4 GHz at 985 W in a steady
// stream), reading the weights below some 150 (6 TB/s), the expansion with 4-bit slots.  A pass of a layer, two launches of the GEMMs ->
// one, with the front end as it is now (us): 16 tokens, d 2048, d_ff 1024, 64 experts, 8 per token 61 -> 55; 128 tokens 72 -> 66;
// 4096 tokens, d 4096, d_ff 6400, 16 experts, 2 per token 1295 -> 1246; 8192 tokens, d 2048, d_ff 1408, 66 experts
// 1225 -> 1227; 4-bit slots of the first shape, 16 tokens 70 -> 52, 512 tokens 128 -> 123.
//
// Every wait is bounded; on a timeout the CTA raises its abort flag, every role leaves its
// loops, tensor memory is freed and the error word tells the host.
#include <cuda.h>

#include "kernels.cuh"

namespace melinoe {

namespace {

constexpr int kBK = 64;                    // K elements per stage (128 bytes)
constexpr int kABytes = 128 * kBK * 2;     // weight tile of a stage: 128 rows
constexpr int kRawBytes = 16384;           // 4-bit slots: codes of one fetch (GEMM 1: 256 columns of 128 rows; GEMM 2: 128 rows f of 256 columns)
constexpr int kRawStages = 3;
constexpr int kEpilogueWarps = 8;          // two per 32 accumulator rows, each with every other 16 tokens
constexpr int kExpandGroups = 4;           // 4-bit slots: groups of four warps that expand k-blocks in turn
constexpr size_t kGemmSmem = 227 * 1024 - 4096;      // dynamic shared memory of a CTA (the static part is below 3 KB)
// threads, tokens of a chunk at most, number of ring stages for CG CTAs per operation and slot format FMT
__host__ __device__ constexpr int gemm_threads(int fmt) { return 32 * (2 + kEpilogueWarps + (fmt ? 4 * kExpandGroups + 1 : 1)); }
__host__ __device__ constexpr int gemm_tokens(int cg) { return cg == 2 ? 256 : 128; }
constexpr int kStageBytes = kABytes + 128 * kBK * 2;      // a CTA stages 128 tokens in both forms
__host__ __device__ constexpr int gemm_stages(int fmt)
{
    return (int)((kGemmSmem - 1024 - (fmt ? kRawStages * kRawBytes : 0)) / kStageBytes);
}
constexpr int kItemRing = 4;               // item numbers on their way to the warps
// k-blocks before the end of an item's loads at which the next item is fetched: late, so that the last ones go to whoever is
// free, but not so late that its first loads wait for the counter (or, with 4-bit slots, the codes, which are fetched further ahead).
constexpr int kAskAhead = 4, kAskAhead4 = 16;
constexpr long long kGemmWaitCycles = 4000000000ll;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

// The same where threads of the other CTA of a pair arrive, too: acquires at the scope of the cluster.
__device__ __forceinline__ bool mbar_try_cluster(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}

template <bool CLUSTER = false>
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag)
{
    auto reached = [&] { return CLUSTER ? mbar_try_cluster(bar, parity) : mbar_try(bar, parity); };
    if (reached())
        return true;
    if (*abort_flag)
        return false;
    const long long t0 = clock64();
    for (;;) {
        for (int i = 0; i < 64; ++i)
            if (reached())
                return true;
        if (*abort_flag)
            return false;
        if (clock64() - t0 > kGemmWaitCycles) {
            *abort_flag = 1;
            return false;
        }
    }
}

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}

// Tiled TMA loads: box at the given coordinates (innermost first) of the tensor map into shared memory.  The forms of a
// CTA pair (CG = 2) may count their completion on the peer CTA's barrier (bar is an address in the
// cluster's shared window).
template <int CG>
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap *map, int x, int y, uint32_t bar)
{
    if (CG == 1)
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
            ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar)
            : "memory");
    else
        asm volatile(
            "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
            ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(bar)
            : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
template <int CG>
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, int w, uint32_t bar)
{
    if (CG == 1)
        asm volatile(
            "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
            ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
            : "memory");
    else
        asm volatile(
            "cp.async.bulk.tensor.4d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];"
            ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(bar)
            : "memory");
}
__device__ __forceinline__ void tma_load_5d(uint32_t dst, const CUtensorMap *map, int x, int y, int z, int w, int v, uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.5d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
        ::"r"(dst), "l"(map), "r"(x), "r"(y), "r"(z), "r"(w), "r"(v), "r"(bar)
        : "memory");
}
// Four rows of a matrix, by index, 64 columns of each: the tensor map's box is one row of 64 columns.
template <int CG>
__device__ __forceinline__ void tma_gather4(uint32_t dst, const CUtensorMap *map, int x, const int (&row)[4], uint32_t bar)
{
    if (CG == 1)
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
            ::"r"(dst), "l"(map), "r"(x), "r"(row[0]), "r"(row[1]), "r"(row[2]), "r"(row[3]), "r"(bar)
            : "memory");
    else
        asm volatile(
            "cp.async.bulk.tensor.2d.shared::cluster.global.tile::gather4.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%2, %3, %4, %5, %6}], [%7];"
            ::"r"(dst), "l"(map), "r"(x), "r"(row[0]), "r"(row[1]), "r"(row[2]), "r"(row[3]), "r"(bar)
            : "memory");
}
// Address of this CTA's shared-memory location `addr` in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t cluster_addr(uint32_t addr, uint32_t rank)
{
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
    return r;
}
// Arrival on the peer CTA's barrier, a release at the scope of the cluster: what it reports (expanded weights in this CTA's
// shared memory, an accumulator that may be overwritten) is used by an operation that a thread of the peer issues.  It
// takes its warp some 1100 cycles.
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar)
{
    asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// A word into the peer's shared memory, whose arrival its barrier counts (as four bytes).  A store and an arrival would need the
// arrival to be a release at the scope of the cluster, which waits for everything that its warp has under way.
__device__ __forceinline__ void st_async(uint32_t cluster_dst, int v, uint32_t cluster_bar)
{
    asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.s32 [%0], %1, [%2];" ::"r"(cluster_dst), "r"(v), "r"(cluster_bar) : "memory");
}
// Arrival where all that was done before it is a read, whose value has been used, of what the peer's thread writes next.
__device__ __forceinline__ void mbar_arrive_cluster_relaxed(uint32_t cluster_bar)
{
    asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap *map)
{
    asm volatile("prefetch.tensormap [%0];" ::"l"(map) : "memory");
}
template <int N>
struct Const {
    static constexpr int value = N;
};
// One lane of a converged warp.
__device__ __forceinline__ bool elect_one()
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "elect.sync _|p, 0xffffffff;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(r));
    return r != 0;
}
__device__ __forceinline__ void cluster_sync_all()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Shared-memory matrix descriptor: K-major operand, 128-byte swizzle, rows of 128 bytes, groups
// of 8 rows 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128(uint32_t addr)
{
    uint64_t d = 0;
    d |= (uint64_t)((addr & 0x3FFFFu) >> 4);          // start address
    d |= (uint64_t)(1024u >> 4) << 32;                // stride between 8-row groups
    d |= (uint64_t)1 << 46;                           // descriptor version of this architecture
    d |= (uint64_t)2 << 61;                           // 128-byte swizzle
    return d;
}

// The same for an M-major A operand made of 64-column boxes (64 K rows of 128 bytes each, 8 KB per
// box): the boxes follow one another along M (leading offset), groups of 8 K rows are 1024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc_sw128_mmajor(uint32_t addr)
{
    uint64_t d = smem_desc_sw128(addr);
    d |= (uint64_t)(8192u >> 4) << 16;                // between 64-column boxes
    return d;
}

// Instruction descriptor: bf16 x bf16 -> fp32, A K-major or M-major, B K-major.
__device__ __forceinline__ uint32_t instr_desc_bf16(int m, int n, bool a_mmajor)
{
    uint32_t d = 0;
    d |= 1u << 4;                    // D format: fp32
    d |= 1u << 7;                    // A format: bf16
    d |= 1u << 10;                   // B format: bf16
    d |= (a_mmajor ? 1u : 0u) << 15; // A major: 0 = K, 1 = M
    d |= (uint32_t)(n >> 3) << 17;
    d |= (uint32_t)(m >> 4) << 24;
    return d;
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void umma_commit(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// The pair forms: one operation over both CTAs' tensor cores; the commit arrives on the barrier at this
// offset in both CTAs of the pair.
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                               uint32_t accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
        ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}
__device__ __forceinline__ void umma_commit_pair(uint32_t bar)
{
    asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
                 ::"r"(bar), "h"((uint16_t)3)
                 : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&r)[16])
{
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=f"(r[0]), "=f"(r[1]), "=f"(r[2]), "=f"(r[3]), "=f"(r[4]), "=f"(r[5]), "=f"(r[6]), "=f"(r[7]),
          "=f"(r[8]), "=f"(r[9]), "=f"(r[10]), "=f"(r[11]), "=f"(r[12]), "=f"(r[13]), "=f"(r[14]), "=f"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// to nearest even, as the low half
__device__ __forceinline__ uint16_t bf16_bits(float v)
{
    uint16_t r;
    asm("cvt.rn.bf16.f32 %0, %1;" : "=h"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ uint32_t bf16_rne(float v)
{
    uint32_t u = __float_as_uint(v);
    u += 0x7fffu + ((u >> 16) & 1u);
    return u >> 16;
}

// Eight 4-bit codes into bf16 weights, as four registers P[j] = (element j, element j + 4); see the decode kernel.
__device__ __forceinline__ void expand8(uint32_t w, uint32_t ss, uint32_t (&P)[4])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t t = ((w >> (4 * j)) & 0x000f000fu) | 0x43004300u;
        asm("sub.rn.bf16x2 %0, %0, %1;" : "+r"(t) : "r"(0x43084308u));
        asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(P[j]) : "r"(t), "r"(ss));
    }
}
// The first two of the four registers: elements (0, 4) and (1, 5) of the word.
__device__ __forceinline__ void expand4(uint32_t w, uint32_t ss, uint32_t (&P)[2])
{
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        uint32_t t = ((w >> (4 * j)) & 0x000f000fu) | 0x43004300u;
        asm("sub.rn.bf16x2 %0, %0, %1;" : "+r"(t) : "r"(0x43084308u));
        asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(P[j]) : "r"(t), "r"(ss));
    }
}
__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ void sts128(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d)
{
    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d) : "memory");
}

struct GemmItem {
    int phase;     // 1 = GEMM 1, 2 = GEMM 2
    int row0;      // first sorted row of the token chunk
    int n;         // tokens of the operation (a multiple of 16 CG)
    int n_live;    // tokens that exist
    int m0;        // first hidden unit (GEMM 1) or output column (GEMM 2) of this CTA's weight tile
    int slot;      // cache slot of the expert, or -1 - index of the shared expert
    int kblocks;   // stages of its reduction
    int q;         // place of its request among the launch's requests
};

// A CTA's share of an item's tokens: so many rows, fetched by index, or the smallest box that holds them, of 32 << cls rows.
struct TokenBox {
    int rows, cls, row;
    __device__ TokenBox(const GemmItem &it, int cg, int rank)
    {
        rows = __shfl_sync(0xffffffffu, it.n, 0) / cg;
        cls = rows <= 32 ? 0 : rows <= 64 ? 1 : 2;
        row = __shfl_sync(0xffffffffu, it.row0, 0) + rank * rows;
    }
    __device__ uint32_t bytes(bool indexed) const { return indexed ? (uint32_t)rows * kBK * 2 : (32u * kBK * 2) << cls; }
};

// The items of both GEMMs in one order: all of GEMM 1, then all of GEMM 2, by request, weight tile, chunk of tokens (the chunks
// of a tile side by side, so that pairs working at the same time share it in L2).  A unit's items come in this order, too, whether a
// CTA pair takes the next one whenever it is about to run out of work (PHASE 0) or has every n-th of one GEMM's.
template <int CG, int PHASE>
struct GemmWalk {
    const int4 *rec;         // first row, tokens, slot (shared expert s: -1 - s), tokens of a chunk
    const int *chunk0;       // chunks of the requests before each
    int m1, m2, k1, k2;      // weight tiles of a request and stages of a reduction in both phases
    int q, phase, rank, total1, total;
    __device__ GemmWalk(const int4 *rec_, const int *chunk0_, int n_reqs, int d, int F, int rank_)
        : rec(rec_), chunk0(chunk0_), m1((F + CG * 64 - 1) / (CG * 64)), m2(d / (CG * 128)), k1(d / kBK), k2((F + kBK - 1) / kBK), q(0),
          phase(1), rank(rank_)
    {
        total1 = chunk0_[n_reqs] * m1;
        total = PHASE == 1 ? total1 : total1 + chunk0_[n_reqs] * m2;
    }
    // PHASE 1, 2: item i of this unit
    __device__ int dealt(uint32_t i) const
    {
        return (PHASE == 2 ? total1 : 0) + (int)blockIdx.x / CG + (int)i * ((int)gridDim.x / CG);
    }
    // item w, which is never before the one asked for last
    __device__ bool at(int w, GemmItem &it)
    {
        if (w >= total)
            return false;
        if (PHASE != 1 && w >= total1) {
            if (phase == 1)
                q = 0;
            phase = 2;
            w -= total1;
        }
        const int ph = PHASE ? PHASE : phase, m = ph == 1 ? m1 : m2;
        while (chunk0[q + 1] * m <= w)
            ++q;
        const int4 r = rec[q];
        const int n = chunk0[q + 1] - chunk0[q], local = w - chunk0[q] * m, tile = local / n, c = local - tile * n;
        it.phase = ph;
        it.m0 = (tile * CG + rank) * (ph == 1 ? 64 : 128);
        it.kblocks = ph == 1 ? k1 : k2;
        it.row0 = r.x + c * r.w;
        it.n_live = min(r.w, r.y - c * r.w);
        it.n = (it.n_live + 16 * CG - 1) / (16 * CG) * (16 * CG);
        it.slot = r.z;
        it.q = q;
        return true;
    }
};

// GEMM 1: h = SiLU(Xs W_g^T) * (Xs W_u^T) -> hs (bf16).  GEMM 2: z = hs W_d^T -> zs (fp32).
//
// PHASE 0: one launch does both.  As two launches, each ended with a round of items that did not fill the GPU (a prompt of 128 tokens
// over some 20 experts has 160 items for 74 pairs in both: 3 rounds for 2.16) and the second began with an empty pipeline; and
// items of unequal sizes were dealt out beforehand.  Now a pair fetches its next item's number from a counter
// in global memory (the loading warp of the even CTA, a few stages before its loads run out; it hands the
// number on to everyone through a ring in shared memory), and GEMM 2 follows GEMM 1 without a break: a request's
// items wait until as many epilogue warps as GEMM 1 has for it have counted themselves out.  That wait ends whatever else is on
// the GPU: GEMM 2's items are handed out after all of GEMM 1's, so what it waits for is in the hands of CTAs
// that are running, and GEMM 1 waits for nobody.
//
// PHASE 1, 2: that GEMM alone, a unit's items known from the start; GEMM 2 loads weights ahead of the end of GEMM 1's grid.  PHASE 0
// has a price: the round trip to the counter and the number's way to the odd CTA before the first load (2 us a launch), and a
// release per item and epilogue warp, which waits for the stores of h, before the next tile is drained.  Reductions of 4 to 12
// k-blocks (d up to 768) do not cover it (4000 tokens, d 512, d_ff 8192, 8 experts, 2 per token, 4-bit slots: 297 us a pass, 262 in two
// launches; of the difference 16 us are the releases, 7 the numbers, the rest loops over a phase that the compiler knows).
template <int CG, int FMT, int PHASE>
__global__ void __launch_bounds__(gemm_threads(FMT), 1) ffn_gemm_kernel(const __grid_constant__ GemmParams p)
{
    constexpr int kStages = gemm_stages(FMT), NT = gemm_tokens(CG);
    static_assert(FMT == 0 || kExpandGroups <= kStages, "a group's wait for its stage has to be for the last use of it");
    // warps that read an item's number: epilogue, activations or expansion and codes, the even CTA's MMA warp, the odd one's warp 0
    constexpr int kReaders = CG * (kEpilogueWarps + (FMT ? 4 * kExpandGroups + 1 : 1)) + CG;
    extern __shared__ __align__(1024) unsigned char smem_raw[];
    __shared__ uint64_t s_bars[2 * kStages + 4 + 2 * kRawStages + 2 * kItemRing];
    __shared__ uint32_t s_tmem_base;
    __shared__ int s_abort;
    __shared__ int s_item[kItemRing];
    __shared__ int s_chunk0[kMaxReq + 1], s_nreq;
    __shared__ int4 s_rec[kMaxReq];                          // see GemmWalk
    __shared__ int s_req[kMaxReq];                           // its place in the plan

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const DevPlan *plan = p.plan;
    // 1024-byte aligned ring (the swizzle pattern repeats every 1024 bytes)
    unsigned char *ring = reinterpret_cast<unsigned char *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    const uint32_t ring_s = smem_u32(ring), raw_s = ring_s + kStages * kStageBytes;
    const uint32_t full0 = smem_u32(s_bars), empty0 = full0 + 8 * kStages;
    const uint32_t tfull0 = empty0 + 8 * kStages, tempty0 = tfull0 + 16, rfull0 = tempty0 + 16, rempty0 = rfull0 + 8 * kRawStages;
    const uint32_t ifull0 = rempty0 + 8 * kRawStages, iempty0 = ifull0 + 8 * kItemRing;
    volatile int *abort_flag = &s_abort;
    // rank within the CTA pair; the even CTA fetches the items, issues the MMAs, owns the "stage full" barriers and counts
    // the drained accumulators of both
    uint32_t rank = 0;
    if (CG == 2)
        asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));

    if (tid == 32) {
        s_abort = 0;
        for (int i = 0; i < kStages; ++i) {
            mbar_init(full0 + 8 * i, FMT ? 1 + 4 * CG : 1);
            mbar_init(empty0 + 8 * i, 1);
        }
        for (int i = 0; i < 2; ++i) {
            mbar_init(tfull0 + 8 * i, 1);
            mbar_init(tempty0 + 8 * i, kEpilogueWarps * CG);
        }
        if (FMT)
            for (int i = 0; i < kRawStages; ++i) {
                mbar_init(rfull0 + 8 * i, 1);
                mbar_init(rempty0 + 8 * i, 4 * kExpandGroups);
            }
        for (int i = 0; i < kItemRing; ++i) {
            mbar_init(ifull0 + 8 * i, 1);
            mbar_init(iempty0 + 8 * i, kReaders);
        }
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 2) {
        // (a pair: the same warp of both CTAs, the same destination, one allocation over the pair)
        if (CG == 1) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)),
                         "r"(2 * NT));
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        } else {
            asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem_base)),
                         "r"(2 * NT));
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;");
        }
    }
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    if (warp == 1 && lane < kMapSlots0 + 2)
        prefetch_map(p.maps + lane);
    if (warp == 1 && lane == 31 && p.by_index)
        prefetch_map(&p.x_map);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    // (a pair: the barriers of both CTAs exist before either signals the other's)
    if (CG == 2)
        cluster_sync_all();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_base = s_tmem_base;
    // All of this runs while the kernels ahead do.  The plan is read once its word announces it: with it the weights of
    // the group are in their slots, and all of the call before it, and so everything ahead of the router, is complete.  Of what is
    // read here, that leaves what the gather kernel makes, where there is one.
    auto claim = [&]() -> int { return lane == 0 ? atomicAdd(&p.counters->next[p.group], 1) : 0; };
    // ---- the launch's requests and their items, by warp 0, a lane per request
    int ahead = 0;                                           // loading warp: the next item's number (lane 0)
    if (warp == 0) {
        uint32_t hdr = 0;
        bool ok = true;
        if (lane == 0) {
            ok = wait_for_ready(plan, p.call_seq, &hdr);
            if (!ok)
                s_abort = 1;
        }
        __syncwarp();
        hdr = __shfl_sync(0xffffffffu, hdr, 0);
        ok = __shfl_sync(0xffffffffu, (int)ok, 0) != 0;
        const int n_req_total = ok && plan_accepted(hdr) ? (int)(hdr & 0xffu) : 0;
        if (PHASE == 0 && rank == 0 && n_req_total > 0)
            ahead = claim();
        int n = 0, sum = 0;
        constexpr int kRounds = (kMaxReq + 31) / 32;
        int4 a[kRounds], b[kRounds];
#pragma unroll
        for (int i = 0; i < kRounds; ++i) {
            const int r = 32 * i + lane;
            a[i] = b[i] = make_int4(0, 0, 0, 0);
            if (r < n_req_total) {
                a[i] = __ldcg(reinterpret_cast<const int4 *>(&plan->req[r].expert));       // expert, slot, hit, evicted
                b[i] = __ldcg(reinterpret_cast<const int4 *>(&plan->req[r].vr_start));     // vr_start, group, tok_off, n_tok
            }
        }
#pragma unroll
        for (int i = 0; i < kRounds; ++i) {
            const int r = 32 * i + lane, n_tok = b[i].w;
            const bool on = r < n_req_total && b[i].y == p.group && n_tok > 0;
            // chunks of equal size, in steps of the operation's N
            int chunks = on ? (n_tok + NT - 1) / NT : 0;
            const int size = on ? ((n_tok + chunks - 1) / chunks + 16 * CG - 1) / (16 * CG) * (16 * CG) : 0;
            chunks = on ? (n_tok + size - 1) / size : 0;
            const unsigned m = __ballot_sync(0xffffffffu, on);
            int inc = chunks;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(0xffffffffu, inc, o);
                inc += lane >= o ? v : 0;
            }
            if (on) {
                const int at = n + __popc(m & ((1u << lane) - 1u));
                s_rec[at] = make_int4(b[i].z, n_tok, a[i].y >= 0 ? a[i].y : -1 - (a[i].x - p.E), size);
                s_req[at] = r;
                s_chunk0[at] = sum + inc - chunks;
            }
            n += __popc(m);
            sum += __shfl_sync(0xffffffffu, inc, 31);
        }
        if (lane == 0) {
            s_chunk0[n] = sum;
            s_nreq = n;
        }
    }
    __syncthreads();
    const int n_reqs = s_nreq;

    GemmWalk<CG, PHASE> walk(s_rec, s_chunk0, n_reqs, p.d, p.F, (int)rank);
    GemmItem it;
    // of a pair, the bytes of both CTAs are expected and counted on the even CTA's barriers
    const uint32_t full_b = CG == 1 ? full0 : cluster_addr(full0, 0);
    // Item i of this unit, for the whole warp; false behind the last one.
    auto next = [&](uint32_t i) -> bool {
        if (PHASE)
            return __all_sync(0xffffffffu, !*abort_flag) && walk.at(walk.dealt(i), it);
        const uint32_t slot = i % kItemRing;
        const bool ok = !*abort_flag && mbar_wait<CG == 2>(ifull0 + 8 * slot, (i / kItemRing) & 1u, abort_flag);
        if (!__all_sync(0xffffffffu, ok))
            return false;
        const int w = *(volatile int *)&s_item[slot];
        const bool more = walk.at(w, it);
        __syncwarp();
        if (lane == 0) {
            if (CG == 1 || rank == 0)
                mbar_arrive(iempty0 + 8 * slot);
            else
                mbar_arrive_cluster_relaxed(cluster_addr(iempty0 + 8 * slot, 0));
        }
        return more;
    };

    // The warps that load activations: those of GEMM 2 are complete once GEMM 1's epilogue warps of the request have counted themselves
    // out, or, if it had a launch of its own, once that has ended.
    int h_of = -1;                                           // the request that was waited for last
    auto wait_for_h = [&]() -> bool {
        if (PHASE || it.phase == 1 || it.q == h_of)
            return true;
        h_of = it.q;
        const int *done = &p.counters->done[s_req[it.q]];
        const int want = (s_chunk0[it.q + 1] - s_chunk0[it.q]) * walk.m1 * CG * kEpilogueWarps;
        const long long t0 = clock64();
        bool ok = true;
        for (;;) {
            int v;
            asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(done) : "memory");
            if (v >= want)
                break;
            if (*abort_flag || clock64() - t0 > kGemmWaitCycles) {
                *abort_flag = 1;
                ok = false;
                break;
            }
        }
        asm volatile("fence.proxy.async.global;" ::: "memory");      // other CTAs' threads stored it, TMA reads it
        return __all_sync(0xffffffffu, ok) != 0;
    };

    // Loads of a k-block of activations: rows of the hidden states by index, four per lane, or a box of Xs or h.
    int tok[4] = {0, 0, 0, 0};
    auto find_tokens = [&](const TokenBox &box) {
        const int last = __shfl_sync(0xffffffffu, it.row0 + it.n_live, 0) - 1;
#pragma unroll
        for (int j = 0; j < 4; ++j)                          // (rows that do not exist: the last one again)
            tok[j] = 4 * lane < box.rows ? __ldcg(p.tok_of_sorted + min(box.row + 4 * lane + j, last)) : 0;
    };
    auto load_tokens = [&](bool indexed, const CUtensorMap *map, const TokenBox &box, int kb, uint32_t dst, uint32_t bar) {
        if (indexed) {
            if (4 * lane < box.rows)
                tma_gather4<CG>(dst + lane * 512, &p.x_map, kb * kBK, tok, bar);
        } else if (elect_one()) {
            tma_load_2d<CG>(dst, map, kb * kBK, box.row, bar);
        }
    };
    if (n_reqs == 0) {
        // nothing to do
    } else if (warp == 0) {
        // ============================================================ loads of the weights (the whole warp, one lane issues)
        // A warp for each operand, and nothing in their loops but the wait, the load and what counts it: one warp loading both, with the
        // item's bookkeeping in its loop, was the limit of the whole kernel (8192 tokens, d 2048, d_ff 1408: 1355 us a pass, 1258 like
        // this).  This one counts the bytes of both operands and, in the even CTA, fetches the items; the weights go ahead of activations
        // that are still being waited for.  With 4-bit slots it loads the activations.
        auto publish = [&](uint32_t i, int w) {              // the even CTA's: item number i of the unit is w
            const uint32_t slot = i % kItemRing;
            bool ok = true;
            if (i >= (uint32_t)kItemRing)
                ok = mbar_wait<CG == 2>(iempty0 + 8 * slot, (i / kItemRing - 1u) & 1u, abort_flag);
            if (__all_sync(0xffffffffu, ok) && lane == 0) {
                *(volatile int *)&s_item[slot] = w;
                mbar_arrive(ifull0 + 8 * slot);
                if (CG == 2)
                    st_async(cluster_addr(smem_u32(&s_item[slot]), 1), w, cluster_addr(ifull0 + 8 * slot, 1));
            }
            __syncwarp();
        };
        if (PHASE == 0 && rank == 0)
            publish(0, ahead);
        // (the odd CTA: the number of an item, which arrives by st.async, is expected two items ahead)
        auto expect_number = [&](uint32_t i) {
            if (PHASE == 0 && CG == 2 && rank == 1 && lane == 0)
                mbar_expect(ifull0 + 8 * (i % kItemRing), 4);
        };
        expect_number(0);
        expect_number(1);
        if (FMT == 1)
            asm volatile("griddepcontrol.wait;" ::: "memory");
        uint32_t s = 0, parity = 1, n = 0;                   // stage of the next k-block, parity of its being free; k-blocks so far
        for (uint32_t i = 0;; ++i) {
            const bool more = PHASE == 0 && rank == 0 ? !*abort_flag && walk.at(__shfl_sync(0xffffffffu, ahead, 0), it) : next(i);
            if (!__all_sync(0xffffffffu, more))
                break;
            expect_number(i + 2);
            const int kblocks = __shfl_sync(0xffffffffu, it.kblocks, 0), m0 = __shfl_sync(0xffffffffu, it.m0, 0);
            const int slot_ = __shfl_sync(0xffffffffu, it.slot, 0), slot = slot_ >= 0 ? slot_ : 0;
            const int phase = PHASE ? PHASE : __shfl_sync(0xffffffffu, it.phase, 0);
            // the weights of the slots, or of the shared expert
            const CUtensorMap *map_w = p.maps + (slot_ >= 0 ? kMapSlots0 : kMapShared0 + 2 * (-1 - slot_)) + (phase - 1);
            const TokenBox box(it, CG, (int)rank);
            // (a pair: the bytes of both CTAs)
            const uint32_t bytes = CG * ((FMT ? 0u : (uint32_t)kABytes) + box.bytes(FMT == 0 && p.by_index && phase == 1));
            const CUtensorMap *map_b = p.maps + (phase == 1 ? kMapXs0 : kMapHs0) + box.cls;
            if (FMT == 1 && !wait_for_h())
                break;
            auto run = [&](auto phase_, int kb, int kb_end) -> bool {
                constexpr int kPhase = decltype(phase_)::value;
                const int row = (slot * p.F + m0) / 8, col = m0 / 64;
                n += (uint32_t)(kb_end - kb);
                for (; kb < kb_end; ++kb) {
                    // (a fresh barrier counts as being past its odd phase)
                    if (!__all_sync(0xffffffffu, mbar_wait(empty0 + 8 * s, parity, abort_flag)))
                        return false;
                    if (elect_one()) {
                        if (CG == 1 || rank == 0)
                            mbar_expect(full0 + 8 * s, bytes);
                        const uint32_t dst = ring_s + s * kStageBytes;
                        if (FMT == 1)
                            tma_load_2d<CG>(dst + kABytes, map_b, kb * kBK, box.row, full_b + 8 * s);
                        else if (kPhase == 1)
                            tma_load_4d<CG>(dst, map_w, kb * kBK, 0, 0, row, full_b + 8 * s);
                        else
                            tma_load_4d<CG>(dst, map_w, 0, kb * kBK, col, slot, full_b + 8 * s);
                    }
                    __syncwarp();
                    if (++s == (uint32_t)kStages) {
                        s = 0;
                        parity ^= 1u;
                    }
                }
                return true;
            };
            auto part = [&](int kb, int kb_end) { return phase == 1 ? run(Const<1>(), kb, kb_end) : run(Const<2>(), kb, kb_end); };
            const int ask = max(kblocks - (FMT ? kAskAhead4 : kAskAhead), 0), tell = min(ask + 2, kblocks);
            if (PHASE == 0 && rank == 0) {
                if (!part(0, ask))
                    break;
                ahead = claim();
                if (!part(ask, tell))
                    break;
                publish(i + 1, ahead);
                if (!part(tell, kblocks))
                    break;
            } else if (!part(0, kblocks)) {
                break;
            }
        }
        if (CG == 2) {
            // The MMA thread's commits arrive on this CTA's barriers from outside: wait for the last
            // ones so that none is still under way when the CTA ends.
            for (uint32_t j = n > (uint32_t)kStages ? n - kStages : 0; j < n && !*abort_flag; ++j)
                mbar_wait(empty0 + 8 * (j % kStages), (j / kStages) & 1u, abort_flag);
        }
    } else if (FMT == 0 && warp == 2 + kEpilogueWarps) {
        // ============================================================ loads of the activations
        if (PHASE == 2 || !p.by_index)
            asm volatile("griddepcontrol.wait;" ::: "memory");
        uint32_t s = 0, parity = 1;
        for (uint32_t i = 0; next(i); ++i) {
            if (!wait_for_h())
                break;
            const int kblocks = __shfl_sync(0xffffffffu, it.kblocks, 0);
            const TokenBox box(it, CG, (int)rank);
            const bool first = PHASE ? PHASE == 1 : __shfl_sync(0xffffffffu, it.phase, 0) == 1;
            const CUtensorMap *map_b = p.maps + (first ? kMapXs0 : kMapHs0) + box.cls;
            auto run = [&](auto indexed) -> bool {
                for (int kb = 0; kb < kblocks; ++kb) {
                    if (!__all_sync(0xffffffffu, mbar_wait(empty0 + 8 * s, parity, abort_flag)))
                        return false;
                    load_tokens(decltype(indexed)::value, map_b, box, kb, ring_s + s * kStageBytes + kABytes, full_b + 8 * s);
                    __syncwarp();
                    if (++s == (uint32_t)kStages) {
                        s = 0;
                        parity ^= 1u;
                    }
                }
                return true;
            };
            bool ok;
            if (p.by_index && first) {
                find_tokens(box);
                ok = run(Const<1>());
            } else {
                ok = run(Const<0>());
            }
            if (!ok)
                break;
        }
    } else if (warp == 1) {
        // ============================================================ MMA issuer (of a pair: the even CTA's)
        // The whole warp goes through the loop and one lane issues: values that are the same in all lanes stay in uniform
        // registers, where the tensor-core instructions want them.
        if (rank == 0) {
            uint32_t s = 0, parity = 0;
            const uint32_t ring_d = (ring_s & 0x3FFFFu) >> 4;
            for (uint32_t item = 0;; ++item) {
                if (!next(item))
                    break;
                const int phase = PHASE ? PHASE : __shfl_sync(0xffffffffu, it.phase, 0), kblocks = __shfl_sync(0xffffffffu, it.kblocks, 0);
                const uint32_t idesc = instr_desc_bf16(CG * 128, __shfl_sync(0xffffffffu, it.n, 0), phase == 2);
                const uint32_t acc = item & 1u;
                bool ok = item < 2 || mbar_wait<CG == 2>(tempty0 + 8 * acc, ((item >> 1) - 1u) & 1u, abort_flag);
                if (!__all_sync(0xffffffffu, ok))
                    break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t d_tmem = tmem_base + acc * NT;
                // 16 K elements: 32 bytes along a K-major row (2 descriptor units), 16 rows of 128 bytes in an M-major box (128)
                auto reduce = [&](auto a_step) {
                    constexpr int kAStep = decltype(a_step)::value;
                    const uint64_t a_hi = kAStep == 2 ? smem_desc_sw128(0) : smem_desc_sw128_mmajor(0), b_hi = smem_desc_sw128(0);
                    uint32_t accumulate = 0;
                    for (int kb = 0; kb < kblocks; ++kb) {
                        ok = mbar_wait<FMT == 1>(full0 + 8 * s, parity, abort_flag);
                        if (!__all_sync(0xffffffffu, ok))
                            break;
                        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                        const uint64_t a_desc = a_hi | (ring_d + s * (kStageBytes >> 4));
                        const uint64_t b_desc = b_hi | (ring_d + s * (kStageBytes >> 4) + (kABytes >> 4));
                        if (elect_one()) {
#pragma unroll
                            for (int ks = 0; ks < kBK / 16; ++ks) {
                                if (CG == 1)
                                    umma_bf16(d_tmem, a_desc + kAStep * ks, b_desc + 2 * ks, idesc, ks ? 1u : accumulate);
                                else
                                    umma_bf16_pair(d_tmem, a_desc + kAStep * ks, b_desc + 2 * ks, idesc, ks ? 1u : accumulate);
                            }
                            // the stage is free once these MMAs have read it
                            if (CG == 1)
                                umma_commit(empty0 + 8 * s);
                            else
                                umma_commit_pair(empty0 + 8 * s);
                            // the accumulator is complete
                            if (kb + 1 == kblocks) {
                                if (CG == 1)
                                    umma_commit(tfull0 + 8 * acc);
                                else
                                    umma_commit_pair(tfull0 + 8 * acc);
                            }
                        }
                        __syncwarp();
                        accumulate = 1u;
                        if (++s == (uint32_t)kStages) {
                            s = 0;
                            parity ^= 1u;
                        }
                    }
                };
                if (phase == 1)
                    reduce(Const<2>());
                else
                    reduce(Const<128>());
            }
        }
    } else if (warp < 2 + kEpilogueWarps) {
        // ============================================================ epilogue (warps 2..9)
        // What bounds it is the instructions of a single warp per scheduler (with four warps, 32 tokens took 1.1 to 2.1 us, and
        // 256 tokens longer than the products of the next tile), hence eight, and no predicates on whole chunks.
        const int quarter = warp & 3;                        // the 32 accumulator rows this warp may read
        const int c_first = (warp - 2) / 4 * 16;             // its chunks of 16 tokens: c_first, c_first + 32, ..
        constexpr bool kGated = FMT == 1;
        if (kGated)          // (the rows' gates are the gather's)
            asm volatile("griddepcontrol.wait;" ::: "memory");
        for (uint32_t item = 0; next(item); ++item) {
            const uint32_t acc = item & 1u;
            const bool first = PHASE ? PHASE == 1 : it.phase == 1;
            // 4-bit slots: lanes l and l + 16 hold the gate of the chunk's token l, the next chunk's is on its way
            auto gate_of = [&](int c) {
                return first && c + (lane & 15) < it.n_live ? __ldcg(p.row_gate + it.row0 + c + (lane & 15)) : 0.0f;
            };
            float next_gate = kGated ? gate_of(c_first) : 0.0f;
            if (!__all_sync(0xffffffffu, mbar_wait(tfull0 + 8 * acc, (item >> 1) & 1u, abort_flag)))
                break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t t_row = tmem_base + ((uint32_t)(quarter * 32) << 16) + acc * NT;
            // the accumulator has been read
            auto drained = [&] {
                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                __syncwarp();
                if (lane == 0) {
                    if (CG == 1 || rank == 0)
                        mbar_arrive(tempty0 + 8 * acc);
                    else
                        mbar_arrive_cluster(cluster_addr(tempty0 + 8 * acc, 0));
                }
            };
            if (first) {
                // lanes 0..7 hold g of eight hidden units, 8..15 u of the same ones, 16..31 those of the next eight.  Of two
                // neighbouring tokens the g lane finishes the first and the u lane the second.
                const int f = it.m0 + quarter * 16 + (lane >> 4) * 8 + (lane & 7);
                const bool is_u = (lane & 8) != 0;
                // this lane stores tokens c + 2 j (+ 1) with c + 2 j below this
                const int left = f < p.F ? it.n_live - (is_u ? 1 : 0) : 0;
                uint16_t *dst = p.hs + (size_t)(it.row0 + c_first + (is_u ? 1 : 0)) * p.F + f;
                const size_t step = (size_t)p.F * 2;
#pragma unroll 1
                for (int c = c_first; c < it.n_live; c += 32, dst += 16 * step) {
                    float v[16];
                    const float gate = next_gate;
                    if (kGated)
                        next_gate = gate_of(c + 32);
                    tmem_ld16(t_row + c, v);
                    uint16_t h[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const float o = __shfl_xor_sync(0xffffffffu, is_u ? v[2 * j] : v[2 * j + 1], 8);
                        const float g = is_u ? o : v[2 * j], u = is_u ? v[2 * j + 1] : o;
                        float hv = __fdividef(g, 1.0f + __expf(-g)) * u;
                        if (kGated)
                            hv *= __shfl_sync(0xffffffffu, gate, 2 * j + (is_u ? 1 : 0));
                        h[j] = bf16_bits(hv);
                    }
                    if (c + 14 < left) {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            dst[j * step] = h[j];
                    } else {
#pragma unroll
                        for (int j = 0; j < 8; ++j)
                            if (c + 2 * j < left)
                                dst[j * step] = h[j];
                    }
                }
                drained();
                // this warp's part of h is written: GEMM 2 of the request, in whichever CTA, counts these
                __syncwarp();
                if (PHASE == 0 && lane == 0)
                    asm volatile("red.release.gpu.global.add.s32 [%0], 1;" ::"l"(&p.counters->done[s_req[it.q]]) : "memory");
            } else {
                float *dst = p.zs + (size_t)(it.row0 + c_first) * p.d + it.m0 + quarter * 32 + lane;
                const size_t step = (size_t)p.d;
#pragma unroll 1
                for (int c = c_first; c < it.n_live; c += 32, dst += 32 * step) {
                    float v[16];
                    tmem_ld16(t_row + c, v);
                    if (c + 16 <= it.n_live) {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            dst[j * step] = v[j];
                    } else {
#pragma unroll
                        for (int j = 0; j < 16; ++j)
                            if (c + j < it.n_live)
                                dst[j * step] = v[j];
                    }
                }
                drained();
            }
        }
    } else if (FMT == 1 && warp < 2 + kEpilogueWarps + 4 * kExpandGroups) {
        // ============================================================ expansion of 4-bit codes (warps 10..25)
        // Groups of four warps take the k-blocks in turn, counted over all items (so that a group is never two uses of
        // a stage ahead, which a barrier's parity could not tell): what a k-block takes is latency, waits, arithmetic and
        // the fence before the tensor cores may read, which the other groups' k-blocks cover.  (512 tokens, us a
        // pass: two groups 140, four 127.)  In the odd CTA the arrival that makes the weights visible to the MMA thread of
        // the even one adds to it (512 tokens 114 -> 137 us, 8192 tokens 1084 -> 1218; a relaying warp, one arrival
        // per k-block by the group's warps in turn, or more stages do not make it less).
        const int row = ((warp - 10) & 3) * 32 + lane, group = (warp - 10) >> 2;     // row of the weight tile, or (column group, f) of GEMM 2's
        const size_t ub = (size_t)p.unit_bytes, scales = 3 * (size_t)(p.d / 2);
        uint32_t n0 = 0, rn = 0;
        for (uint32_t item = 0; next(item); ++item) {
            const char *blob = it.slot >= 0 ? p.slots + (size_t)it.slot * p.slot_stride : p.shared_blobs[-1 - it.slot];
            const int kblocks = it.kblocks;
            auto expand = [&](auto phase_) {
                constexpr int kPhase = decltype(phase_)::value;
                constexpr int kRawBlocks = kPhase == 1 ? 4 : 2;           // k-blocks of one fetch of codes
                // GEMM 1: rows of eight g, eight u, ..; GEMM 2: rows f, 64 of the first column group, 64 of the second
                const int f_row = kPhase == 1 ? it.m0 + (row >> 4) * 8 + (row & 7) : (row & 63);
                const int part = (row >> 3) & 1, cg = row >> 6;
                const char *sc_base = kPhase == 1 ? blob + (size_t)f_row * ub + scales + (size_t)part * (p.d / 32)
                                                 : blob + (size_t)f_row * ub + scales + 2 * (size_t)(p.d / 32) + (size_t)(it.m0 / 64 + cg) * 2;
                // the scale of the next k-block is in flight while this one is expanded
                auto scale_of = [&](int kb) -> uint32_t {
                    if (kPhase == 1)
                        return f_row < p.F && kb < kblocks ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(sc_base) + kb) : 0u;
                    return kb * kBK + f_row < p.F ? (uint32_t)__ldg(reinterpret_cast<const uint16_t *>(sc_base + (size_t)kb * kBK * ub)) : 0u;
                };
                uint32_t sc = scale_of((group - (int)n0) & (kExpandGroups - 1));
                bool ok = true;
                for (int kr = 0; kr < kblocks && ok; kr += kRawBlocks, ++rn) {
                    const uint32_t rs = rn % kRawStages;
                    ok = mbar_wait(rfull0 + 8 * rs, (rn / kRawStages) & 1u, abort_flag);
                    for (int sub = (group - (int)n0 - kr) & (kExpandGroups - 1); sub < kRawBlocks && kr + sub < kblocks && ok; sub += kExpandGroups) {
                        const int kb = kr + sub;
                        const uint32_t n = n0 + (uint32_t)kb, s = n % kStages;
                        if (n >= (uint32_t)kStages)
                            ok = mbar_wait(empty0 + 8 * s, ((n / kStages) - 1u) & 1u, abort_flag);
                        if (!ok)
                            break;
                        const uint32_t ss = sc * 0x10001u;
                        const uint32_t raw = raw_s + rs * kRawBytes, a_dst = ring_s + s * kStageBytes + row * 128;
                        const uint32_t x = (uint32_t)(row & 7);      // = f mod 8 in both phases
                        if (kPhase == 1) {
                            // 64 columns = pieces 2 sub, 2 sub + 1 of this row's 128 bytes of codes -> eight pieces of bf16
                            const uint32_t src = raw + row * 128;
#pragma unroll
                            for (int h = 0; h < 2; ++h) {
                                const uint4 c4 = lds128(src + (((2 * sub + h) ^ x) << 4));
                                const uint32_t cw[4] = {c4.x, c4.y, c4.z, c4.w};
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    uint32_t P[4];
                                    expand8(cw[i], ss, P);
                                    sts128(a_dst + (((4 * h + i) ^ x) << 4), P[0], P[1], P[2], P[3]);
                                }
                            }
                        } else {
                            // one f, one group of 64 columns; nibble q of word w is column 8 q + w
                            const uint32_t src = raw + (sub * 64 + (row & 63)) * 128;
                            const uint32_t pc0 = (uint32_t)((it.m0 / 32) & 7) + 2u * cg;      // first piece of the group in its 128 bytes
                            const uint4 ca = lds128(src + ((pc0 ^ x) << 4)), cb = lds128(src + (((pc0 + 1) ^ x) << 4));
                            // (half of the nibbles at a time, to save registers)
#pragma unroll
                            for (int side = 0; side < 2; ++side) {
                                const uint32_t cw[8] = {ca.x >> (8 * side), ca.y >> (8 * side), ca.z >> (8 * side), ca.w >> (8 * side),
                                                        cb.x >> (8 * side), cb.y >> (8 * side), cb.z >> (8 * side), cb.w >> (8 * side)};
                                uint32_t o[4][4];
#pragma unroll
                                for (int i = 0; i < 4; ++i) {
                                    uint32_t P[2], Q[2];
                                    expand4(cw[2 * i], ss, P);
                                    expand4(cw[2 * i + 1], ss, Q);
#pragma unroll
                                    for (int q = 0; q < 2; ++q) {
                                        o[q][i] = __byte_perm(P[q], Q[q], 0x5410);
                                        o[q + 2][i] = __byte_perm(P[q], Q[q], 0x7632);
                                    }
                                }
#pragma unroll
                                for (int q = 0; q < 4; ++q)
                                    sts128(a_dst + ((((q & 1) + 2 * side + 4 * (q >> 1)) ^ x) << 4), o[q][0], o[q][1], o[q][2], o[q][3]);
                            }
                        }
                        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");       // the tensor cores read what was just stored
                        __syncwarp();
                        if (lane == 0) {
                            if (rank == 0)
                                mbar_arrive(full0 + 8 * s);
                            else
                                mbar_arrive_cluster(cluster_addr(full0 + 8 * s, 0));
                        }
                        sc = scale_of(kb + kExpandGroups);       // (in front of the arrival, that would wait for it)
                    }
                    if (lane == 0)
                        mbar_arrive(rempty0 + 8 * rs);
                }
            };
            if (PHASE ? PHASE == 1 : it.phase == 1)
                expand(Const<1>());
            else
                expand(Const<2>());
            n0 += (uint32_t)kblocks;
        }
    } else if (FMT == 1 && warp == 2 + kEpilogueWarps + 4 * kExpandGroups) {
        // ============================================================ fetch of 4-bit codes
        uint32_t rn = 0;
        for (uint32_t item = 0; next(item); ++item) {
            const int phase = PHASE ? PHASE : it.phase;
            const CUtensorMap *map_w = p.maps + (it.slot >= 0 ? kMapSlots0 : kMapShared0 + 2 * (-1 - it.slot)) + (phase - 1);
            const int slot = it.slot >= 0 ? it.slot : 0;
            for (int kb = 0; kb < it.kblocks; kb += phase == 1 ? 4 : 2, ++rn) {
                const uint32_t rs = rn % kRawStages;
                const bool ok = rn < (uint32_t)kRawStages || mbar_wait(rempty0 + 8 * rs, ((rn / kRawStages) - 1u) & 1u, abort_flag);
                if (!__all_sync(0xffffffffu, ok))
                    break;
                if (lane == 0) {
                    const uint32_t dst = raw_s + rs * kRawBytes, bar = rfull0 + 8 * rs;
                    mbar_expect(bar, kRawBytes);
                    if (phase == 2)
                        tma_load_3d(dst, map_w, it.m0 / 256 * 128, kb * kBK, slot, bar);
                    else
                        tma_load_5d(dst, map_w, kb * 32, 0, 0, it.m0 / 8, slot, bar);
                }
                __syncwarp();
            }
        }
    }

    if (warp == 2)           // (no kernel of the chain ends before the one ahead of it has)
        asm volatile("griddepcontrol.wait;" ::: "memory");
    // ---- everyone is done with tensor memory: free it
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // (a pair: neither CTA goes while the other may still signal it or read its shared memory)
    if (CG == 2)
        cluster_sync_all();
    if (warp == 2) {
        if (CG == 1)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(2 * NT));
        else
            asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(2 * NT));
    }
    if (*abort_flag && tid == 0)
        atomicExch(p.err, MELINOE_ERR_TIMEOUT);
}

// y_t = sum_j gate[t][j] * Z[inv_pos[t*k+j]] + sum_s Z[T*k + s*T + t], fp32 in rank order, bf16 out (GATED = false: the
// rows of Z are weighted already).  Memory-bound: full occupancy (32 registers a thread), the rows of four experts at a
// time in flight; work is (token, 1024 columns).  DEPTH 8: where there are no more than a few blocks per SM, so that latency is
// the time, eight rows at a time (128 tokens of 8 experts: 3.7 -> 2.9 us).
template <bool GATED, int DEPTH>
__global__ void __launch_bounds__(256, 32 / DEPTH) combine_rows_kernel(const DevPlan *plan, const float *__restrict__ gate,
                                                              const int32_t *__restrict__ inv_pos, const float *__restrict__ zs,
                                                              uint16_t *out, int T, int d, int k, int n_shared)
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const bool ok = plan->status == MELINOE_OK;
    for (int t = blockIdx.x; t < T; t += gridDim.x) {
        const int32_t *pos = inv_pos + t * k;
        auto gate_of = [&](int j) { return GATED ? gate[t * k + j] : 1.0f; };
        for (int c = (blockIdx.y * 256 + threadIdx.x) * 4; c < d; c += gridDim.y * 1024) {
            float4 y = make_float4(0.f, 0.f, 0.f, 0.f);
            if (ok) {
                const float *zc = zs + c;
                auto row = [&](int r) { return *reinterpret_cast<const float4 *>(zc + (size_t)r * d); };
                auto add = [&](float g, const float4 &z) {
                    y.x = fmaf(g, z.x, y.x);
                    y.y = fmaf(g, z.y, y.y);
                    y.z = fmaf(g, z.z, y.z);
                    y.w = fmaf(g, z.w, y.w);
                };
                int j = 0;
                if (DEPTH == 8)
                    for (; j + 8 <= k; j += 8) {
                        float4 z[8];
                        float g[8];
#pragma unroll
                        for (int i = 0; i < 8; ++i) {
                            z[i] = row(pos[j + i]);
                            g[i] = gate_of(j + i);
                        }
#pragma unroll
                        for (int i = 0; i < 8; ++i)
                            add(g[i], z[i]);
                    }
                for (; j + 4 <= k; j += 4) {
                    const float4 z0 = row(pos[j]), z1 = row(pos[j + 1]), z2 = row(pos[j + 2]), z3 = row(pos[j + 3]);
                    add(gate_of(j), z0);
                    add(gate_of(j + 1), z1);
                    add(gate_of(j + 2), z2);
                    add(gate_of(j + 3), z3);
                }
                if (j + 2 <= k) {
                    const float4 z0 = row(pos[j]), z1 = row(pos[j + 1]);
                    add(gate_of(j), z0);
                    add(gate_of(j + 1), z1);
                    j += 2;
                }
                if (j < k)
                    add(gate_of(j), row(pos[j]));
                for (int s = 0; s < n_shared; ++s)
                    add(1.0f, row(T * k + s * T + t));
            }
            uint2 o;
            o.x = bf16_rne(y.x) | (bf16_rne(y.y) << 16);
            o.y = bf16_rne(y.z) | (bf16_rne(y.w) << 16);
            *reinterpret_cast<uint2 *>(out + (size_t)t * d + c) = o;
        }
    }
}

// Launch with programmatic stream serialisation (the kernel waits for the one ahead itself) and, for CG = 2, clusters of
// two CTAs on neighbouring SMs.
template <typename... Params, typename... Args>
cudaError_t launch_after(cudaStream_t stream, void (*kernel)(Params...), dim3 grid, int threads, size_t smem, int cluster, const Args &...args)
{
    cudaLaunchConfig_t lc = {};
    lc.gridDim = grid;
    lc.blockDim = dim3(threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = stream;
    cudaLaunchAttribute attr[2];
    int n = 0;
    if (pdl_enabled()) {
        attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[n++].val.programmaticStreamSerializationAllowed = 1;
    }
    if (cluster > 1) {
        attr[n].id = cudaLaunchAttributeClusterDimension;
        attr[n].val.clusterDim.x = cluster;
        attr[n].val.clusterDim.y = 1;
        attr[n++].val.clusterDim.z = 1;
    }
    lc.attrs = attr;
    lc.numAttrs = n;
    const cudaError_t e = cudaLaunchKernelEx(&lc, kernel, args...);
    count_launch();
    return e;
}

constexpr size_t gemm_smem(int fmt)
{
    return (size_t)gemm_stages(fmt) * kStageBytes + (fmt ? kRawStages * kRawBytes : 0) + 1024;
}

template <int CG, int FMT, int PHASE>
cudaError_t gemm_launch(cudaStream_t stream, int n_sms, const GemmParams &p)
{
    return launch_after(stream, ffn_gemm_kernel<CG, FMT, PHASE>, dim3(n_sms / CG * CG), gemm_threads(FMT), gemm_smem(FMT), CG, p);
}

template <int FMT>
cudaError_t gemm_launch(cudaStream_t stream, int n_sms, int ctas, bool apart, const GemmParams &p)
{
    if (ctas == 1)
        return gemm_launch<1, FMT, 0>(stream, n_sms, p);
    if (!apart)
        return gemm_launch<2, FMT, 0>(stream, n_sms, p);
    const cudaError_t e = gemm_launch<2, FMT, 1>(stream, n_sms, p);
    return e != cudaSuccess ? e : gemm_launch<2, FMT, 2>(stream, n_sms, p);
}

template <int CG, int FMT, int PHASE>
cudaError_t gemm_configure()
{
    return cudaFuncSetAttribute(ffn_gemm_kernel<CG, FMT, PHASE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)gemm_smem(FMT));
}

}  // namespace

bool ffn_gemm_supported(int d, int F) { return d % 256 == 0 && F % kUnitRows == 0; }

cudaError_t ffn_gemm_configure()
{
    const cudaError_t e[] = {gemm_configure<1, 0, 0>(), gemm_configure<1, 1, 0>(), gemm_configure<2, 0, 0>(), gemm_configure<2, 1, 0>(),
                             gemm_configure<2, 0, 1>(), gemm_configure<2, 0, 2>(), gemm_configure<2, 1, 1>(), gemm_configure<2, 1, 2>()};
    for (cudaError_t r : e)
        if (r != cudaSuccess)
            return r;
    return cudaSuccess;
}

cudaError_t launch_ffn_gemm(cudaStream_t stream, int n_sms, int fmt, bool single_only, const GemmParams &p, int T, int k)
{
    const long long pairs_of_all = (long long)T * k;     // (token, expert) pairs
    // CTA pairs for bf16 slots (MELINOE_MOE_GEMM_SINGLE in the environment keeps them on single CTAs).  4-bit slots: single CTAs while
    // an expert has few tokens.  They expand the codes without waiting for a peer's stores to be seen, but take chunks of 128
    // tokens instead of 256 and expand a tile again for each.  (d 2048, d_ff 1024, 64 experts, 8 per token, us a pass, pairs and single
    // CTAs: 16 tokens 67 and 55, 64 tokens 78 and 67, 200 tokens 101 and 95, 512 tokens 129 and 132, 2048 tokens 327 and 383.)
    const int ctas = fmt != 0 ? (pairs_of_all > 32ll * p.E ? 2 : 1) : single_only ? 1 : 2;
    // A launch for each GEMM where GEMM 1's reductions are short and its tiles many: there the way from one item to the next counts
    // (see ffn_gemm_kernel) and a last round that is not full does not.  us a pass, one launch and two (experts, per token, tokens):
    // bf16, d 512, d_ff 512 (32, 4, 400) 35.2 and 35.9, d_ff 1024 51.7 and 46.4; d 256, d_ff 4096 (8, 2, 800) 61.6 and 58.0; d 768,
    // d_ff 768 (32, 4, 400) 52.8 and 50.4; d 1024 (8, 2, 400), d_ff 4096 71.3 and 69.8, d_ff 8192 109.8 and 106.5, d_ff 1024 (32, 4, 400)
    // 65.1 and 66.7; d 4096, d_ff 1024 (16, 2, 400) 103 and 109.  4-bit, d 512, d_ff 8192 (8, 2, 2000) 201 and 183; d 1024, d_ff 6144
    // (8, 2), 400 tokens 119.0 and 113.8, 2000 tokens, two chunks for an expert, 225.8 and 234.2; d 2048, d_ff 8384 (8, 2, 160) 190.8 and 187.9.
    const bool apart = p.F > 512 && (p.d < 1024 || (pairs_of_all <= 256ll * p.E && (fmt != 0 ? 2 * p.F >= 5 * p.d : p.d == 1024 && p.F >= 6 * p.d)));
    return fmt != 0 ? gemm_launch<1>(stream, n_sms, ctas, apart, p) : gemm_launch<0>(stream, n_sms, ctas, apart, p);
}

cudaError_t launch_combine_rows(cudaStream_t stream, const DevPlan *plan, const float *gate, const int32_t *inv_pos,
                                const float *zs, uint16_t *out, int T, int d, int k, int n_shared, int n_sms)
{
    // a whole row per block once that fills the GPU
    const int x = T < 8 * n_sms ? T : 8 * n_sms, y = T < 4 * n_sms ? (d + 1023) / 1024 : 1;
    const bool deep = x * y <= 4 * n_sms;
    return launch_after(stream, gate ? (deep ? combine_rows_kernel<true, 8> : combine_rows_kernel<true, 4>)
                                     : (deep ? combine_rows_kernel<false, 8> : combine_rows_kernel<false, 4>),
                        dim3(x, y), 256, 0, 1, plan, gate, inv_pos, zs, out, T, d, k, n_shared);
}

}  // namespace melinoe
