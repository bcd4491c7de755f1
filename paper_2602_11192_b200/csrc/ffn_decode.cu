// Decode expert FFN (Eq. 3) with the gate-weighted combine (Eq. 2) fused in: one launch serves up
// to 8 tokens.  The work is reading every needed expert once (from HBM, or over the host link for
// an expert that is not resident), so the kernel is built around one contiguous stream per SM and
// no synchronisation between SMs until the very end.
//
// Layout of an expert ("blob", written by melinoe_moe_pack_expert): for f = 0 .. d_ff - 1 the
// three rows that belong to hidden unit f back to back,
//     W_g[f][0..d) | W_u[f][0..d) | W_d[0..d)[f]   (the last one is row f of W_d transposed),
// 6 d bytes, and inside each row the 16-byte pieces of every 128-byte group are stored at
// position (piece xor (f mod 8)).  Consequences:
//   - the rows f0 .. f0 + m - 1 are ONE contiguous byte range, fetched by one bulk copy;
//   - everything hidden unit f contributes to the output, gate * SiLU(g_f) * u_f * W_d[:, f], can be
//     formed by the SM that read those three rows: no other SM is involved, so the d_ff rows of all
//     requested experts are simply dealt out evenly (single-row granularity) and every CTA ends up
//     with a partial output vector;
//   - eight consecutive rows, read at the same logical column, fall into eight different groups
//     of shared-memory banks (the xor), so the tensor-core fragment loads (ldmatrix) are free of
//     bank conflicts although the rows sit at a pitch that is a multiple of 128 bytes.
//
// One CTA per SM: 16 consumer warps and one producer warp.  The consumers work on a tile together, or, where a tile is little work, in
// two or four groups on tiles of their own (decode_groups).
//   producer  one thread; per tile (up to 8 rows f of one expert) one cp.async.bulk into a ring
//             stage, completion on the stage's mbarrier.  A missed expert's rows come straight from
//             the page-locked host store (the device reads host memory over the link).
//   gate/up   D[16 x 8] = [W_g rows ; W_u rows] (16 x d) * x^T (d x 8 tokens) on mma.sync m16n8k16
//             (bf16 in, fp32 accumulate): decode is one multiply-add per weight byte pair, far
//             below what even this legacy tensor path delivers, so it is free compute.  The warps
//             split the columns; their partial tiles meet in shared memory once per tile and every
//             warp forms the complete g_f, u_f (thread-local: a thread holds g and u of the same f and
//             the same two tokens), then h = gate[token][expert] * SiLU(g) * u, rounded once to bf16.
//             The gate is folded in here so that all experts accumulate into one output tile.
//   down      Y[c][t] += sum_f W_d^T[f][c] * h[f][t]: the same 8 rows f are now the K dimension
//             (padded to 16 with zeros), A = W_d^T rows read transposed (ldmatrix.trans), every warp
//             owns d / NW output columns (of a group's warps, d / 8 or d / 4) and keeps their fp32 accumulators in registers for the
//             whole kernel.
//   fetched   a tile of a missed expert that stays resident after the call is also stored into its
//   experts   cache slot (bulk copy shared -> global) while it is being computed with.
//   combine   every CTA adds its partial [tokens][d] into the call's accumulator in global memory as
//             64-bit fixed point (units of 2^-40; integer atomics: the sum is exact, so it does not
//             depend on the order of arrival and results are bit-identical from run to run), counts
//             itself out and exits; whoever finds all the others gone
//             converts the sums to bf16, writes the output and clears accumulator and counter.  No CTA
//             ever waits for another.  The counting out is per consumer warp: warp w of every CTA owns the same
//             columns, has a counter of its own, and the last of them converts those columns: sixteen
//             warps, of whichever CTAs were last, share the conversion and no warp waits for its CTA.
//   4-bit     the same structure on 4-bit blobs (melinoe_moe_pack_expert_q4): the codes are expanded in
//   blobs     registers on their way into the tensor-core fragments, see consume_q4 below.
//
// Every wait is bounded: when an mbarrier or the wait for the plan does not complete in time the warp
// raises the CTA's abort flag, later waits fall through, copies in flight are given a bounded time
// to land, the kernel ends normally and the error word tells the host.

#include "kernels.cuh"

namespace melinoe {

namespace {

constexpr int kMaxStages = 8;
// Bound of every wait, in SM clock cycles (about 2 s).
constexpr long long kWaitLimitCycles = 4000000000ll;

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

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

// Bounded wait.  Returns false (and raises the CTA's abort flag) when the limit runs out.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *abort_flag)
{
    if (mbar_try(bar, parity))
        return true;
    if (*abort_flag)
        return false;
    const long long t0 = clock64();
    for (;;) {
        for (int i = 0; i < 64; ++i)
            if (mbar_try(bar, parity))
                return true;
        if (*abort_flag)
            return false;
        if (clock64() - t0 > kWaitLimitCycles) {
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

__device__ __forceinline__ void ldmatrix_x4(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
__device__ __forceinline__ void ldmatrix_x4_trans(uint32_t addr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3)
{
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(addr));
}
// D(16x8) += A(16x16) * B(16x8), bf16 in, fp32 accumulate.
__device__ __forceinline__ void mma_16816(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1)
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t lds32(uint32_t addr)
{
    uint32_t v;
    asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(addr));
    return v;
}

__device__ __forceinline__ uint4 lds128(uint32_t addr)
{
    uint4 v;
    asm volatile("ld.shared.v4.b32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr));
    return v;
}
__device__ __forceinline__ uint32_t lds16(uint32_t addr)
{
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(addr));
    return v;
}

// Eight 4-bit codes (one 32-bit word: element j in nibble j) into bf16 weights, as four registers
// P[j] = (element j, element j + 4).  A nibble n placed in the mantissa of 0x4300 is the bf16 number
// 128 + n; minus 136 is the integer n - 8, exactly; times the group's scale, rounded once to nearest
// even, is the weight the format defines.  ss = the scale in both halves.
__device__ __forceinline__ void dequant8(uint32_t w, uint32_t ss, uint32_t (&P)[4])
{
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        uint32_t t = ((w >> (4 * j)) & 0x000f000fu) | 0x43004300u;
        asm("sub.rn.bf16x2 %0, %0, %1;" : "+r"(t) : "r"(0x43084308u));
        asm("mul.rn.bf16x2 %0, %1, %2;" : "=r"(P[j]) : "r"(t), "r"(ss));
    }
}

// Tensor memory as a per-thread operand store: 32 consecutive 32-bit columns of the thread's own lane.
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32])
{
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
        "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
        "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};"
        ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
          "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]),
          "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]),
          "r"(r[30]), "r"(r[31])
        : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_ld4(uint32_t taddr, uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3)
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3)
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t bf16_rne(float v)
{
    uint32_t u = __float_as_uint(v);
    u += 0x7fffu + ((u >> 16) & 1u);
    return u >> 16;
}

__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void *src, uint32_t bytes, uint32_t bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(dst), "l"(src), "r"(bytes), "r"(bar)
                 : "memory");
}
__device__ __forceinline__ void bulk_s2g(void *dst, uint32_t src, uint32_t bytes)
{
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Add without a return value, on the global address space (a generic atomicAdd compiles to the
// returning form on the generic space).
__device__ __forceinline__ void red_add_u64(unsigned long long *addr, unsigned long long v)
{
    asm volatile("red.global.add.u64 [%0], %1;" ::"l"(__cvta_generic_to_global(addr)), "l"(v) : "memory");
}
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }

template <int N>
struct Count {
    static constexpr int value = N;
};

constexpr int NW = 16;                           // consumer warps
// Groups of consumer warps.  A tile takes its warps through two barriers, a sum and the division of SiLU, one behind the other, while
// a scheduler's other warps wait at the same place.  So the warps work in two groups of eight (bf16 slots up to d_model 512: four of
// four), on a tile each, in turn: the groups drift apart, one computes while the other waits, and h is formed by fewer warps.  The number
// of stages is a multiple of the groups', so that a stage belongs to one.  At the end the groups' sums of the same columns meet in
// shared memory, and from then on warp w of group g of n stands for warp n w + g of sixteen.
// One group
//   - with bf16 slots where a call may have less than kGroupRows rows for a CTA (`rows`: those of its top_k and shared experts; a launch of
//     one compute group may have fewer, which beside its transfers was not to be measured): a tile is over sooner with sixteen warps (d 1024,
//     one token of 4 experts, 8 layers, one group and two: d_ff 256, 7 rows, 85.8 and 90.4 us; d_ff 768, 21 rows, 108.8 and 108.3; d 256,
//     d_ff 512, 8 tokens 173 and 152); four from twice as many on (d 256, 14 rows 80.9 with two, 82.6 with four);
//   - where a warp's output columns of two would not fit its 96 registers: 4-bit slots of d_model 4096, and of 2048 with more
//     than 4 tokens (with spills 428 us instead of 387 for one token of 16 layers, 894 instead of 721 for 8 of 8);
//   - with 4-bit slots of d_model 2048 where a CTA may have a single row, so that the second group would only be met at the end (one token of 2
//     experts, 4 layers, one group and two: d_ff 64 45.2 and 46.9 us, d_ff 256, 3 rows, 48.5 and 48.4);
//   - where four stages of tiles of eight rows do not fit, so that a group's next tile would not be on its way while it works: bf16 slots
//     beyond d_model 1024 (where HBM is the limit from 2048 on).
// Measured, against one group with the width taken at run time (which spilled), us: bf16, d 512, d_ff 8192, 4 tokens of 4 experts, 4 layers
// 535 -> 256; d 256 the same 545 -> 159 (206 in two groups); d 1024, d_ff 11136, 7 tokens of 2, 3 layers 374 -> 283; a token of a tiny
// layer 11.2 -> 9.6; 4-bit, d 2048, d_ff 1024, one token of 8, 16 layers 387 -> 341; d 1024, d_ff 2048, 8 layers 288 -> 175.
constexpr int kGroupRows = 12;
__host__ __device__ constexpr int decode_groups(int d, int tokens, int fmt, int rows_per_cta)
{
    return fmt == 0 ? (d > 1024 || rows_per_cta < kGroupRows ? 1 : d <= 512 && rows_per_cta >= 2 * kGroupRows ? 4 : 2) : d <= 1024 || (d == 2048 && tokens <= 4 && rows_per_cta >= 2) ? 2 : 1;
}
constexpr int kThreads = (NW + 1) * 32;          // + the producer warp
constexpr int kBufPitch = 130;                   // floats between the warps' partial tiles (keeps the column sums conflict-free)

// ---------------------------------------------------------------------------------------------------
// The consumer warps' work on 4-bit blobs.  One hidden unit f is a unit of geo.row_bytes bytes: the
// codes of W_g[f], W_u[f], W_d[:, f] (d / 2 bytes each) and their scales (one bf16 per 64 elements).
// A 32-bit word of codes is eight consecutive elements and expands into four registers that pair
// element j with element j + 4 (dequant8).  A tensor-core operand register holds two neighbours
// along the contraction, and a sum does not care in which order its terms are met, so:
//   gate/up   the contraction runs over the columns: a thread takes one word of its W_g row and one of
//             its W_u row (columns c .. c + 7) and feeds two products, the k-slots being columns
//             (c, c + 4, c + 1, c + 5) and (c + 2, c + 6, c + 3, c + 7); the hidden state was staged
//             in the same pairing, so one 16-byte load is the matching token operand of both.  The
//             warps split the columns in steps of 32.
//   down      the contraction runs over f, and the two halves of a register are two COLUMNS of one f.
//             They are made two k-slots of that f, and the token operand carries h[f][t] in the first
//             of them for the output columns n = 0..3 (tokens 0..3) and in the second for n = 4..7
//             (again tokens 0..3): the product's left half is column j of every row of output, its right
//             half column j + 4.  One product so covers 8 hidden units x 32 output columns x 4 tokens;
//             tokens 4..7 take a second product.  The warps split the columns in steps of 32.  (The codes
//             of W_d[:, f] are stored interleaved within every 64, nibble j of word g being column
//             g + 8 j, so that the lanes of one product row own neighbouring output columns.)

// One tile as the loop sees it.
struct Q4Tile {
    uint32_t stage, st;   // shared-memory address of its ring stage, index of the stage
    int m, f0;            // rows, first hidden unit
    int req;              // its request
    bool stored;          // this thread issued the tile's store into the cache slot
};

// NG: groups of warps; TG: 1 = at most 4 tokens
template <int MT_, int NG, int TG>
__device__ __forceinline__ void consume_q4(const DecParams &p, const DecGeometry &geo, const FastReq *s_req, float *s_sums, float *buf, uint32_t ring_s, uint32_t xs_s, uint32_t full0,
                                           uint32_t empty0, volatile int *abort_flag, int q_lo, int q_hi, unsigned long long *trace)
{
    constexpr int NWG = NW / NG;                                 // warps of a group
    constexpr int WS = MT_ / 2 * NG;                             // 32-column steps of a warp
    const int tid = threadIdx.x, lane = tid & 31, g = lane >> 2, tig = lane & 3;
    const int grp = NG == 1 ? 0 : tid / (32 * NWG), warp = (tid >> 5) & (NWG - 1);       // warp: within the group
    const int d = p.d, F = p.F;
    const int TR = geo.tile_rows, S = geo.n_stages, RB = geo.row_bytes, STAGE = geo.stage_bytes, XP = geo.x_pitch, Tc = geo.tokens;
    buf += grp * (NWG * kBufPitch);
    s_sums += grp * 128;
    float acc[WS][TG][4];
#pragma unroll
    for (int i = 0; i < WS; ++i)
#pragma unroll
        for (int j = 0; j < TG; ++j)
            acc[i][j][0] = acc[i][j][1] = acc[i][j][2] = acc[i][j][3] = 0.f;
    const bool has_tok = g < Tc, two = TG == 2 && Tc > 4;
    const uint32_t xrow = xs_s + g * XP + (warp * WS * 32 + tig * 8) * 2;
    const uint32_t sc_off = 3 * (uint32_t)(d / 2), sc_len = (uint32_t)(d / 32);     // scales: offset in the unit, bytes per vector
    const int t0 = g & 3, sh = g < 4 ? 0 : 16;

    // ---- the tiles of this CTA in order; taking one waits until it has landed and starts its copy into the slot
    int left = q_hi - q_lo;                         // rows still to take
    int a = q_lo / F, f0 = q_lo % F;
    uint32_t st = 0, ph = 0;                        // ring stage of the next tile and the parity of its barrier phase
    bool first = true;
    auto skip = [&](int m) {
        if (++st == (uint32_t)S) {
            st = 0;
            ph ^= 1u;
        }
        left -= m;
        f0 += m;
        if (f0 == F) {
            f0 = 0;
            ++a;
        }
    };
    if (grp == 1 && left > 0)
        skip(min(min(TR, F - f0), left));
    auto take = [&](Q4Tile &t) -> bool {
        if (left <= 0)
            return false;
        t.m = min(min(TR, F - f0), left);
        t.f0 = f0;
        t.st = st;
        t.stage = ring_s + st * STAGE;
        mbar_wait(full0 + 8 * st, ph, abort_flag);
        if (trace && first && tid == 0)
            trace[2] = globaltimer_ns();
        first = false;
        t.req = a;
        char *wb = s_req[a].wb;
        t.stored = wb != nullptr && tid % (32 * NWG) == 0;
        if (t.stored)
            bulk_s2g(wb + (size_t)f0 * RB, t.stage, (uint32_t)t.m * RB);
        skip(t.m);
        if (NG == 2 && left > 0)         // the other group's
            skip(min(min(TR, F - f0), left));
        return true;
    };
    // ---- gate/up of one tile: this warp's columns, into registers.  Rows the tile does not have read row 0;
    // their results are dropped when h is formed.
    auto gate_up = [&](const Q4Tile &t, float (&cg)[4][4]) {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            cg[i][0] = cg[i][1] = cg[i][2] = cg[i][3] = 0.f;
        const int rr = g < t.m ? g : 0;
        const uint32_t fx16 = (uint32_t)((t.f0 + rr) & 7) << 4;
        const uint32_t row = t.stage + rr * RB;
        // piece ws of the codes sits at ((ws & ~7) | ((ws ^ f) & 7)) * 16: the warp's first step, then xor per step
        const uint32_t ws0 = (uint32_t)(warp * WS);
        const uint32_t cbase = row + (ws0 & ~7u) * 16 + tig * 4, sbase = row + sc_off + (ws0 >> 1) * 2;
        uint32_t sg = 0, su = 0;
#pragma unroll
        for (int i = 0; i < WS; ++i) {
            const uint32_t wsl = (ws0 & 7u) + (uint32_t)i;
            const uint32_t off = ((wsl << 4) ^ fx16) & 0x70u, hi = (wsl >> 3) * 128u;
            const uint32_t wg = lds32(cbase + hi + off);
            const uint32_t wu = lds32(cbase + hi + off + (uint32_t)(d / 2));
            if ((i & 1) == 0) {
                sg = lds16(sbase + (i >> 1) * 2) * 0x10001u;
                su = lds16(sbase + (i >> 1) * 2 + sc_len) * 0x10001u;
            }
            uint4 xb = make_uint4(0u, 0u, 0u, 0u);
            if (has_tok)
                xb = lds128(xrow + i * 64);
            uint32_t Pg[4], Pu[4];
            dequant8(wg, sg, Pg);
            dequant8(wu, su, Pu);
            mma_16816(cg[(2 * i) & 3], Pg[0], Pu[0], Pg[1], Pu[1], xb.x, xb.y);
            mma_16816(cg[(2 * i + 1) & 3], Pg[2], Pu[2], Pg[3], Pu[3], xb.z, xb.w);
        }
    };
    // The warps' partial tiles meet in shared memory: every warp of the group stores its 128 partial values, sums 8 NG of the 128
    // over the group's warps (4 / NG lanes per value, each adding four warps' parts in warp order, then a fixed tree), and reads the
    // complete tile.  Two named barriers of the group order this.  The buffers alternate from tile to tile, though one would do: its 8 KB
    // go to the ring then, which is worth 1 to 2 % up to d_model 2048, but a fourth stage at 4096 makes one token slower (2 experts of
    // d_ff 1024, 4 layers 84 -> 92 us).  (Measured and dropped: counting mbarriers in their place, with
    // the loop running one tile ahead so that a warp has other work between arriving and waiting -- the
    // hardware barrier is the cheaper way for 16 warps to meet; and h formed once per tile by the summing
    // warps instead of by every warp for itself -- it lengthens the path between the two barriers.)
    auto store_partials = [&](const float (&cg)[4][4], uint32_t sel) {
        float *b = buf + sel * (NW * kBufPitch) + warp * kBufPitch;
#pragma unroll
        for (int i = 0; i < 4; ++i)
            b[i * 32 + lane] = (cg[0][i] + cg[1][i]) + (cg[2][i] + cg[3][i]);
    };
    auto column_sums = [&](uint32_t sel) {
        const float *b = buf + sel * (NW * kBufPitch);
        constexpr int kOwn = 8 * NG;                         // values of a warp
        const int e = warp * kOwn + (lane & (kOwn - 1)), pg = lane / kOwn;
        float v = b[(pg * 4) * kBufPitch + e];
        v += b[(pg * 4 + 1) * kBufPitch + e];
        v += b[(pg * 4 + 2) * kBufPitch + e];
        v += b[(pg * 4 + 3) * kBufPitch + e];
        if (NG == 1)
            v += __shfl_xor_sync(0xffffffffu, v, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 16);
        if (lane < kOwn)
            s_sums[e] = v;
    };
    // ---- h of the tile from the complete sums, then the down product
    auto down = [&](const Q4Tile &t) {
        // g_f[t] and u_f[t] of the tile sit at (t & 1) * 32 + 4 f + (t >> 1) and 64 further on (the
        // accumulator layout of the product).  This thread needs h of f = tig, tig + 4 for token g mod 4
        // (and that token + 4).
        const float *sums = s_sums;      // (one buffer: whoever writes the next tile's is behind a barrier that everyone enters behind this)
        // (h rounded to bf16 once, to nearest even; it goes to the register half of this thread's output column)
        auto hval = [&](int f, int tk) -> uint32_t {
            const int o = (tk & 1) * 32 + f * 4 + (tk >> 1);
            const float vg = sums[o], vu = sums[64 + o];
            const float gt = s_req[t.req].gate[tk];
            float h = __fdividef(vg, 1.0f + __expf(-vg)) * vu * gt;
            if (f >= t.m || gt == 0.0f)
                h = 0.f;
            uint32_t r;
            asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(sh ? h : 0.f), "f"(sh ? 0.f : h));
            return r;
        };
        const uint32_t b0 = hval(tig, t0), b1 = hval(tig + 4, t0);
        uint32_t b0h = 0u, b1h = 0u;
        if (two) {
            b0h = hval(tig, t0 + 4);
            b1h = hval(tig + 4, t0 + 4);
        }
        const int ra = tig < t.m ? tig : 0, rb = tig + 4 < t.m ? tig + 4 : 0;
        const uint32_t fa16 = (uint32_t)((t.f0 + ra) & 7) << 4, fb16 = (uint32_t)((t.f0 + rb) & 7) << 4;
        const uint32_t rowa = t.stage + ra * RB, rowb = t.stage + rb * RB;
        // block = 64 output columns = one scale group = two 16-byte pieces of codes; this thread's word is in piece
        // 2 block + g / 4
        const uint32_t blk0 = (uint32_t)(warp * WS) >> 1, pc0 = blk0 * 2 + (uint32_t)(g >> 2);
        const uint32_t cofs = (uint32_t)d + (pc0 & ~7u) * 16 + (g & 3) * 4, sofs = sc_off + 2 * sc_len + blk0 * 2;
#pragma unroll
        for (int b = 0; b < WS / 2; ++b) {
            // (pc0 + 2 b) & 7 = (pc0 & 7) + 2 b for b < 4: pc0 & 7 is 0, 1 (four blocks), 0..5 (two), 0..7 (one)
            const uint32_t pin = ((pc0 & 7u) + 2u * (uint32_t)b) << 4;
            const uint32_t hi = (pin >> 7) * 128u;
            const uint32_t wa = lds32(rowa + cofs + hi + ((pin ^ fa16) & 0x70u));
            const uint32_t wb = lds32(rowb + cofs + hi + ((pin ^ fb16) & 0x70u));
            const uint32_t sa = lds16(rowa + sofs + b * 2) * 0x10001u;
            const uint32_t sb = lds16(rowb + sofs + b * 2) * 0x10001u;
            uint32_t Pa[4], Pb[4];
            dequant8(wa, sa, Pa);
            dequant8(wb, sb, Pb);
            mma_16816(acc[2 * b][0], Pa[0], Pa[1], Pb[0], Pb[1], b0, b1);
            mma_16816(acc[2 * b + 1][0], Pa[2], Pa[3], Pb[2], Pb[3], b0, b1);
            if (two) {
                mma_16816(acc[2 * b][TG - 1], Pa[0], Pa[1], Pb[0], Pb[1], b0h, b1h);
                mma_16816(acc[2 * b + 1][TG - 1], Pa[2], Pa[3], Pb[2], Pb[3], b0h, b1h);
            }
        }
        if (t.stored)
            bulk_wait_read();         // the slot store has read the stage
        __syncwarp();
        if (lane == 0)
            mbar_arrive(empty0 + 8 * t.st);
    };

    Q4Tile cur;
    float cg[4][4];
    for (uint32_t i = 0; take(cur); ++i) {
        gate_up(cur, cg);
        store_partials(cg, i & 1u);
        asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(NWG * 32) : "memory");      // every warp's partial sums of the tile are stored
        column_sums(i & 1u);
        asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(NWG * 32) : "memory");      // the complete sums of the tile are there
        down(cur);
    }
    if (trace && tid == 0)
        trace[3] = globaltimer_ns();
    // ---- two groups: group 0's warp takes the first half of the columns it shares with its partner, group 1's the second
    if constexpr (NG == 2) {
        constexpr int H = WS / 2;        // steps of a half
        asm volatile("bar.sync 3, %0;" ::"n"(NW * 32) : "memory");      // no tile is read any more: the ring is free
        auto at = [&](int to, int i, int tg) { return ring_s + (uint32_t)((((to * NWG + warp) * (WS / 2) + i) * TG + tg) * 512 + lane * 16); };
#pragma unroll
        for (int i = 0; i < H; ++i) {
#pragma unroll
            for (int tg = 0; tg < TG; ++tg)
                if (tg == 0 || two) {
                    uint32_t v[4];
#pragma unroll
                    for (int c = 0; c < 4; ++c)
                        v[c] = __float_as_uint(grp ? acc[i][tg][c] : acc[H + i][tg][c]);
                    asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(at(1 - grp, i, tg)), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]) : "memory");
                }
        }
        asm volatile("bar.sync 3, %0;" ::"n"(NW * 32) : "memory");
#pragma unroll
        for (int i = 0; i < H; ++i) {
#pragma unroll
            for (int tg = 0; tg < TG; ++tg)
                if (tg == 0 || two) {
                    const uint4 o = lds128(at(grp, i, tg));
                    const uint32_t ov[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
                    for (int c = 0; c < 4; ++c)      // (group 0's part first in both groups)
                        acc[i][tg][c] = grp ? __uint_as_float(ov[c]) + acc[H + i][tg][c] : acc[i][tg][c] + __uint_as_float(ov[c]);
                }
        }
    }
    // ---- this CTA's partial output into the call's accumulator (64-bit fixed point, as in the bf16 path).
    // Accumulator i of the warp is the 32-column step hb: block hb / 2, and within the
    // block's 64 columns (whose codes are stored interleaved: nibble j of word g is column g + 8 j),
    // column g + 16 (hb mod 2) + {0, 8} for the product's rows g, g + 8, plus 32 for the product's right
    // half (tig >= 2); its columns there are tokens 2 (tig mod 2), + 1.  Eight lanes of an add are
    // eight neighbouring columns.
    {
        unsigned long long *yacc = reinterpret_cast<unsigned long long *>(p.yacc);
        auto add = [&](int t, int c, float v) {
            if (t < Tc) {
                const long long fx = __float2ll_rn(v * 1099511627776.0f);
                red_add_u64(yacc + (size_t)t * d + c, (unsigned long long)fx);
            }
        };
#pragma unroll
        for (int i = 0; i < WS / NG; ++i) {
            const int hb = (warp * NG + grp) * (WS / NG) + i;
            const int c = (hb >> 1) * 64 + g + 16 * (hb & 1) + 32 * (tig >> 1);
            const int t = 2 * (tig & 1);
#pragma unroll
            for (int tg = 0; tg < TG; ++tg) {
                if (tg == 0 || two) {
                    add(t + 4 * tg, c, acc[i][tg][0]);
                    add(t + 4 * tg + 1, c, acc[i][tg][1]);
                    add(t + 4 * tg, c + 8, acc[i][tg][2]);
                    add(t + 4 * tg + 1, c + 8, acc[i][tg][3]);
                }
            }
        }
    }
}

// MT_: k-steps of the gate/up phase and m-tiles of the down phase per warp with all warps on a tile (d / 256).
// FMT: 0 = bf16 expert blobs, 1 = 4-bit blobs (melinoe_moe_pack_expert_q4), expanded in registers on
// the way into the tensor-core fragments.
// XT: 1 = the hidden states' tensor-core operand fragments are kept in tensor memory instead of shared
// memory (bf16 blobs of d_model from 3072 on: up to 64 KB of shared memory go to the ring instead, which makes the tiles that
// fit up to twice as high).
// NG, TG: 4-bit blobs, groups of consumer warps and of four tokens (see consume_q4).
template <int MT_, int FMT, int XT = 0, int NG = 1, int TG = 2>
__global__ void __launch_bounds__(kThreads, 1) ffn_decode_kernel(const __grid_constant__ DecParams p, const __grid_constant__ DecGeometry geo)
{
    static_assert(XT == 0 || (FMT == 0 && MT_ >= 12), "tensor-memory operands: bf16 blobs, d_model from 3072 on");
    __shared__ uint32_t s_tmem;
    extern __shared__ __align__(128) unsigned char smem[];
    __shared__ int s_abort, s_nact, s_last, s_deferred;
    __shared__ int s_hdr[4];                        // status, n_groups, first request, one past the last
    __shared__ FastReq s_req[kMaxReq];              // the launch's active requests
    __shared__ unsigned long long s_ready;
    __shared__ float s_sums[NG == 4 ? 512 : 256];
    __shared__ __align__(8) uint64_t s_bars[2 * kMaxStages + 1];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int d = p.d, F = p.F;
    const int G = (int)gridDim.x;
    const int TR = geo.tile_rows, S = geo.n_stages, RB = geo.row_bytes, STAGE = geo.stage_bytes, XP = geo.x_pitch;
    const int Tc = geo.tokens, tok0 = p.chunk * kTokPerVr;
    constexpr int MT = MT_;

    unsigned long long *trace = p.trace ? p.trace + (size_t)blockIdx.x * 8 : nullptr;
    if (trace && tid == 0)
        trace[0] = globaltimer_ns();

    // ring | staged hidden rows | the warps' partial gate/up tiles
    unsigned char *ring = smem;
    unsigned char *xs = smem + (size_t)S * STAGE;
    float *buf = reinterpret_cast<float *>(xs + (XT ? 0 : (size_t)Tc * XP));        // [NW][kBufPitch]
    // tables of a launch whose requests have to be matched with its tokens here (plans made for several launches); they
    // lie in the ring, whose first copies are issued once they have done their work
    struct MatchTables {
        DecReq raw[kMaxReq];
        float gate[kMaxReq][kTokPerVr];             // gate of (request, token of the launch); 0 = not routed
        unsigned match[kMaxReq];
        int32_t of_expert[kMaxReq];                 // request of an expert id (routed 0..E-1, shared E..), -1 = none
        int32_t idx[kTokPerVr * 32];
        float gw[kTokPerVr * 32];
    };
    MatchTables &tab = *reinterpret_cast<MatchTables *>(smem);
    const uint32_t ring_s = smem_u32(ring), xs_s = smem_u32(xs);
    const uint32_t full0 = smem_u32(s_bars), empty0 = full0 + 8 * kMaxStages, hzbar = empty0 + 8 * kMaxStages;
    volatile int *abort_flag = &s_abort;

    if (tid == 0) {
        s_abort = 0;
        s_nact = 0;
        for (int i = 0; i < kMaxStages; ++i) {
            mbar_init(full0 + 8 * i, 1);
            mbar_init(empty0 + 8 * i, NW / NG);
        }
        mbar_init(hzbar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (tid == 1)
        s_deferred = 0;
    // Nothing above reads what an earlier kernel wrote.  With programmatic stream serialisation this
    // CTA may be running while the kernel ahead of it in the stream (the planner) still is.  It does
    // not wait for that grid to drain (which costs microseconds) but acquires what the planner releases when the records
    // that this launch reads are complete: the plan's word, or for one token the records themselves.  The planner itself
    // has waited for everything ahead of it in the stream, so whatever else this kernel reads (hidden states, resident
    // weights) is in memory then.  A programmatically launched grid never
    // starts before every CTA of the grid ahead of it is running, and the planner waits for nobody
    // behind it, so the wait ends; it is bounded all the same.
    // This grid must not end before the planner's either, which is still writing cache state, token lists and
    // statistics when it announces the plan: whatever comes behind this kernel (the next planner, a preload, a copy of
    // the statistics) is ordered behind both by this kernel's end alone.  The producer's thread waits for it when its
    // last copy is on the way, where the wait costs nothing.
    auto planner_ended = [] { asm volatile("griddepcontrol.wait;" ::: "memory"); };
    if (p.wait_prior)
        planner_ended();
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const DevPlan *plan = p.plan;
    // One token: if every expert is resident, the requests' records come without that word and say themselves that they
    // are there (one round trip instead of two); otherwise as for more tokens.
    const int n_one = XT == 0 && p.fast && Tc == 1 ? p.k + p.n_shared : 0;
    bool got = true;
    if (tid < max(n_one, 1)) {
        got = false;
        const long long t0 = clock64();
        for (unsigned i = 0;; ++i) {
            if (n_one) {
                unsigned long long src, tag;
                asm volatile(
                    "{\n\t.reg .b128 v;\n\t"
                    "ld.acquire.gpu.global.b128 v, [%2];\n\t"
                    "mov.b128 {%0, %1}, v;\n\t}"
                    : "=l"(src), "=l"(tag)
                    : "l"(&plan->one[tid])
                    : "memory");
                if ((unsigned)(tag >> 32) == p.call_seq) {
                    FastReq r = {};
                    r.src = reinterpret_cast<const char *>(src);
                    r.gate[0] = __uint_as_float((unsigned)tag);
                    s_req[tid] = r;
                    got = true;
                    break;
                }
                if (i & 3u)             // (the word comes instead only where experts are fetched, which takes far longer)
                    continue;
            }
            unsigned long long v;
            asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(&plan->ready) : "memory");
            if ((unsigned)v == p.call_seq) {
                s_ready = v;
                break;
            }
            if (clock64() - t0 > kWaitLimitCycles) {
                s_abort = 1;
                break;
            }
        }
    }
    const bool quick = __syncthreads_and(got) != 0 && n_one > 0;
    const bool fast = quick || (p.fast && (p.group < 0 || ((s_ready >> 32) & 0xffu) != 0));

    // the producer's place: copies issued, ring stage of the next one and parity of its being free, rows left of this CTA's
    // share, request and row of the next one
    struct Feed {
        uint32_t n, st, ph;
        int left, a, f0;
        __device__ void begin(int rows, int F, int G)
        {
            const int lo = (int)((long long)blockIdx.x * rows / G), hi = (int)((long long)(blockIdx.x + 1) * rows / G);
            n = st = 0;
            ph = 1;
            left = hi - lo;
            a = lo / F;
            f0 = lo % F;
        }
    } feed;
    feed.n = 0;
    auto issue = [&] {
        const int m = min(min(TR, F - feed.f0), feed.left);
        const uint32_t bytes = (uint32_t)m * RB;
        mbar_expect(full0 + 8 * feed.st, bytes);
        bulk_g2s(ring_s + feed.st * STAGE, s_req[feed.a].src + (size_t)feed.f0 * RB, bytes, full0 + 8 * feed.st);
        ++feed.n;
        if (++feed.st == (uint32_t)S) {
            feed.st = 0;
            feed.ph ^= 1u;
        }
        feed.left -= m;
        feed.f0 += m;
        if (feed.f0 == F) {
            feed.f0 = 0;
            ++feed.a;
        }
    };

    // ---- everything the launch needs to know, in one round trip to memory
    if (quick) {
        if (tid == kThreads - 1) {
            s_hdr[0] = MELINOE_OK;
            s_hdr[1] = 1;
            s_hdr[2] = 0;
            s_hdr[3] = n_one;
            s_nact = n_one;
        }
        // the first copies go out while the others stage the hidden state
        if (warp == NW && lane == 0) {
            feed.begin(n_one * F, F, G);
            while (feed.left > 0 && feed.n < (uint32_t)S)
                issue();
        }
    } else if (fast) {
        // the plan word says how many requests there are; their records come as the loops below want them
        const unsigned hdr = (unsigned)(s_ready >> 32);
        const int n = min((int)(hdr & 0xffu), kMaxReq);
        if (warp == NW) {
            bool lost = s_abort != 0 || ((hdr >> 8) & 0xffu) != MELINOE_OK;
            for (int i = lane; i < 4 * n; i += 32) {
                const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(plan->fast) + i);
                reinterpret_cast<uint4 *>(s_req)[i] = v;
                lost = lost || (i % 4 == 0 && (v.x | v.y) == 0u);       // no pointer: cannot be read from here
            }
            lost = __any_sync(0xffffffffu, lost);
            __syncwarp();
            if (XT == 0 && lane == 0) {
                feed.begin(lost ? 0 : n * F, F, G);
                while (feed.left > 0 && feed.n < (uint32_t)S)
                    issue();
            }
        }
        if (tid == kThreads - 1) {
            s_hdr[0] = (int)((hdr >> 8) & 0xffu);
            s_hdr[1] = 1;
            s_hdr[2] = 0;
            s_hdr[3] = n;
            s_nact = n;
            s_deferred = (int)((hdr >> 16) & 1u);
        }
    } else if (tid == kThreads - 1) {
        const int n_groups = plan->n_groups;
        s_hdr[0] = plan->status;
        s_hdr[1] = n_groups;
        if (p.group < 0) {
            s_hdr[2] = 0;
            s_hdr[3] = plan->n_dreq;
        } else {
            s_hdr[2] = plan->group_vr_begin[p.group];
            s_hdr[3] = plan->group_vr_begin[p.group + 1];
        }
    }
    for (int i = tid; !fast && i < kMaxReq; i += kThreads) {
        tab.match[i] = 0u;
        tab.of_expert[i] = -1;
    }
    if (!fast && tid < kMaxReq) {
        const uint4 *src = reinterpret_cast<const uint4 *>(plan->dreq + tid);
        uint4 *dst = reinterpret_cast<uint4 *>(tab.raw + tid);
        dst[0] = src[0];
        dst[1] = src[1];
    }
    for (int i = tid; !fast && i < Tc * p.k; i += kThreads) {
        tab.idx[i] = p.idx[(size_t)tok0 * p.k + i];
        tab.gw[i] = p.gate[(size_t)tok0 * p.k + i];
    }
    if (XT == 0) {
        const int per_row = d / 8;                  // 16-byte pieces of a hidden row
        for (int i = tid; i < Tc * per_row; i += kThreads) {
            const int t = i / per_row, c = i % per_row;
            uint4 v = *reinterpret_cast<const uint4 *>(p.x + (size_t)(tok0 + t) * d + c * 8);
            if (FMT == 1)       // elements (0,4) (1,5) (2,6) (3,7): the pairing of the expanded weight registers
                v = make_uint4(__byte_perm(v.x, v.z, 0x5410), __byte_perm(v.x, v.z, 0x7632), __byte_perm(v.y, v.w, 0x5410),
                               __byte_perm(v.y, v.w, 0x7632));
            *reinterpret_cast<uint4 *>(xs + (size_t)t * XP + c * 16) = v;
        }
    }
    __syncthreads();
    const int status = s_abort == 1 ? (int)MELINOE_ERR_TIMEOUT : s_hdr[0], n_groups = s_hdr[1], rq0 = s_hdr[2];
    const int nrq = s_hdr[3] - rq0;
    if (status != MELINOE_OK || nrq < 0 || nrq > kMaxReq) {
        if (s_abort == 1 && tid == 0)
            atomicExch(p.err, MELINOE_ERR_TIMEOUT);
        // the call was refused on the device: the output is all zeros, the status tells why
        if (p.group <= 0)
            for (size_t i = (size_t)blockIdx.x * kThreads + tid; i < (size_t)Tc * d; i += (size_t)G * kThreads)
                p.out[(size_t)tok0 * d + i] = 0;
        // the counters advance once per CTA and launch, whatever happens
        if (tid < NW && atomicAdd(p.sync + tid * kSyncPitch, 1u) == (unsigned)(G - 1))
            p.sync[tid * kSyncPitch] = 0u;
        planner_ended();
        return;
    }
    if (XT) {
        // 128 columns of tensor memory: 16 warps x 32 columns of operand fragments (see below)
        if (warp == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(128));
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    if (!fast) {
        // gate of every (request, token): the token's gate for that expert if the router chose it
        for (int i = tid; i < nrq * kTokPerVr; i += kThreads) {
            const int r = i / kTokPerVr, t = i % kTokPerVr;
            const int e = tab.raw[rq0 + r].expert;
            if (t == 0 && e >= 0 && e < kMaxReq)
                tab.of_expert[e] = r;
            float gv = 0.0f;
            if (t < Tc) {
                if (e >= p.E) {
                    gv = 1.0f;              // shared expert: every token, gate 1
                    atomicOr(&tab.match[r], 1u << t);
                } else {
                    for (int j = 0; j < p.k; ++j)
                        if (tab.idx[t * p.k + j] == e) {
                            gv = tab.gw[t * p.k + j];
                            atomicOr(&tab.match[r], 1u << t);
                        }
                }
            }
            tab.gate[r][t] = gv;
        }
        __syncthreads();
        // The requests that have a token in this launch, in ascending expert id (shared experts last): the
        // rows are dealt out in that order, so the order of every sum depends only on which experts the
        // tokens use, not on which of them happened to be resident.
        if (warp == 0) {
            int base = 0;
            for (int e0 = 0; e0 < kMaxReq; e0 += 32) {
                const int e = e0 + lane;
                const int r = e < kMaxReq ? tab.of_expert[e] : -1;
                // a fetched expert that stays resident is streamed (and stored into its slot) by the launch whose
                // job that is even if none of this launch's tokens uses it
                bool act = r >= 0 && tab.match[r] != 0u;
                bool pull = false, stays = false, hazard = false;
                if (r >= 0 && p.group < 0 && (tab.raw[rq0 + r].flags & kDecMiss)) {
                    const int fl = tab.raw[rq0 + r].flags;
                    pull = true;
                    stays = (fl & kDecStays) != 0 && p.write_back != 0;
                    hazard = (fl & kDecHazard) != 0;
                    if (stays && (hazard ? p.chunk == p.n_chunks - 1 : p.chunk == 0))
                        act = true;
                }
                const unsigned m = __ballot_sync(0xffffffffu, act);
                if (act) {
                    const DecReq q = tab.raw[rq0 + r];
                    FastReq sr;
                    sr.src = q.blob;
                    sr.wb = sr.deferred = nullptr;
                    sr.expert = e;
#pragma unroll
                    for (int t = 0; t < kTokPerVr; ++t)
                        sr.gate[t] = tab.gate[r][t];
                    if (pull) {
                        // Where a call is made in several launches (more than 8 tokens): the first one stores
                        // the expert into its slot and the later ones read it there, unless the slot still
                        // holds an expert the call computes with: then every launch reads the host store and
                        // the last one stores it once all CTAs are done.
                        if (stays && !hazard && p.chunk > 0) {
                            sr.src = q.blob;
                        } else {
                            sr.src = q.host;
                            if (q.host == nullptr)
                                s_abort = 2;
                            if (stays && !hazard)
                                sr.wb = const_cast<char *>(q.blob);
                            if (stays && hazard && p.chunk == p.n_chunks - 1) {
                                sr.deferred = const_cast<char *>(q.blob);
                                s_deferred = 1;
                            }
                        }
                    }
                    s_req[base + __popc(m & ((1u << lane) - 1u))] = sr;
                }
                base += __popc(m);
            }
            if (lane == 0)
                s_nact = base;
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");      // the ring's first copies come over these tables
    } else if (tid < nrq && s_req[tid].src == nullptr) {
        s_abort = 2;
    }
    __syncthreads();
    const int nact = s_nact;
    const bool no_host = s_abort == 2;      // a missed expert cannot be read from here: nothing is computed
    if (trace && tid == 0)
        trace[1] = globaltimer_ns();

    // ---- this CTA's share of the rows: f rows of the active requests, request-major, dealt out evenly
    const int rows = no_host ? 0 : nact * F;
    const int q_lo = (int)((long long)blockIdx.x * rows / G), q_hi = (int)((long long)(blockIdx.x + 1) * rows / G);

    if (warp == NW) {
        // =================================================================== producer
        if (lane == 0) {
            if (XT != 0 || !fast)
                feed.begin(rows, F, G);
            while (feed.left > 0) {
                if (feed.n >= (uint32_t)S && !mbar_wait(empty0 + 8 * feed.st, feed.ph, abort_flag))
                    break;
                issue();
            }
            if (*abort_flag) {
                // a wait ran out: give the copies still in flight a bounded time to land before this
                // CTA's shared memory goes away
                const long long t0 = clock64();
                for (uint32_t j = feed.n > (uint32_t)S ? feed.n - S : 0; j < feed.n; ++j)
                    while (!mbar_try(full0 + 8 * (j % S), (j / S) & 1u) && clock64() - t0 < kWaitLimitCycles) {
                    }
            }
            planner_ended();
        }
    } else {
        // =================================================================== consumers
        const int g = lane >> 2, tig = lane & 3;
        if constexpr (FMT == 1) {
            consume_q4<MT_, NG, TG>(p, geo, s_req, s_sums, buf, ring_s, xs_s, full0, empty0, abort_flag, q_lo, q_hi, trace);
        } else {
            // groups of warps (see decode_groups): this warp's group and place in it, k-steps and m-tiles of a warp
            constexpr int NWG = NW / NG, kTiles = MT_ * NG;
            const int grp = NG == 1 ? 0 : warp / NWG, gw = NG == 1 ? warp : warp % NWG;
            buf += grp * (NWG * kBufPitch);
            float *sums = s_sums + grp * 128;
            float acc[kTiles][4];
#pragma unroll
            for (int i = 0; i < kTiles; ++i)
                acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
            const bool has_tok = g < Tc;
            const uint32_t xrow = xs_s + g * XP + tig * 4 + gw * kTiles * 32;     // this warp's columns of token g
            // XT: the token operand of this thread's 16 gate/up steps (two registers each) never changes, so it is
            // written once into the thread's own lane of tensor memory (warp w may use lanes 32 (w mod 4) ..,
            // the four warps of a lane quarter take 32 columns each) and fetched from there step by step.
            uint32_t xt = 0;
            if constexpr (XT == 1) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                xt = s_tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(warp >> 2) * 32;
                uint32_t r[32];
                const uint16_t *xr = p.x + (size_t)(tok0 + (has_tok ? g : 0)) * d + warp * (MT * 16) + 2 * tig;
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const bool on = has_tok && i < MT;
                    r[2 * i] = on ? __ldcg(reinterpret_cast<const uint32_t *>(xr + i * 16)) : 0u;
                    r[2 * i + 1] = on ? __ldcg(reinterpret_cast<const uint32_t *>(xr + i * 16 + 8)) : 0u;
                }
                tmem_st32(xt, r);
            }
            // ldmatrix lane roles.  gate/up: matrices (W_g rows, k low), (W_u rows, k low), (W_g rows, k high),
            // (W_u rows, k high); down: four consecutive 8-column pieces of the W_d^T rows
            const int r8 = lane & 7, sel_gu = (lane >> 3) & 1, kh = lane >> 4, mat = lane >> 3;
            const uint32_t src0 = (uint32_t)((2 * tig) * 4 + (g >> 1)), src1 = src0 + 4;
            uint32_t st = 0, ph = 0;                    // ring stage of the tile and the parity of its barrier phase
            int left = q_hi - q_lo, a = q_lo / F, f0 = q_lo % F;
            auto skip = [&] {
                const int m = min(min(TR, F - f0), left);
                if (++st == (uint32_t)S) {
                    st = 0;
                    ph ^= 1u;
                }
                left -= m;
                f0 += m;
                if (f0 == F) {
                    f0 = 0;
                    ++a;
                }
            };
#pragma unroll 1
            for (int i = 0; i < grp && left > 0; ++i)
                skip();
            while (left > 0) {
                const int m = min(min(TR, F - f0), left);
                const uint32_t stage = ring_s + st * STAGE;
                mbar_wait(full0 + 8 * st, ph, abort_flag);
                if (p.trace && tid == 0 && left == q_hi - q_lo)
                    p.trace[(size_t)blockIdx.x * 8 + 2] = globaltimer_ns();
                char *wb = s_req[a].wb;
                const bool store_tile = wb != nullptr && tid % (32 * NWG) == 0;
                if (store_tile)
                    bulk_s2g(wb + (size_t)f0 * RB, stage, (uint32_t)m * RB);
                const int rr = r8 < m ? r8 : 0;               // rows the tile does not have read row 0 (never used)
                const uint32_t swz = (uint32_t)((f0 + rr) & 7);
                const uint32_t rowbase = stage + rr * RB;
                // ---- gate/up: this warp's columns of the tile's rows.  A dependent mma.sync issues only every
                // ~110 cycles, so the k-steps go to four independent accumulators, and the fragment loads of
                // four steps are issued before their four products.
                // (Where a warp has 16 m-tiles of output accumulators, d_model above 2048, registers only allow
                // two steps at a time.)
                constexpr int GG = kTiles > 8 ? 2 : 4;
                float cg[GG][4];
#pragma unroll
                for (int i = 0; i < GG; ++i)
                    cg[i][0] = cg[i][1] = cg[i][2] = cg[i][3] = 0.f;
                {
                    const uint32_t arow = rowbase + sel_gu * 2 * d;
                    const uint32_t ch0 = (uint32_t)(2 * gw * kTiles + kh);
#pragma unroll
                    for (int i0 = 0; i0 < kTiles; i0 += GG) {
                        if (i0 < kTiles) {
                            uint32_t af[GG][4], bf[GG][2];
#pragma unroll
                            for (int j = 0; j < GG; ++j) {
                                const int i = i0 + j < kTiles ? i0 + j : i0;     // beyond the warp's last step: a valid address, product unused
                                ldmatrix_x4(arow + (((ch0 + 2 * i) ^ swz) << 4), af[j][0], af[j][1], af[j][2], af[j][3]);
                                if constexpr (XT == 0) {
                                    bf[j][0] = has_tok ? lds32(xrow + i * 32) : 0u;
                                    bf[j][1] = has_tok ? lds32(xrow + i * 32 + 16) : 0u;
                                }
                            }
                            if constexpr (XT == 1) {
                                static_assert(XT == 0 || GG == 2, "two steps per group");
                                tmem_ld4(xt + 2 * i0, bf[0][0], bf[0][1], bf[GG - 1][0], bf[GG - 1][1]);
                                tmem_wait_ld();
                            }
#pragma unroll
                            for (int j = 0; j < GG; ++j)
                                if (i0 + j < kTiles)
                                    mma_16816(cg[j], af[j][0], af[j][1], af[j][2], af[j][3], bf[j][0], bf[j][1]);
                        }
                    }
                }
                // ---- the warps' partial tiles meet: warp w sums 8 of the tile's 128 values over all warps (four
                // lanes per value, each adding four warps' parts in warp order, then a fixed tree), then every
                // warp reads the complete tile
#pragma unroll
                for (int i = 0; i < 4; ++i)
                    buf[gw * kBufPitch + i * 32 + lane] = GG == 4 ? (cg[0][i] + cg[1][i]) + (cg[2][i] + cg[3][i]) : cg[0][i] + cg[GG - 1][i];
                auto meet = [&] {
                    if (NG == 1)
                        asm volatile("bar.sync 1, %0;" ::"n"(NW * 32) : "memory");
                    else
                        asm volatile("bar.sync %0, %1;" ::"r"(1 + grp), "n"(NWG * 32) : "memory");
                };
                meet();
                {
                    constexpr int kOwn = 8 * NG;         // values of a warp
                    const int e = gw * kOwn + (lane & (kOwn - 1)), pg = lane / kOwn;
                    float v = buf[(pg * 4) * kBufPitch + e];
                    v += buf[(pg * 4 + 1) * kBufPitch + e];
                    v += buf[(pg * 4 + 2) * kBufPitch + e];
                    v += buf[(pg * 4 + 3) * kBufPitch + e];
                    if (NG == 1)
                        v += __shfl_xor_sync(0xffffffffu, v, 8);
                    if (NG <= 2)
                        v += __shfl_xor_sync(0xffffffffu, v, 16);
                    if (lane < kOwn)
                        sums[e] = v;
                }
                meet();
                const float s0 = sums[lane], s1 = sums[32 + lane], s2 = sums[64 + lane], s3 = sums[96 + lane];
                // rows g and g + 8 of the tile are g_f and u_f of f = f0 + g, columns are tokens 2 tig, 2 tig + 1
                const float gt0 = s_req[a].gate[2 * tig], gt1 = s_req[a].gate[2 * tig + 1];
                // (the fast division: the exact one takes its slow path for the zeros of unused token columns)
                float h0 = __fdividef(s0, 1.0f + __expf(-s0)) * s2 * gt0;
                float h1 = __fdividef(s1, 1.0f + __expf(-s1)) * s3 * gt1;
                if (g >= m || gt0 == 0.0f)
                    h0 = 0.f;
                if (g >= m || gt1 == 0.0f)
                    h1 = 0.f;
                const uint32_t hp = bf16_rne(h0) | (bf16_rne(h1) << 16);
                // B fragment of the down product: h[f = 2 tig', 2 tig' + 1][token g'] from the lanes that hold them
                const uint32_t v0 = __shfl_sync(0xffffffffu, hp, src0), v1 = __shfl_sync(0xffffffffu, hp, src1);
                const uint32_t bd = (g & 1) ? ((v0 >> 16) | (v1 & 0xffff0000u)) : ((v0 & 0xffffu) | (v1 << 16));
                // ---- down: the tile's rows are the K dimension (rows the tile does not have count as zero)
                {
                    const uint32_t km = (2 * tig < m ? 0x0000ffffu : 0u) | (2 * tig + 1 < m ? 0xffff0000u : 0u);
                    const uint32_t drow = rowbase + 4 * d;
                    const uint32_t cc0 = (uint32_t)(gw * kTiles * 2);
                    constexpr int DG = kTiles > 8 ? 2 : 4;      // loads (of two m-tiles each) per group
#pragma unroll
                    for (int m0 = 0; m0 < kTiles; m0 += 2 * DG) {
                        if (m0 < kTiles) {
                            // fragment loads of up to eight m-tiles first, then their products
                            uint32_t rf[DG][4];
#pragma unroll
                            for (int j = 0; j < DG; ++j) {
                                // a load covers two m-tiles; an odd last one is fetched together with the one before
                                // it (or, if it is the warp's only one, with 16 columns that are not used)
                                int mi = m0 + 2 * j;
                                if (mi >= kTiles)
                                    mi = m0;
                                else if (mi + 1 >= kTiles && mi > 0)
                                    mi -= 1;
                                ldmatrix_x4_trans(drow + (((cc0 + 2 * mi + mat) ^ swz) << 4), rf[j][0], rf[j][1], rf[j][2], rf[j][3]);
                            }
#pragma unroll
                            for (int j = 0; j < DG; ++j) {
                                const int mi = m0 + 2 * j;
                                if (mi + 1 < kTiles) {
                                    mma_16816(acc[mi], rf[j][0] & km, rf[j][1] & km, 0u, 0u, bd, 0u);
                                    mma_16816(acc[mi + 1], rf[j][2] & km, rf[j][3] & km, 0u, 0u, bd, 0u);
                                } else if (mi < kTiles) {
                                    if (mi > 0)
                                        mma_16816(acc[mi], rf[j][2] & km, rf[j][3] & km, 0u, 0u, bd, 0u);
                                    else
                                        mma_16816(acc[mi], rf[j][0] & km, rf[j][1] & km, 0u, 0u, bd, 0u);
                                }
                            }
                        }
                    }
                }
                if (store_tile)
                    bulk_wait_read();         // the slot store has read the stage
                __syncwarp();
                if (lane == 0)
                    mbar_arrive(empty0 + 8 * st);
                skip();
#pragma unroll
                for (int i = 1; i < NG; ++i)     // the other groups'
                    if (left > 0)
                        skip();
            }
            if (trace && tid == 0)
                trace[3] = globaltimer_ns();
            if constexpr (NG > 1) {
                // the groups' sums, in their order: a warp keeps those of its columns that are its group's
                asm volatile("bar.sync 8, %0;" ::"n"(NW * 32) : "memory");      // no tile is read any more: the ring is free
                auto at = [&](int of, int i) { return ring_s + (uint32_t)(((of * NWG + gw) * kTiles + i) * 512 + lane * 16); };
#pragma unroll
                for (int i = 0; i < kTiles; ++i)
                    asm volatile("st.shared.v4.f32 [%0], {%1,%2,%3,%4};" ::"r"(at(grp, i)), "f"(acc[i][0]), "f"(acc[i][1]), "f"(acc[i][2]), "f"(acc[i][3]) : "memory");
                asm volatile("bar.sync 8, %0;" ::"n"(NW * 32) : "memory");
#pragma unroll
                for (int i = 0; i < MT; ++i) {
                    acc[i][0] = acc[i][1] = acc[i][2] = acc[i][3] = 0.f;
#pragma unroll
                    for (int of = 0; of < NG; ++of) {
                        const uint4 v = lds128(at(of, grp * MT + i));
                        acc[i][0] += __uint_as_float(v.x);
                        acc[i][1] += __uint_as_float(v.y);
                        acc[i][2] += __uint_as_float(v.z);
                        acc[i][3] += __uint_as_float(v.w);
                    }
                }
            }
            // ---- this CTA's partial output, added into the call's accumulator as 64-bit fixed point (2^-40):
            // integer addition is exact, so the sum does not depend on the order in which the CTAs arrive.
            // (Adds without a return value: atomics that return the old word, which would let the last adder
            // of an element finish it on the spot, measured three times slower under this contention.)
            {
                unsigned long long *yacc = reinterpret_cast<unsigned long long *>(p.yacc);
                auto add = [&](int t, int c, float v) {
                    const long long fx = __float2ll_rn(v * 1099511627776.0f);    // exact scaling, then to the nearest 2^-40
                    red_add_u64(yacc + (size_t)t * d + c, (unsigned long long)fx);
                };
#pragma unroll
                for (int mi = 0; mi < kTiles; ++mi) {
                    if (mi < MT) {
                        const int c = ((gw * NG + grp) * MT + mi) * 16 + g;
                        if (2 * tig < Tc) {
                            add(2 * tig, c, acc[mi][0]);
                            add(2 * tig, c + 8, acc[mi][2]);
                        }
                        if (2 * tig + 1 < Tc) {
                            add(2 * tig + 1, c, acc[mi][1]);
                            add(2 * tig + 1, c + 8, acc[mi][3]);
                        }
                    }
                }
            }
        }
        // ---- count this warp out; the last CTA's warp turns the sums of its columns into the output
        // (groups: see decode_groups)
        const int col_warp = NG == 1 ? warp : warp % (NW / NG) * NG + warp / (NW / NG);
        __syncwarp();
        unsigned ticket = 0;
        if (lane == 0) {
            // (the warp barrier orders the other lanes' adds before lane 0's fence, which is cumulative)
            __threadfence();
            ticket = atomicAdd(p.sync + col_warp * kSyncPitch, 1u);
        }
        ticket = __shfl_sync(0xffffffffu, ticket, 0);
        if (trace && tid == 0)
            trace[4] = globaltimer_ns();
        if (ticket == (unsigned)(G - 1)) {
            if (lane == 0)
                p.sync[col_warp * kSyncPitch] = 0u;   // the counter is back at zero for the next launch
            __threadfence();
            if (trace)
                trace[5] = globaltimer_ns();
            const bool acc_in = p.group > 0, acc_out = p.group >= 0 && p.group < n_groups - 1;
            // The warp's columns: `own` contiguous ones, except that the 4-bit path's column steps of 32, where a warp has only
            // one of them, are 16 columns in each half of a block of 64.  All loads of some tokens before any store: this
            // warp is the whole grid's critical path, and a load behind a store that may alias it would wait for it.
            // For the same reason the forms differ by what there is to convert: four tokens' predicated instructions
            // for one token were 1.5 us per launch.
            const int own = MT * 16;
            const bool halves = FMT == 1 && MT == 2;
            // n elements per lane: element j is column column(j) of token token(j), if on(j)
            auto convert = [&](auto n, auto on, auto token, auto column) {
                constexpr int N = decltype(n)::value;
                long long fx[N];
                float carry[N];
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    fx[j] = on(j) ? __ldcg(p.yacc + token(j) * d + column(j)) : 0ll;
                    carry[j] = acc_in && on(j) ? __ldcg(p.ybuf + (size_t)(tok0 + token(j)) * d + column(j)) : 0.0f;
                }
#pragma unroll
                for (int j = 0; j < N; ++j) {
                    if (on(j)) {
                        p.yacc[token(j) * d + column(j)] = 0;    // the accumulator is left clean for the next launch
                        float v = __ll2float_rn(fx[j]) * (1.0f / 1099511627776.0f);     // one rounding, then an exact scaling
                        const size_t o = (size_t)(tok0 + token(j)) * d + column(j);
                        if (acc_in)
                            v += carry[j];
                        if (acc_out)
                            p.ybuf[o] = v;
                        else
                            p.out[o] = (uint16_t)bf16_rne(v);
                    }
                }
            };
            if constexpr ((MT_ == 2 && FMT == 0) || MT_ == 4 || MT_ == 8 || MT_ == 16) {
                constexpr int kSteps = MT_ / 2, kToks = 16 / kSteps;
                const int c0 = col_warp * own + lane;
                if (Tc == 1) {
                    convert(Count<kSteps>(), [](int) { return true; }, [](int) { return 0; }, [&](int j) { return c0 + j * 32; });
                } else if (kSteps <= 2 && Tc <= 4) {
                    // (narrow models: of sixteen elements most would be off; d 512, d_ff 512, 2 tokens of 2 experts, 4 layers
                    // 54.0 us with sixteen, 48.5 like this; d 1024 55.9 and 51.7)
                    convert(Count<4 * kSteps>(), [&](int j) { return j / kSteps < Tc; }, [](int j) { return j / kSteps; },
                            [&](int j) { return c0 + j % kSteps * 32; });
                } else {
#pragma unroll 1
                    for (int t0 = 0; t0 < Tc; t0 += kToks)
                        convert(Count<16>(), [&](int j) { return t0 + j / kSteps < Tc; }, [&](int j) { return t0 + j / kSteps; },
                                [&](int j) { return c0 + j % kSteps * 32; });
                }
            } else {
                // other widths: the warp's columns of all tokens end to end
                const int total = own * Tc;
                auto flat = [&](auto n, int e0) {
                    int tok[decltype(n)::value], col[decltype(n)::value];
#pragma unroll
                    for (int j = 0; j < decltype(n)::value; ++j) {
                        const int e = e0 + 32 * j;
                        tok[j] = e / own;
                        const int i = e - tok[j] * own;
                        col[j] = halves ? (col_warp >> 1) * 64 + 16 * (col_warp & 1) + (i & 15) + 32 * (i >> 4) : col_warp * own + i;
                    }
                    convert(n, [&](int j) { return e0 + 32 * j < total; }, [&](int j) { return tok[j]; }, [&](int j) { return col[j]; });
                };
                if (total <= 64) {
#pragma unroll 1
                    for (int e0 = lane; e0 < total; e0 += 32)
                        flat(Count<1>(), e0);
                } else {
#pragma unroll 1
                    for (int e0 = lane; e0 < total; e0 += 128)
                        flat(Count<4>(), e0);
                }
            }
            if (trace)
                trace[6] = globaltimer_ns();
        }
        if (tid % (NW / NG * 32) == 0)
            bulk_wait_all();              // the slot stores of this thread have completed
    }

    if (*abort_flag && lane == 0)
        atomicExch(p.err, no_host ? MELINOE_ERR_STATE : MELINOE_ERR_TIMEOUT);
    if (XT) {
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (warp == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(128));
    }
    if (trace && tid == 0)
        trace[7] = globaltimer_ns();
    if (!s_deferred)
        return;

    // ---- fetched experts whose slot was still being computed with: stored by the last CTA, once every CTA is done
    __syncthreads();
    if (tid == 0) {
        __threadfence();
        s_last = atomicAdd(p.sync + NW * kSyncPitch, 1u) == (unsigned)(G - 1);
        if (s_last)
            p.sync[NW * kSyncPitch] = 0u;
    }
    __syncthreads();
    if (s_last && tid == 0) {
        uint32_t phase = 0;
        bool any = false;
        for (int a = 0; a < nact && *abort_flag != 1; ++a) {
            char *slot = s_req[a].deferred;
            if (slot == nullptr)
                continue;
            const char *src = s_req[a].src;
            for (int f = 0; f < F; f += TR) {
                const uint32_t bytes = (uint32_t)min(TR, F - f) * RB;
                if (any)
                    bulk_wait_read();
                asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
                mbar_expect(hzbar, bytes);
                bulk_g2s(ring_s, src + (size_t)f * RB, bytes, hzbar);
                if (!mbar_wait(hzbar, phase & 1u, abort_flag))
                    break;
                ++phase;
                bulk_s2g(slot + (size_t)f * RB, ring_s, bytes);
                any = true;
            }
        }
        if (any)
            bulk_wait_all();
        if (*abort_flag == 1)
            atomicExch(p.err, MELINOE_ERR_TIMEOUT);
    }
}

}  // namespace

bool ffn_decode_supported(int d, int F) { return d % 256 == 0 && d >= 256 && d <= 4096 && F % kUnitRows == 0; }
// 4-bit slots: the warps split the columns in steps of 32 (one 16-byte piece of codes), 16 warps; a warp's
// steps are 1, 2, 4 or 8 (whole scale groups, or half of one shared by two warps).
bool ffn_decode_supported_q4(int d, int F)
{
    return ffn_decode_supported(d, F) && (d == 512 || d == 1024 || d == 2048 || d == 4096);
}

cudaError_t ffn_decode_configure(int n_sms, size_t max_smem, DecLaunchCfg *cfg)
{
    size_t stat = 0;
#define MELINOE_FN(...) reinterpret_cast<const void *>(ffn_decode_kernel<__VA_ARGS__>)
    // (In the order in which their code is loaded, behind the planner's.  Where it lies beside the planner's, with which it alternates, is
    // worth up to 4 % of a short call; of six orders, for one token of 16 layers of d_model 2048, this one gave 344 us with 4-bit slots and 419
    // with bf16 ones, the others 344 to 360 and 417 to 424.  Other widths come as they come: from build to build a short call of theirs
    // differs by up to 2 %.  Nothing but speed hangs on it.  Asking for all of them costs a process's first handle nothing that was to be
    // measured: 25 ms as with seven.)
    const void *fns[] = {MELINOE_FN(16, 0), MELINOE_FN(8, 0), MELINOE_FN(8, 1, 0, 2, 1), MELINOE_FN(16, 0, 1), MELINOE_FN(8, 1),
                         MELINOE_FN(16, 1, 0, 1, 1), MELINOE_FN(16, 1), MELINOE_FN(4, 1, 0, 2, 1), MELINOE_FN(4, 1, 0, 2),
                         MELINOE_FN(2, 1, 0, 2, 1), MELINOE_FN(2, 1, 0, 2), MELINOE_FN(1, 0), MELINOE_FN(1, 0, 0, 2), MELINOE_FN(2, 0),
                         MELINOE_FN(2, 0, 0, 2), MELINOE_FN(3, 0), MELINOE_FN(3, 0, 0, 2), MELINOE_FN(4, 0), MELINOE_FN(4, 0, 0, 2),
                         MELINOE_FN(5, 0), MELINOE_FN(6, 0), MELINOE_FN(7, 0), MELINOE_FN(9, 0), MELINOE_FN(10, 0), MELINOE_FN(11, 0),
                         MELINOE_FN(12, 0), MELINOE_FN(13, 0), MELINOE_FN(14, 0), MELINOE_FN(15, 0), MELINOE_FN(12, 0, 1),
                         MELINOE_FN(13, 0, 1), MELINOE_FN(14, 0, 1), MELINOE_FN(15, 0, 1)};
    // (shared memory of a kilobyte more than the others; rings of narrow models, which do not need it)
    const void *fns4[] = {MELINOE_FN(1, 0, 0, 4), MELINOE_FN(2, 0, 0, 4)};
#undef MELINOE_FN
    for (const void *fn : fns) {
        cudaFuncAttributes fa;
        const cudaError_t e = cudaFuncGetAttributes(&fa, fn);
        if (e != cudaSuccess)
            return e;
        if (fa.sharedSizeBytes > stat)
            stat = fa.sharedSizeBytes;
    }
    const size_t usable = (max_smem - stat - 1024) / 128 * 128;
    for (const void *fn : fns) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)usable);
        if (e != cudaSuccess)
            return e;
    }
    for (const void *fn : fns4) {
        const cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)usable - 1024);
        if (e != cudaSuccess)
            return e;
    }
    // One CTA per SM, but for the SM where the planner is still finishing its records when it announces the plan: a CTA
    // there would enter microseconds after the others and end as much later.  (The other SMs of the planner's cluster
    // are free by then, and one SM less does not slow the stream.)
    cfg->grid = n_sms > 1 ? n_sms - 1 : 1;
    cfg->max_smem = usable;
    cfg->pdl = pdl_enabled();
    return cudaSuccess;
}

cudaError_t ffn_decode_geometry(const DecLaunchCfg &cfg, int d, int F, int tokens, int fmt, int min_req, DecGeometry *geo)
{
    if (!(fmt == 0 ? ffn_decode_supported(d, F) : fmt == 1 && ffn_decode_supported_q4(d, F)) || tokens < 1 || tokens > kTokPerVr)
        return cudaErrorInvalidValue;
    geo->n_warps = NW;
    // bytes of one hidden unit; pitch of the staged hidden rows (the pad keeps the fragment loads of neighbouring
    // tokens in different banks: 4-byte loads in the bf16 path, 16-byte loads in the 4-bit path)
    geo->row_bytes = fmt == 0 ? 6 * d : (3 * (d / 2) + 3 * (d / 64) * 2 + 15) / 16 * 16;
    geo->x_pitch = fmt == 0 ? 2 * d + 16 : 2 * d + 64;
    geo->tokens = tokens;
    // staged hidden rows + the warps' partial tiles; the largest tile (at most 8 rows) of which two
    // stages fit beside them
    const size_t bufs = (size_t)(fmt == 0 ? 1 : 2) * NW * kBufPitch * sizeof(float), rows = (size_t)tokens * geo->x_pitch;
    auto tile = [&](size_t fixed) {
        int tr = 8;
        while (tr > 0 && cfg.max_smem < fixed + (size_t)2 * tr * geo->row_bytes)
            --tr;
        return tr;
    };
    // Wide models with several tokens: the hidden states would take up to a third of the shared memory and leave room for tiles of
    // four rows or less, at which the per-tile work of the warps, not HBM, sets the pace.  Where that makes tiles higher, their operand
    // fragments go to tensor memory instead (d_ff 4096, 2 experts out of 16 per token, 4 layers, us: d 3584, 8 tokens, 3 -> 5 rows 811 -> 675; d 3072,
    // 8 tokens, 4 -> 5 rows 596 -> 563; d 4096, 3 tokens, 3 -> 4 rows 355 -> 293 (2 layers of d_ff 6400); from 5 rows on it loses: d 2560, 8 tokens,
    // 5 -> 7 rows 491 -> 506), as far as that makes a CTA's share a tile less: the set-up takes about a microsecond (d 4096, 2 experts out of 8, 4 layers,
    // without and with: 4 tokens, d_ff 256, 3 rows of a CTA, 128 and 134, d_ff 1024, 14 rows, 202 and 195; 8 tokens 179 and 183, 272 and 259).
    const int with_rows = tile(bufs + rows), more_rows = tile(bufs), share = min_req * F / cfg.grid;
    geo->x_tmem = fmt == 0 && d >= 3072 && tokens > 1 && with_rows <= 4 && share * (more_rows - with_rows) >= with_rows * more_rows ? 1 : 0;
    const size_t fixed = bufs + (geo->x_tmem ? 0 : rows);
    const int tr = tile(fixed);
    if (tr == 0)
        return cudaErrorInvalidConfiguration;
    const size_t avail = cfg.max_smem - fixed;
    geo->tile_rows = tr;
    geo->stage_bytes = tr * geo->row_bytes;
    size_t n = avail / geo->stage_bytes;
    if (n > (size_t)kMaxStages)
        n = kMaxStages;
    geo->groups = decode_groups(d, tokens, fmt, min_req * F / cfg.grid);
    n -= n % geo->groups;            // a stage belongs to one group
    geo->n_stages = (int)n;
    geo->smem_bytes = n * geo->stage_bytes + fixed;
    return cudaSuccess;
}

cudaError_t launch_ffn_decode(cudaStream_t stream, const DecLaunchCfg &cfg, const DecGeometry &geo, const DecParams &p)
{
    // Programmatic stream serialisation: the CTAs may be scheduled, and set up their barriers, while the
    // kernel ahead in the stream is still running; the kernel waits for the plan word before it reads
    // anything that kernel writes.  No CTA waits for another, so nothing depends on co-residency.
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(cfg.grid);
    lc.blockDim = dim3(kThreads);
    lc.dynamicSmemBytes = geo.smem_bytes;
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    int na = 0;
    if (cfg.pdl) {
        attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
        attr[na].val.programmaticStreamSerializationAllowed = 1;
        ++na;
    }
    lc.attrs = attr;
    lc.numAttrs = na;
    const int mt = p.d / (16 * NW), ng = geo.groups;
    auto launch = [&](auto kernel) { return cudaLaunchKernelEx(&lc, kernel, p, geo); };
    cudaError_t e;
    if (p.fmt == 0) {
        // (loops over the width that the compiler knows, which hardly spill, 12 bytes at most: d 1536, d_ff 4096, 4 tokens of 4 experts,
        // 4 layers 382 -> 349 us)
        switch (mt) {
        case 1:
            e = ng == 4   ? launch(ffn_decode_kernel<1, 0, 0, 4>)
                : ng == 2 ? launch(ffn_decode_kernel<1, 0, 0, 2>)
                          : launch(ffn_decode_kernel<1, 0>);
            break;
        case 2:
            e = ng == 4   ? launch(ffn_decode_kernel<2, 0, 0, 4>)
                : ng == 2 ? launch(ffn_decode_kernel<2, 0, 0, 2>)
                          : launch(ffn_decode_kernel<2, 0>);
            break;
        case 3: e = ng == 2 ? launch(ffn_decode_kernel<3, 0, 0, 2>) : launch(ffn_decode_kernel<3, 0>); break;
        case 4: e = ng == 2 ? launch(ffn_decode_kernel<4, 0, 0, 2>) : launch(ffn_decode_kernel<4, 0>); break;
        case 5: e = launch(ffn_decode_kernel<5, 0>); break;
        case 6: e = launch(ffn_decode_kernel<6, 0>); break;
        case 7: e = launch(ffn_decode_kernel<7, 0>); break;
        case 8: e = launch(ffn_decode_kernel<8, 0>); break;
        case 9: e = launch(ffn_decode_kernel<9, 0>); break;
        case 10: e = launch(ffn_decode_kernel<10, 0>); break;
        case 11: e = launch(ffn_decode_kernel<11, 0>); break;
        case 12: e = geo.x_tmem ? launch(ffn_decode_kernel<12, 0, 1>) : launch(ffn_decode_kernel<12, 0>); break;
        case 13: e = geo.x_tmem ? launch(ffn_decode_kernel<13, 0, 1>) : launch(ffn_decode_kernel<13, 0>); break;
        case 14: e = geo.x_tmem ? launch(ffn_decode_kernel<14, 0, 1>) : launch(ffn_decode_kernel<14, 0>); break;
        case 15: e = geo.x_tmem ? launch(ffn_decode_kernel<15, 0, 1>) : launch(ffn_decode_kernel<15, 0>); break;
        case 16: e = geo.x_tmem ? launch(ffn_decode_kernel<16, 0, 1>) : launch(ffn_decode_kernel<16, 0>); break;
        default: e = cudaErrorInvalidValue; break;
        }
    } else if (mt == 16) {
        e = geo.tokens <= 4 ? launch(ffn_decode_kernel<16, 1, 0, 1, 1>) : launch(ffn_decode_kernel<16, 1>);
    } else if (mt == 8) {
        e = ng == 2 ? launch(ffn_decode_kernel<8, 1, 0, 2, 1>) : launch(ffn_decode_kernel<8, 1>);
    } else if (mt == 4) {
        e = geo.tokens <= 4 ? launch(ffn_decode_kernel<4, 1, 0, 2, 1>) : launch(ffn_decode_kernel<4, 1, 0, 2>);
    } else {
        e = geo.tokens <= 4 ? launch(ffn_decode_kernel<2, 1, 0, 2, 1>) : launch(ffn_decode_kernel<2, 1, 0, 2>);
    }
    count_launch();
    return e;
}

}  // namespace melinoe
