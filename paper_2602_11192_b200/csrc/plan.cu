// Planning kernel: slot lookup with LRU eviction, miss queue; token lists and the gather of activations.
//
// One block per call, behind the router.  What bounds it is the latency of a few dependent steps, so the steps are
// few and each is done by many threads; whatever needs the pairs themselves is left to the kernels around it: the
// router counts per block how often each expert was chosen, and the gather kernel places the pairs (of calls of few
// tokens this one does, beside its planning).  (One block
// counting and sorting the pairs itself took 100 us for 49152 of them, 11 us for 1024; now 17 and 8 us.)  What the kernels behind it need is
// announced by a word, which they wait for: what goes to host memory then delays nobody (2 us).  It makes
//   (a) from the router's counts, the experts' offsets in the sorted order of the (token, rank) pairs and the pairs
//       of each expert in the blocks before each block: where the gather kernel puts a block's pairs,
//   (b) the call's cache requests: one per distinct expert, experts resident at call entry
//       first (ascending id), then the missing ones (ascending id); a miss takes the lowest
//       empty slot, else the least recently stamped slot (Section 3.2: experts are fetched on
//       demand, "evicting cached experts as dictated by the cache policy"; the policy is LRU),
//   (c) compute groups: group 0 = resident experts (+ shared experts); the misses follow in
//       waves, a new wave starting whenever a miss would overwrite an expert of the current
//       wave, so every wave's transfers can be in flight while earlier groups compute,
//   (d) the miss queue, in page-locked host memory, from which the host issues the transfers, and
//   (e) the call's statistics (hard miss count of Appendix C.1).
#include "kernels.cuh"

namespace melinoe {

namespace {

constexpr int kPlanThreads = 1024;
constexpr int kPlanSegs = kPlanThreads / kMaxExperts;    // parts in which the router's blocks are summed
constexpr int kPlanKeep = 8;                             // counts a thread keeps between the two passes

__global__ void __launch_bounds__(kPlanThreads) plan_kernel(PlanParams p, PromptParams q)
{
    __shared__ int32_t s_counts[kMaxReq];
    __shared__ int32_t s_offsets[kMaxReq + 1];
    __shared__ int32_t s_seg[kPlanSegs][kMaxExperts];
    __shared__ DevCache s_cache;
    __shared__ int32_t s_group_of_expert[kMaxExperts];
    __shared__ int32_t s_req_of_expert[kMaxReq];
    __shared__ ReqRec s_req[kMaxReq];
    __shared__ HostMiss s_miss[kMaxExperts];
    __shared__ int32_t s_group_vr_begin[kMaxGroups + 1];
    __shared__ int32_t s_grp_first[kMaxGroups + 1];              // count policy: first miss of a wave
    __shared__ unsigned long long s_key[kMaxExperts];            // victim-order key of a slot
    __shared__ int32_t s_victim[kMaxExperts];                    // V: slots in victim order
    __shared__ int32_t s_miss_expert[kMaxExperts];               // expert of miss number i
    __shared__ int32_t s_entry_occ[kMaxExperts];                 // occupant of a slot at call entry
    __shared__ int32_t s_miss_flags[kMaxExperts];                // kDecStays / kDecHazard of miss number i
    __shared__ int32_t s_misc[8];  // 0 n_req(routed) 1 n_hits 2 n_miss 3 n_evict 4 n_groups 5 n_dreq 6 status 7 n_req_total

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n_pairs = p.T * p.k;
    const int E = p.E, C = p.C;

    // ---- load persistent cache state, clear tables.  The router, which may still be running (programmatic launch), lets
    // this kernel start only once everything ahead of it is complete.
    {
        const uint32_t *src = reinterpret_cast<const uint32_t *>(p.cache);
        uint32_t *dst = reinterpret_cast<uint32_t *>(&s_cache);
        for (int i = tid; i < (int)(sizeof(DevCache) / 4); i += kPlanThreads)
            dst[i] = __ldcg(src + i);
    }
    for (int i = tid; i < kMaxReq; i += kPlanThreads) {
        s_counts[i] = 0;
        s_req_of_expert[i] = -1;
    }
    if (tid < 8)
        s_misc[tid] = 0;
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // (token lists below: this thread's first pair, on its way meanwhile)
    const int q_first = tid - 32;
    int my_e = 0;
    if (q.lists && q_first >= 0 && q_first < n_pairs)
        my_e = __ldcg(p.idx + q_first);

    // ---- (a) the pairs of each expert: every thread sums one expert over a run of blocks, then the runs are put in order
    {
        const int e = tid & (kMaxExperts - 1), seg = tid / kMaxExperts;
        const int per = (p.n_blocks + kPlanSegs - 1) / kPlanSegs;
        const int b_lo = min(seg * per, p.n_blocks), n = min(b_lo + per, p.n_blocks) - b_lo;
        int32_t *col = p.block_counts + (size_t)b_lo * kMaxExperts + e;
        int keep[kPlanKeep], sum = 0;
#pragma unroll
        for (int i = 0; i < kPlanKeep; ++i)
            keep[i] = i < n ? __ldcg(col + (size_t)i * kMaxExperts) : 0;
#pragma unroll
        for (int i = 0; i < kPlanKeep; ++i)
            sum += keep[i];
#pragma unroll 8
        for (int i = kPlanKeep; i < n; ++i)
            sum += __ldcg(col + (size_t)i * kMaxExperts);
        s_seg[seg][e] = sum;
        __syncthreads();
        int run = 0, total = 0;
#pragma unroll
        for (int i = 0; i < kPlanSegs; ++i) {
            const int v = s_seg[i][e];
            run += i < seg ? v : 0;
            total += v;
        }
        if (seg == 0 && e < E)
            s_counts[e] = total;
#pragma unroll
        for (int i = 0; i < kPlanKeep; ++i) {
            if (i < n)
                col[(size_t)i * kMaxExperts] = run;
            run += keep[i];
        }
        for (int i0 = kPlanKeep; i0 < n; i0 += kPlanKeep) {
#pragma unroll
            for (int i = 0; i < kPlanKeep; ++i)
                keep[i] = i0 + i < n ? col[(size_t)(i0 + i) * kMaxExperts] : 0;
#pragma unroll
            for (int i = 0; i < kPlanKeep; ++i) {
                if (i0 + i < n)
                    col[(size_t)(i0 + i) * kMaxExperts] = run;
                run += keep[i];
            }
        }
    }
    __syncthreads();
    // count policy (Definition C.1): one time step per call, count <- gamma * count + request
    if (p.policy == MELINOE_POLICY_COUNT && tid < E)
        s_cache.count[tid] = __fadd_rn(__fmul_rn(p.gamma, s_cache.count[tid]), s_counts[tid] > 0 ? 1.0f : 0.0f);
    if (warp == 0) {
        // offsets: a scan over the experts, then the shared experts' blocks of T
        const int c0 = lane < E ? s_counts[lane] : 0, c1 = lane + 32 < E ? s_counts[lane + 32] : 0;
        int i0 = c0, i1 = c1;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int a = __shfl_up_sync(0xffffffffu, i0, o), b = __shfl_up_sync(0xffffffffu, i1, o);
            i0 += lane >= o ? a : 0;
            i1 += lane >= o ? b : 0;
        }
        i1 += __shfl_sync(0xffffffffu, i0, 31);
        if (lane < E)
            s_offsets[lane] = i0 - c0;
        if (lane + 32 < E)
            s_offsets[lane + 32] = i1 - c1;
        __syncwarp();
        if (lane <= p.n_shared) {
            s_offsets[E + lane] = n_pairs + lane * p.T;
            if (lane < p.n_shared)
                s_counts[E + lane] = p.T;
        }
    }
    __syncthreads();

    // ---- (b), (c): cache requests, by warp 0; lane owns experts lane and lane + 32 and slots lane and
    // lane + 32.  The sequential rules (hits in ascending id, then misses in ascending id, a miss
    // takes the lowest empty slot, else the least recently stamped one; a new wave starts when a
    // miss would overwrite an expert of the current wave) have a closed form:
    //   - hit number r (ascending id) stamps its slot with counter + r + 1;
    //   - let V be the slots ordered by (empty first, by index), then by stamp after the hits were
    //     stamped; miss number i (ascending id) takes V[i mod C], because every slot it could prefer
    //     has either been taken by an earlier miss (and stamped newer) or comes later in V;
    //   - the expert it displaces is V[i]'s occupant at call entry for i < C, and miss i - C otherwise;
    //   - miss i belongs to wave 1 + i / C; it must wait for group i / C (i >= C), for group 0 if it
    //     displaces one of the call's hits, for nothing otherwise.
    if (warp == 0) {
        const int e0 = lane, e1 = lane + 32;
        const int c0 = e0 < E ? s_counts[e0] : 0, c1 = e1 < E ? s_counts[e1] : 0;
        const int soe0 = e0 < E ? s_cache.slot_of_expert[e0] : -1, soe1 = e1 < E ? s_cache.slot_of_expert[e1] : -1;
        const int eos0 = lane < C ? s_cache.expert_of_slot[lane] : -1, eos1 = lane + 32 < C ? s_cache.expert_of_slot[lane + 32] : -1;
        const uint64_t st0 = lane < C ? s_cache.stamp[lane] : 0ull, st1 = lane + 32 < C ? s_cache.stamp[lane + 32] : 0ull;
        uint64_t counter = s_cache.counter;
        auto ballot64 = [](bool lo, bool hi) {
            return (uint64_t)__ballot_sync(0xffffffffu, lo) | ((uint64_t)__ballot_sync(0xffffffffu, hi) << 32);
        };
        auto rank_below = [](uint64_t mask, int bit) { return __popcll(mask & ((1ull << bit) - 1ull)); };
        const uint64_t need = ballot64(c0 > 0, c1 > 0);
        const uint64_t resident = ballot64(soe0 >= 0, soe1 >= 0);
        const uint64_t hit_mask = need & resident, miss_mask = need & ~resident;
        const int n_hits = __popcll(hit_mask), n_miss = __popcll(miss_mask), n_req = n_hits + n_miss;
        __syncwarp();
        s_key[lane] = lane < C ? (eos0 < 0 ? (uint64_t)lane : ((1ull << 63) | st0)) : ~0ull;
        s_key[lane + 32] = lane + 32 < C ? (eos1 < 0 ? (uint64_t)(lane + 32) : ((1ull << 63) | st1)) : ~0ull;
        s_entry_occ[lane] = eos0;
        s_entry_occ[lane + 32] = eos1;
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = h ? e1 : e0, soe = h ? soe1 : soe0;
            if ((hit_mask >> e) & 1ull) {
                const int r = rank_below(hit_mask, e);
                const uint64_t st = counter + (uint64_t)r + 1ull;
                s_key[soe] = (1ull << 63) | st;
                s_cache.stamp[soe] = st;
                s_req[r] = ReqRec{e, soe, 1, -1, 0, 0, s_offsets[e], s_counts[e]};
                s_req_of_expert[e] = r;
                s_group_of_expert[e] = 0;
            }
            if ((miss_mask >> e) & 1ull)
                s_miss_expert[rank_below(miss_mask, e)] = e;
        }
        __syncwarp();
        // V: rank of each slot among the keys (keys are distinct); only misses under LRU take victims from it
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int sl = lane + 32 * h;
            if (sl < C && n_miss > 0 && p.policy != MELINOE_POLICY_COUNT) {
                const uint64_t mine = s_key[sl];
                int r = 0;
#pragma unroll 8
                for (int s2 = 0; s2 < C; ++s2)
                    r += s_key[s2] < mine;
                s_victim[r] = sl;
            }
        }
        __syncwarp();
        bool ev_flag[2] = {false, false};
        int n_groups = n_miss ? 1 + (n_miss + C - 1) / C : 1;
        int n_evict_seq = 0;
        if (p.policy == MELINOE_POLICY_COUNT) {
            // The count policy has no closed form (a victim depends on the counts of what the
            // earlier misses of the call brought in): one search per miss, in ascending expert id.
            // Victim: lowest empty slot, else the smallest (count of the occupant, stamp).
            int cur_group = 1, i = 0;
            if (lane == 0)
                s_grp_first[1] = 0;
            for (uint64_t m = miss_mask; m; m &= m - 1, ++i) {
                const int e = __ffsll((long long)m) - 1;
                uint64_t khi = ~0ull, klo = ~0ull;
                int slot = -1;
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    const int sl = lane + 32 * h;
                    if (sl < C) {
                        const int occ = s_cache.expert_of_slot[sl];
                        const uint64_t hi = occ < 0 ? 0ull : ((1ull << 32) | (uint64_t)__float_as_uint(s_cache.count[occ]));
                        const uint64_t lo = occ < 0 ? (uint64_t)sl : s_cache.stamp[sl];
                        if (hi < khi || (hi == khi && lo < klo)) {
                            khi = hi;
                            klo = lo;
                            slot = sl;
                        }
                    }
                }
#pragma unroll
                for (int mm = 16; mm >= 1; mm >>= 1) {
                    const uint64_t ohi = __shfl_xor_sync(0xffffffffu, khi, mm);
                    const uint64_t olo = __shfl_xor_sync(0xffffffffu, klo, mm);
                    const int os = __shfl_xor_sync(0xffffffffu, slot, mm);
                    if (ohi < khi || (ohi == khi && olo < klo)) {
                        khi = ohi;
                        klo = olo;
                        slot = os;
                    }
                }
                const int ev = s_cache.expert_of_slot[slot];
                int dep = -1;
                if (ev >= 0) {
                    ++n_evict_seq;
                    if ((need >> ev) & 1ull)
                        dep = s_group_of_expert[ev];
                }
                if (dep == cur_group) {
                    ++cur_group;      // it would overwrite an expert of the current wave: next wave
                    if (lane == 0)
                        s_grp_first[cur_group] = i;
                }
                __syncwarp();
                if (lane == 0) {
                    if (ev >= 0)
                        s_cache.slot_of_expert[ev] = -1;
                    s_cache.expert_of_slot[slot] = e;
                    s_cache.slot_of_expert[e] = slot;
                    s_cache.stamp[slot] = counter + (uint64_t)(n_hits + i) + 1ull;
                    s_req[n_hits + i] = ReqRec{e, slot, 0, ev, 0, cur_group, s_offsets[e], s_counts[e]};
                    s_req_of_expert[e] = n_hits + i;
                    s_group_of_expert[e] = cur_group;
                    s_miss[i] = HostMiss{e, slot, (int16_t)cur_group, (int16_t)dep, 0u};
                }
                __syncwarp();
            }
            n_groups = n_miss ? cur_group + 1 : 1;
            // a miss stays if it still occupies its slot when the call ends; storing it there has to
            // wait for the call's compute if the slot held one of the call's hits at entry
            for (int j = lane; j < n_miss; j += 32) {
                const int e = s_miss[j].expert, slot = s_miss[j].slot, occ = s_entry_occ[slot];
                const bool stays = s_cache.expert_of_slot[slot] == e;
                const bool hazard = stays && occ >= 0 && ((need >> occ) & 1ull);
                s_miss_flags[j] = (stays ? kDecStays : 0) | (hazard ? kDecHazard : 0);
            }
        } else
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = h ? e1 : e0;
            if ((miss_mask >> e) & 1ull) {
                const int i = rank_below(miss_mask, e);
                const int slot = s_victim[i % C];
                const int ev = i < C ? s_entry_occ[slot] : s_miss_expert[i - C];
                const int group = 1 + i / C;
                int dep = -1;
                if (i >= C)
                    dep = i / C;
                else if (ev >= 0 && ((need >> ev) & 1ull))
                    dep = 0;
                ev_flag[h] = ev >= 0;
                s_req[n_hits + i] = ReqRec{e, slot, 0, ev, 0, group, s_offsets[e], s_counts[e]};
                s_req_of_expert[e] = n_hits + i;
                s_miss[i] = HostMiss{e, slot, (int16_t)group, (int16_t)dep, 0u};
                // cache update: the last miss that lands in a slot keeps it
                const bool stays = i + C >= n_miss;
                {
                    const int occ = s_entry_occ[slot];
                    const bool hazard = stays && occ >= 0 && ((need >> occ) & 1ull);
                    s_miss_flags[i] = (stays ? kDecStays : 0) | (hazard ? kDecHazard : 0);
                }
                s_cache.slot_of_expert[e] = stays ? slot : -1;
                if (stays) {
                    s_cache.expert_of_slot[slot] = e;
                    s_cache.stamp[slot] = counter + (uint64_t)(n_hits + i) + 1ull;
                }
                if (i < C && ev >= 0)
                    s_cache.slot_of_expert[ev] = -1;
            }
        }
        const int n_evict = p.policy == MELINOE_POLICY_COUNT ? n_evict_seq : __popcll(ballot64(ev_flag[0], ev_flag[1]));
        counter += (uint64_t)n_req;
        __syncwarp();
        // shared experts: always resident, group 0.  Records for the compute kernels, grouped: the hits, the shared
        // experts, then the misses wave by wave.
        const int n_req_total = n_req + p.n_shared, ndr = n_req_total;
        if (lane < p.n_shared) {
            s_req[n_req + lane] = ReqRec{E + lane, -1, 1, -1, 0, 0, s_offsets[E + lane], p.T};
            s_req_of_expert[E + lane] = n_req + lane;
        }
        __syncwarp();
        for (int r = lane; r < n_req_total; r += 32)
            s_req[r].vr_start = r < n_hits ? r : r < n_req ? r + p.n_shared : r - n_miss;
        int status = s_misc[6];
        if (n_groups > (int)p.gmax)
            status = MELINOE_ERR_STATE;
        const bool ok = status == MELINOE_OK;      // otherwise nothing is left for the compute kernels to do
        for (int g = lane; g <= kMaxGroups; g += 32) {
            int b = 0;
            if (ok && g >= 1) {
                // misses served before wave g: (g - 1) * C under LRU, the wave's recorded first miss otherwise
                const int done = p.policy == MELINOE_POLICY_COUNT ? (g < n_groups ? s_grp_first[g] : n_miss) : (g - 1) * C;
                b = n_hits + p.n_shared + (done < n_miss ? done : n_miss);
            }
            s_group_vr_begin[g] = b;
        }
        if (lane == 0) {
            s_cache.counter = counter;
            s_cache.tot_hits += (uint64_t)n_hits;
            s_cache.tot_misses += (uint64_t)n_miss;
            s_cache.tot_evictions += (uint64_t)n_evict;
            s_cache.call_no += 1;
            s_misc[0] = n_req;
            s_misc[1] = n_hits;
            s_misc[2] = n_miss;
            s_misc[3] = n_evict;
            s_misc[4] = n_groups;
            s_misc[5] = ok ? ndr : 0;
            s_misc[6] = status;
            s_misc[7] = n_req_total;
        }
    } else if (q.lists) {
        // beside it: every pair's place among its expert's, in the blocks of one token each
        for (int j = q_first; j < n_pairs; j += kPlanThreads - 32) {
            const int t = j / p.k, e = j == q_first ? my_e : __ldcg(p.idx + j);
            const int pos = s_offsets[e] + __ldcg(p.block_counts + (size_t)t * kMaxExperts + e);
            p.perm[pos] = j;
            p.inv_pos[j] = pos;
            p.tok_of_sorted[pos] = t;
        }
        for (int i = q_first; i < p.n_shared * p.T; i += kPlanThreads - 32)
            p.tok_of_sorted[n_pairs + i] = i % p.T;
    }
    __syncthreads();

    // ---- write the plan for the grouped GEMM and announce it (see DevPlan::ready): the kernels behind this one wait for the word and not
    // for this grid to drain, which takes 2 us for what is written to host memory below
    const int n_req_total = s_misc[7];
    const bool ok = s_misc[6] == MELINOE_OK;
    DevPlan *plan = p.plan;
    if (tid == 0) {
        plan->n_tokens = p.T;
        plan->n_req = s_misc[0];
        plan->n_hits = s_misc[1];
        plan->n_miss = s_misc[2];
        plan->n_evict = s_misc[3];
        plan->n_groups = s_misc[4];
        plan->n_dreq = s_misc[5];
        plan->status = s_misc[6];
    }
    for (int i = tid; i <= kMaxGroups; i += kPlanThreads)
        plan->group_vr_begin[i] = s_group_vr_begin[i];
    if (q.counters)
        for (int i = tid; i < (int)(sizeof(GemmCounters) / 4); i += kPlanThreads)
            reinterpret_cast<int32_t *>(q.counters)[i] = 0;
    for (int i = tid; i < kMaxReq; i += kPlanThreads) {
        plan->counts[i] = s_counts[i];
        plan->req_of_expert[i] = s_req_of_expert[i];
    }
    for (int i = tid; i <= kMaxReq; i += kPlanThreads)
        plan->offsets[i] = i <= E + p.n_shared ? s_offsets[i] : 0;
    for (int i = tid; i < n_req_total; i += kPlanThreads)
        plan->req[i] = s_req[i];
    __syncthreads();
    if (tid == 0)
        asm volatile("st.release.gpu.global.u64 [%0], %1;"
                     ::"l"(&plan->ready), "l"(ready_word(p.call_seq, n_req_total, s_misc[6], false)) : "memory");

    // ---- (d) miss queue for the host, (e) statistics
    if (tid < s_misc[2]) {
        s_miss[tid].seq = p.call_seq;
        store16_host(&p.hplan->miss[tid], &s_miss[tid]);
    }
    if (tid == kPlanThreads - 32) {
        const int n_miss = s_misc[2];
        const HostPlanHeader hdr{n_miss, s_misc[4], s_misc[6], p.call_seq};
        store16_host(&p.hplan->hdr, &hdr);
        if (p.stats) {
            melinoe_moe_stats st;
            st.status = s_misc[6];
            st.n_tokens = p.T;
            st.n_distinct = s_misc[0];
            st.hits = s_misc[1];
            st.misses = n_miss;
            st.evictions = s_misc[3];
            st.groups = s_misc[4];
            st.reserved = 0;
            st.bytes_h2d = (uint64_t)n_miss * (uint64_t)p.expert_bytes;
            st.call_no = s_cache.call_no;
            *p.stats = st;
        }
    }

    // ---- the decode kernel's records (of calls that the grouped GEMM does not take; it waits for this grid's end) and the cache state
    if (ok) {
        const int n_hits = s_misc[1];
        for (int r = tid; r < n_req_total; r += kPlanThreads) {
            const ReqRec rec = s_req[r];
            DecReq q;
            q.blob = rec.slot >= 0 ? p.slots + (size_t)rec.slot * p.slot_stride : p.shared_blobs[rec.expert - E];
            q.host = nullptr;
            q.expert = rec.expert;
            q.flags = 0;
            q.group = rec.group;
            q.reserved = 0;
            if (!rec.hit) {
                q.host = p.host_blobs ? p.host_blobs[rec.expert] : nullptr;
                q.flags = kDecMiss | s_miss_flags[r - n_hits];
            }
            plan->dreq[rec.vr_start] = q;
        }
    }
    {
        uint32_t *dst = reinterpret_cast<uint32_t *>(p.cache);
        const uint32_t *src = reinterpret_cast<const uint32_t *>(&s_cache);
        for (int i = tid; i < (int)(sizeof(DevCache) / 4); i += kPlanThreads)
            dst[i] = src[i];
    }

    // the call's request-trace record, if one is being kept
    if (p.trace_rec) {
        const TraceLayout tl = trace_layout(E, p.k, p.trace_max_tokens);
        melinoe_moe_request *rq = reinterpret_cast<melinoe_moe_request *>(p.trace_rec + tl.req_off);
        for (int i = tid; i < s_misc[0]; i += kPlanThreads)
            rq[i] = melinoe_moe_request{s_req[i].expert, s_req[i].slot, s_req[i].hit, s_req[i].evicted};
        const int nt = p.T < p.trace_max_tokens ? p.T : p.trace_max_tokens;
        for (int i = tid; i < nt * p.k; i += kPlanThreads) {
            reinterpret_cast<int32_t *>(p.trace_rec + tl.idx_off)[i] = p.idx[i];
            reinterpret_cast<float *>(p.trace_rec + tl.gate_off)[i] = p.gate ? p.gate[i] : 0.0f;
        }
        if (tid == 0) {
            melinoe_moe_trace_header th;
            th.call_no = s_cache.call_no;
            th.n_tokens = p.T;
            th.n_requests = s_misc[0];
            th.hits = s_misc[1];
            th.misses = s_misc[2];
            th.status = s_misc[6];
            th.reserved = 0;
            *reinterpret_cast<melinoe_moe_trace_header *>(p.trace_rec) = th;
        }
    }
}

// Token lists and Xs[pos] = hidden[token of pos].  A block takes the tokens that one block of the router took: a pair's
// position is its expert's offset, plus the pairs of that expert in the blocks before (both from the planning kernel),
// plus those before it in this block.  A token's row is read once and written k times (and once per shared
// expert).  early: the GEMM may come while this one waits for the plan.  4-bit slots want that, as their codes are fetched and expanded
// meanwhile (60 tokens, d 4096, d_ff 6400, 8 experts, 2 per token: 192 us a pass, 190 early), but not where its CTAs would take the SMs that a
// block per token or more is still working on (d 2048, d_ff 1024, 64 experts, 8 per token, 400 tokens: 209 early, 206); bf16 slots
// lose by it always (80 tokens 145.6 and 144.9, 800 tokens 183.9 and 183.2; d 512, d_ff 2048, 800 tokens 56.9 and 56.3).  PERMUTE: elements (0,4) (1,5) (2,6) (3,7) of every eight, the order in which 4-bit codes expand.
constexpr int kGatherMaxPairs = 512;       // pairs of one router block at most (see router_shape)

template <bool PERMUTE>
__global__ void __launch_bounds__(256) gather_rows_kernel(PlanParams p, PromptParams q, const uint16_t *__restrict__ x, uint16_t *__restrict__ xs, int d,
                                                          int early)
{
    __shared__ int32_t s_run[kMaxExperts];
    __shared__ int32_t s_pos[kGatherMaxPairs];
    __shared__ int s_ok;
    const int tid = threadIdx.x, lane = tid & 31;
    const int t0 = blockIdx.x * q.tokens_per_block, n = min(q.tokens_per_block, p.T - t0);
    const int k = p.k, n_pairs = p.T * k;
    if (early)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // The planning kernel, which may still be running, has waited for the router and all before it.
    if (tid == 0) {
        uint32_t hdr;
        bool known = wait_for_ready(p.plan, p.call_seq, &hdr);
        if (!known) {
            // The wait ran out: the planner may have been held up, but behind its end the word stands.  If it does not even
            // then, the call has failed, and says so: the kernels behind must not pass for good what the last call's lists give.
            asm volatile("griddepcontrol.wait;" ::: "memory");
            known = plan_announced(p.plan, p.call_seq, &hdr);
            if (!known)
                atomicExch(q.err, MELINOE_ERR_TIMEOUT);
        }
        s_ok = known && plan_accepted(hdr);
    }
    __syncthreads();
    if (!early)
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    // (what comes behind this grid is behind the planning kernel's, too)
    auto leave = [] { asm volatile("griddepcontrol.wait;" ::: "memory"); };
    if (!s_ok)
        return leave();
    if (tid < 32) {          // (every part of a block's copies works the positions out, the first part writes them down)
        const bool first = blockIdx.y == 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int e = lane + 32 * h;
            s_run[e] = e < p.E ? __ldcg(&p.plan->offsets[e]) + __ldcg(p.block_counts + (size_t)blockIdx.x * kMaxExperts + e) : 0;
        }
        __syncwarp();
        for (int i0 = 0; i0 < n * k; i0 += 32) {
            const int i = i0 + lane, j = t0 * k + i;
            const int e = i < n * k ? __ldcg(p.idx + j) : -1 - lane;
            const unsigned same = __match_any_sync(0xffffffffu, e);
            const int r = __popc(same & ((1u << lane) - 1u));
            int pos = 0;
            if (e >= 0) {
                pos = s_run[e] + r;
                s_pos[i] = pos;
                if (first) {
                    if (q.row_gate)
                        q.row_gate[pos] = __ldcg(p.gate + j);
                    p.perm[pos] = j;
                    p.inv_pos[j] = pos;
                    p.tok_of_sorted[pos] = t0 + i / k;
                }
            }
            __syncwarp();
            if (e >= 0 && r == 0)
                s_run[e] = pos + __popc(same);
            __syncwarp();
        }
    }
    for (int i = tid; blockIdx.y == 0 && i < n * p.n_shared; i += 256) {
        const int pos = n_pairs + i / n * p.T + t0 + i % n;
        p.tok_of_sorted[pos] = t0 + i % n;
        if (q.row_gate)
            q.row_gate[pos] = 1.0f;
    }
    if (xs != nullptr) {
        __syncthreads();
        const int row16 = d / 8;                  // 16-byte pieces of a row
#pragma unroll 2
        for (int i = blockIdx.y * 256 + tid; i < n * row16; i += 256 * gridDim.y) {
            const int t = i / row16, c = i % row16;
            uint4 v = __ldg(reinterpret_cast<const uint4 *>(x + (size_t)(t0 + t) * d) + c);
            if (PERMUTE)
                v = make_uint4(__byte_perm(v.x, v.z, 0x5410), __byte_perm(v.x, v.z, 0x7632), __byte_perm(v.y, v.w, 0x5410),
                               __byte_perm(v.y, v.w, 0x7632));
            uint4 *dst = reinterpret_cast<uint4 *>(xs) + c;
            for (int j = 0; j < k; ++j)
                dst[(size_t)s_pos[t * k + j] * row16] = v;
            for (int j = 0; j < p.n_shared; ++j)
                dst[((size_t)n_pairs + (size_t)j * p.T + t0 + t) * row16] = v;
        }
    }
    leave();
}

}  // namespace

cudaError_t launch_gather_rows(cudaStream_t stream, int n_sms, const PlanParams &p, const PromptParams &q, const uint16_t *x, uint16_t *xs, int d,
                               bool permute)
{
    if (q.tokens_per_block * p.k > kGatherMaxPairs)
        return cudaErrorInvalidValue;
    // four blocks per SM, no more than one per 256 pieces to copy
    const int pieces = (q.tokens_per_block * (d / 8) + 255) / 256, want = (4 * n_sms + p.n_blocks - 1) / p.n_blocks;
    const int parts = xs == nullptr || want < 1 ? 1 : want < pieces ? want : pieces;
    const int early = permute && p.n_blocks * parts <= n_sms ? 1 : 0;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(p.n_blocks, parts);
    lc.blockDim = dim3(256);
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = pdl_enabled() ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&lc, permute ? gather_rows_kernel<true> : gather_rows_kernel<false>, p, q, x, xs, d, early);
    count_launch();
    return e;
}

cudaError_t launch_plan(cudaStream_t stream, const PlanParams &p, const PromptParams &q)
{
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(1);
    lc.blockDim = dim3(kPlanThreads);
    lc.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = attr;
    lc.numAttrs = pdl_enabled() ? 1 : 0;
    const cudaError_t e = cudaLaunchKernelEx(&lc, plan_kernel, p, q);
    count_launch();
    return e;
}

}  // namespace melinoe
