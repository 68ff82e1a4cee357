// One-launch event kernel for prefill-sized pools (bf16, d = 128, per-head signatures, 256 < N <= 5120, budgets up to 128):
// two CTAs per SM, so that one event's selection, which is latency, overlaps another one's stream of K.
// (event_stream_kernel, one CTA per SM, keeps larger N and larger budgets.) One CTA of nine warps per event.
//
//   1. K streams through a ring of four 64-row stages (cp.async.bulk + full/empty mbarriers, one producer warp, eight
//      scoring warps); every row is scored as it lands and only its score stays on chip.
//   2. Every thread takes a run of consecutive slots' keys into registers; s_(b) by bisection (four-way, counts packed in one
//      word per warp), lists in slot order by one block-wide scan.
//   3. lambda > 0: the best rows of the pool of possible arg-maxima, at most 192 (the active set), as an operand tile;
//      their raw cosines by two tcgen05 products into 256 columns of tensor memory, the lower triangle to shared memory,
//      Algorithm 1 in one warp over it. No candidate left out has a value above `bound`, so the loop is exact while its
//      winning values stay above that. Where one does not (4096 random rows to 128 at lambda = 0.5: about one event in a
//      hundred), the picks made stand and the next active set is formed: Eq. 2's values only fall, so a row's value
//      when it was last known, or its score, is an upper bound, and the rows with the best of those make up the set; their
//      running maxima come from one more product, against the rows picked. A round may make no pick (all of its rows have
//      fallen below one left out), but it leaves their values known: 4096 scores close together take about 40 rounds for 128
//      picks. Where infinite value rows make picks impossible, the event is done over the whole pool with plain dot products.
//   4. Kept K and V rows are staged on chip and written to slots 0..b-1 of the same buffers.
//
// FUSED: score + select + compact; otherwise selection only (scores are read from a.scores and nothing is rewritten).
// SPLIT: the scoring of an event is shared by a cluster of so many CTAs, for calls of few and long events (akv_split_rule.cuh says
// which). Each streams its part of K; the others store their scores to the first one's shared memory and leave, the first one selects.
#pragma once
#include "akv_event_stream.cuh"
#include "akv_split_rule.cuh"

namespace akv {

constexpr int kPfStages = 4;
constexpr unsigned kPfRing = kPfStages * kStStageBytes;
constexpr int kPfActive = 192;              // rows of the active set: 2 x 192 - 128 columns of tensor memory for its products
constexpr int kPfEnough = 184;              // rows that an active set is content with
constexpr int kPfLeast = 160;               // the same once the search has gone on for fourteen bits
constexpr uint32_t kPfCols = 256;
constexpr int kPfKeys = 21;                 // most keys per thread (an odd run per thread: no bank conflicts)
constexpr int kPfMaxN = 5120;
constexpr int kPfMaxBudget = 128;
constexpr int kPfRanked = kStWork;          // most rows that top-k ranks (one per thread)

struct PfSmem {
    unsigned region, spos, s, act, ar, am, pr, order, gain, idx, gtab, sect, misc, total;
};
// The region holds, in turn: the ring + positions, the V rows of an active set and of the rows picked, the triangle, the
// flags of kept slots, the kept rows on their way out; the plain-dot route keeps its per-candidate arrays there.
__host__ __device__ inline PfSmem plan_pf_smem(int N, int budget) {
    PfSmem p;
    const unsigned np = (unsigned)((N + 3) & ~3);
    unsigned region = kPfRing + np * 4;
    const unsigned tile = (kPfActive + kPfMaxBudget) * 256u, plain = 3 * np * 4 + align16(np * 2) + align16(np);
    if (region < tile) region = tile;
    if (region < plain) region = plain;
    p.region = 0;
    p.spos = kPfRing;
    unsigned o = align16(region);
    p.s = o;      o += np * 4;
    p.act = o;    o += kPfActive * 2;
    p.ar = o;     o += kPfActive * 4;
    p.am = o;     o += kPfActive * 4;
    p.pr = o;     o += kPfMaxBudget * 4;
    p.order = o;  o += align16((unsigned)budget * 4);
    p.gain = o;   o += align16((unsigned)budget * 4);
    p.idx = o;    o += align16((unsigned)budget * 4);
    p.gtab = o;   o += 1024;   // folded statistic and phase steps
    p.sect = o;   o += 256;
    p.misc = o;   o += 256;    // mbarriers (full 4, empty 4, product), tensor-memory base, counters, arg-max exchange
    p.total = o + 1024;        // room to align the base to 1024 bytes
    return p;
}

// Thread-block clusters: rank of this CTA, its arrival at the cluster's barrier and the wait for the others' (the aligned forms:
// a warp's lanes come together first, whatever branches they come from), and a float or an int stored to another CTA's shared
// memory (at the address of this CTA's own).
__device__ __forceinline__ int cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return (int)r;
}
__device__ __forceinline__ void cluster_arrive() {
    __syncwarp();
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_wait() {
    __syncwarp();
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_address(uint32_t own, int rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(own), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_store(uint32_t addr, uint32_t v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

// TAIL: a call of two launches (see launch_prefill), one CTA per event and several. The first lets the second start as soon as all of its own CTAs have, the second ends
// only when the first has, so that whatever follows on the stream comes after both.
__device__ __forceinline__ void let_dependents_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_for_launch_ahead() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <bool FUSED, int SPLIT, bool TAIL>
__global__ void __launch_bounds__(kStThreads, 2) event_prefill_kernel(const __grid_constant__ EventArgs a, const __grid_constant__ ScoreTab tab) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    __shared__ __align__(16) uint32_t part[2][kStWarps];       // per-warp partial counts, double-buffered
    __shared__ __align__(16) uint4 best_of[2][kStWarps];       // per-warp arg-max: key, 0xFFFFFFFF - slot, row
    const DevLayout& lay = a.lay;
    const EventId id = decode_event(lay, TAIL && SPLIT > 1 ? a.first_event + (int)blockIdx.x / SPLIT : blockIdx.x / SPLIT);
    const int rank = SPLIT > 1 ? cluster_rank() : 0;
    const int n = event_n(a, id.b);
    const int N = lay.N;
    const int bud = event_budget(a, id);
    const int picks = min(bud, n);
    const PfSmem sp = plan_pf_smem(N, a.budget);
    unsigned char* region = smem + sp.region;
    float* s = reinterpret_cast<float*>(smem + sp.s);
    int* spos = reinterpret_cast<int*>(region + sp.spos);
    unsigned short* act = reinterpret_cast<unsigned short*>(smem + sp.act);
    float* ar = reinterpret_cast<float*>(smem + sp.ar);   // norms of the active set's rows
    float* am = reinterpret_cast<float*>(smem + sp.am);   // their running maxima
    float* pr = reinterpret_cast<float*>(smem + sp.pr);   // norms of the rows picked
    int* order = reinterpret_cast<int*>(smem + sp.order);
    float* gain = reinterpret_cast<float*>(smem + sp.gain);
    int* idx = reinterpret_cast<int*>(smem + sp.idx);
    float2* gtab = reinterpret_cast<float2*>(smem + sp.gtab);
    unsigned long long* phitab = reinterpret_cast<unsigned long long*>(gtab + 64);
    float2* sect = reinterpret_cast<float2*>(smem + sp.sect);
    const uint32_t bar_full = smem_u32(smem + sp.misc), bar_empty = bar_full + 8 * kPfStages, barM = bar_full + 64;
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + sp.misc + 72);
    int* cnt = reinterpret_cast<int*>(smem + sp.misc + 80);  // [0] a wait ran out, [1] newest position, [2] irregular positions, [3] a round's picks, [4] the same at a bound, [5] see picks_cosine: tie_slot, [6] the active set's bound
    const uint32_t region_u32 = smem_u32(region);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool worker = warp < kStWarps;
    const bool similarity = a.greedy != 0 && picks > 1;   // (the first pick is the highest score in any case)
    const bool dense = lay.page_size == 0;
    const long long ev_off = dense ? id.b * lay.sb + id.l * lay.sl + id.h * lay.sh : 0;
    auto rowoff = [&](int j) -> long long {
        return dense ? ev_off + (long long)j * lay.sn : row_offset(lay, id.b, id.l, id.h, j);
    };
    __nv_bfloat16* Kg = reinterpret_cast<__nv_bfloat16*>(a.K);
    __nv_bfloat16* Vg = reinterpret_cast<__nv_bfloat16*>(a.V);
    const int* gpos = event_pos(a.pos, id);
    const bool rotate = gpos != nullptr;

    // (a cluster's first CTA alone stamps its phases: the others' clocks are those of other SMs)
    if (rank == 0) phase_stamp(id.e, 0);  // phases: 0 start, 1 tables + positions, 2 K scored, 3 s_(b), 4 active set / top-k, 5 triangle, 6 picks, 7 outputs, 8 end
    // ---- set-up: barriers, tensor memory, tables ----------------------------------------------------------
    if (tid == 0) {
        for (int i = 0; i < kPfStages; ++i) {
            mbar_init(bar_full + 8 * i, 1);
            mbar_init(bar_empty + 8 * i, kStWarps);
        }
        mbar_init(barM, 1);
        mbar_init_fence();
        cnt[0] = 0;
        cnt[1] = INT_MIN;
        cnt[2] = 0;
        if (TAIL && SPLIT == 1) let_dependents_launch();
    }
    if (warp == 0) {
        // (both resident CTAs' columns fit the SM; the right to allocate is given up at once, or the next CTA would not start)
        if (similarity && rank == 0) tmem_alloc(smem_u32(tmem_holder), kPfCols);
        else tmem_relinquish();
    }
    if (FUSED) {
        if (warp == 1) fill_sector_table(sect, lane);
        fill_statistic_tables(a, id.l * lay.H + id.h, tab, tid, gtab, phitab);
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (SPLIT > 1) cluster_arrive();   // (the others may write to this CTA's memory once all have come here)

    int bad = 0;
    if (FUSED) {
        // the stages of this CTA: all, or its share of them (in eights, so that rotations are taken afresh where they are
        // without a split and the scores are the same to the bit)
        const int all = (n + kStStageRows - 1) / kStStageRows;
        static_assert(kSplitStages == kChainRounds && kSplitStageRows == kStStageRows, "the rule of the split counts these stages");
        const int share = SPLIT > 1 ? ((all + SPLIT - 1) / SPLIT + kSplitStages - 1) / kSplitStages * kSplitStages : all;
        const int first = rank * share, stages = max(min(all - first, share), 0);
        // (the testing aid: where others have stages too only they are starved, and the first CTA has to learn of it from them)
        const bool starve = a.starve && (SPLIT == 1 || rank != 0 || all <= share);
        const int polls = SPLIT > 1 && !starve ? kWaitPolls : a.wait_polls;
        if (!worker) {
            // ---- producer: K through the ring ---------------------------------------------------------------------
            if (lane == 0) {
                for (int st = 0; st < stages; ++st) {
                    const int sl = st & (kPfStages - 1);
                    if (st >= kPfStages && !mbar_wait_bounded(bar_empty + 8 * sl, (uint32_t)((st / kPfStages - 1) & 1), polls)) {
                        atomicExch(&cnt[0], 1);
                        break;
                    }
                    const int r0 = (first + st) * kStStageRows, r1 = min(n, r0 + kStStageRows);
                    mbar_expect_tx(bar_full + 8 * sl, (uint32_t)(r1 - r0) * 256u);
                    // as few copies as the layout allows: the whole stage when its rows are contiguous, whole pages
                    // when pages are, else row by row (starve, a testing aid: none at all, the scoring warps' wait runs out)
                    for (int row = r0; row < r1 && !starve;) {
                        int run = 1;
                        if (dense && lay.sn == kTcD) run = r1 - row;
                        else if (!dense && lay.s_page_n == kTcD) run = min(r1 - row, lay.page_size - row % lay.page_size);
                        bulk_g2s(region_u32 + (uint32_t)sl * kStStageBytes + (uint32_t)(row - r0) * 256u, Kg + rowoff(row),
                                 (uint32_t)run * 256u, bar_full + 8 * sl);
                        row += run;
                    }
                }
            }
        } else {
            // ---- positions on chip; D: the spacing of rows one stage apart at the newest end, which a cache filled token
            // by token has everywhere (found once, the scoring loop then chains without looking at positions)
            // (every load of a thread is requested before the first is used: 896 events of 4096 rows 383.0 -> 379.4 us, without picks
            // 284.2 -> 280.6, a gain of 1 %, hardly more than runs of the same code differ by)
            const int p_last = rotate && n > kStStageRows ? gpos[n - 1] : 0, p_back = rotate && n > kStStageRows ? gpos[n - 1 - kStStageRows] : 0;
            const int p_ref = rotate && a.p_ref ? a.p_ref[id.b] : 0;
            int p[kPfKeys];
#pragma unroll
            for (int i = 0; i < kPfKeys; ++i) p[i] = rotate && tid + i * kStWork < n ? gpos[tid + i * kStWork] : 0;
            const long long D = (long long)p_last - (long long)p_back;
            int pmax = INT_MIN;
#pragma unroll
            for (int i = 0; i < kPfKeys; ++i)
                if (tid + i * kStWork < n) {
                    spos[tid + i * kStWork] = p[i];
                    pmax = max(pmax, p[i]);
                }
            pmax = __reduce_max_sync(0xFFFFFFFFu, pmax);
            if (lane == 0) atomicMax(&cnt[1], pmax);
            work_barrier();
            bool uni = true;
            for (int j = kStStageRows + tid; j < n; j += kStWork) uni &= (long long)spos[j] - (long long)spos[j - kStStageRows] == D;
            if (!uni) cnt[2] = 1;
            work_barrier();
            const bool uniform = cnt[2] == 0;
            long long pref = 0;
            if (rotate) pref = a.p_ref ? (long long)p_ref : (long long)cnt[1] + 1;
            if (rank == 0) phase_stamp(id.e, 1);
            // ---- scores -------------------------------------------------------------------------------------------
            const int grp = lane >> 3, f0 = (lane & 7) * 8;
            // A lane group scores two rows of every stage, 32 slots apart, as two independent chains; each chain steps by
            // one stage = 64 slots.
            const int D32 = (int)D;
            const bool d_fits = (long long)D32 == D;
            ChainScore ca, cb;  // cb uses ca's S
            ca.set_step(D, phitab + f0, sect);
            if (SPLIT > 1) cluster_wait();
            const uint32_t s_first = SPLIT > 1 ? cluster_address(smem_u32(s), 0) : 0u;
            for (int st = 0; st < stages; ++st) {
                const int sl = st & (kPfStages - 1);
                if (!mbar_wait_bounded(bar_full + 8 * sl, (uint32_t)((st / kPfStages) & 1), polls)) {
                    atomicExch(&cnt[0], 1);
                    break;
                }
                const int ja = (first + st) * kStStageRows + 4 * warp + grp, jb = ja + kStRoundRows;
                const bool la = ja < n, lb = jb < n;
                const unsigned char* krow = region + sl * kStStageBytes + (4 * warp + grp) * 256 + (lane & 7) * 16;
                bool fresh = (st & (kChainRounds - 1)) == 0 || a.no_chain || !d_fits;
                int pa = 0, pb = 0;
                if (fresh || !uniform) {
                    pa = la ? spos[ja] : 0;
                    pb = lb ? spos[jb] : 0;
                }
                if (!fresh && !uniform)
                    fresh = !__all_sync(0xFFFFFFFFu, (!la || pa - spos[ja - kStStageRows] == D32) && (!lb || pb - spos[jb - kStStageRows] == D32));
                if (fresh) {
                    if (la) ca.anchor(pref - (long long)pa, gtab + f0, phitab + f0, sect);
                    if (lb) cb.anchor(pref - (long long)pb, gtab + f0, phitab + f0, sect);
                } else {
                    ca.advance();
                    cb.advance_by(ca);
                }
                float acca = 0.f, accb = 0.f;
                if (la) acca = ca.dot(*reinterpret_cast<const uint4*>(krow), *reinterpret_cast<const uint4*>(krow + 128));
                if (lb) accb = cb.dot(*reinterpret_cast<const uint4*>(krow + kStRoundRows * 256), *reinterpret_cast<const uint4*>(krow + kStRoundRows * 256 + 128));
                __syncwarp();
                if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar_empty + 8 * sl) : "memory");
                // both rows' sums in three exchanges: lanes 0..3 of a group go on with row a, lanes 4..7 with row b
                const bool second = lane & 4;
                float acc = (second ? accb : acca) + __shfl_xor_sync(0xFFFFFFFFu, second ? acca : accb, 4);
                acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 2);
                acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 1);
                const int j = second ? jb : ja;
                if ((lane & 3) == 0 && j < n) {
                    if (SPLIT > 1 && rank != 0) cluster_store(s_first + 4u * (uint32_t)j, __float_as_uint(acc));
                    else s[j] = acc;
                    if (a.scores) a.scores[(long long)id.e * N + j] = acc;
                }
            }
        }
        if (SPLIT > 1 && !worker) cluster_wait();
        __syncthreads();
        if (SPLIT > 1) {
            // the first CTA goes on with all scores; what the others did lies in its memory, a wait that ran out there included
            if (rank != 0 && tid == 0 && cnt[0]) cluster_store(cluster_address(smem_u32(cnt), 0), 1u);
            cluster_arrive();
            if (rank == 0) cluster_wait();
            else if (!cnt[0]) return;
        }
        if (cnt[0]) {
            // a wait ran out: report it, give copies that may still be in flight a bounded chance to land, leave
            if (tid == 0) {
                if (a.status && rank == 0) a.status[id.e] = 3;
                for (int sl = 0; sl < kPfStages; ++sl) {
                    mbar_wait_bounded(bar_full + 8 * sl, 0, a.wait_polls);
                    mbar_wait_bounded(bar_full + 8 * sl, 1, a.wait_polls);
                }
            }
            if (similarity && rank == 0 && warp == 0) tmem_dealloc(*tmem_holder, kPfCols);
            if (TAIL && SPLIT > 1 && tid == 0) wait_for_launch_ahead();
            return;
        }
    } else {
        for (int j = tid; j < n; j += kStThreads) s[j] = a.scores[(long long)id.e * N + j];
        __syncthreads();
    }
    if (!worker) return;  // the producer warp is done; the work warps meet at their own barrier from here on

    phase_stamp(id.e, 2);
    // ---- keys: a run of consecutive slots per thread ----------------------------------------------------------
    const int run = (n + kStWork - 1) / kStWork | 1, j0 = tid * run;
    uint32_t key[kPfKeys];   // 0: no slot
#pragma unroll
    for (int i = 0; i < kPfKeys; ++i) {
        key[i] = 0u;
        if (i < run && j0 + i < n) {
            float v = s[j0 + i];
            if (!isfinite(v)) {
                bad = 1;
                v = -INFINITY;
                s[j0 + i] = v;
            }
            key[i] = orderable(v);
        }
    }
    int turn = 0;   // which half of `part` the next count uses
    // three counts over all keys, summed over the block (at most 5120 each)
    auto count3 = [&](uint32_t v1, uint32_t v2, uint32_t v3, int& t1, int& t2, int& t3) {
        uint32_t c = 0u;
#pragma unroll
        for (int i = 0; i < kPfKeys; ++i) c += (key[i] >= v1 ? 1u : 0u) + (key[i] >= v2 ? 1u << 10 : 0u) + (key[i] >= v3 ? 1u << 20 : 0u);
        c = __reduce_add_sync(0xFFFFFFFFu, c);   // (at most 32 x 21 per field)
        if (lane == 0) part[turn][warp] = c;
        work_barrier();
        t1 = t2 = t3 = 0;
        const uint4 p0 = *reinterpret_cast<const uint4*>(part[turn]), p1 = *reinterpret_cast<const uint4*>(part[turn] + 4);
        const uint32_t w[8] = {p0.x, p0.y, p0.z, p0.w, p1.x, p1.y, p1.z, p1.w};
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            t1 += w[i] & 1023u;
            t2 += (w[i] >> 10) & 1023u;
            t3 += w[i] >> 20;
        }
        turn ^= 1;
    };
    // A v with at least `want` keys >= v and `reach` their number: at most `enough` of them, which a few rounds (two bits each)
    // bring about, or, where too many keys are equal for that, the largest such v (its bits below `last` open, 0).
    auto search = [&](int last, int want, int enough, int& reach) -> uint32_t {
        uint32_t v = 0u;
        reach = n;
        for (int lo = 30; lo >= last && reach > enough; lo -= 2) {
            const uint32_t v1 = v | (1u << lo), v2 = v | (2u << lo), v3 = v | (3u << lo);
            int t1, t2, t3;
            count3(v1, v2, v3, t1, t2, t3);
            if (t1 >= want) {
                v = t3 >= want ? v3 : (t2 >= want ? v2 : v1);
                reach = t3 >= want ? t3 : (t2 >= want ? t2 : t1);
            }
        }
        return v;
    };
    // exclusive prefix over the threads of two counts (16 bits each), and their totals
    auto scan2 = [&](uint32_t mine, uint32_t& total) -> uint32_t {
        uint32_t inc = mine;
#pragma unroll
        for (int off = 1; off < 32; off <<= 1) {
            const uint32_t o = __shfl_up_sync(0xFFFFFFFFu, inc, off);
            if (lane >= off) inc += o;
        }
        if (lane == 31) part[turn][warp] = inc;
        work_barrier();
        uint32_t before = 0u;
        total = 0u;
#pragma unroll
        for (int w = 0; w < kStWarps; ++w) {
            const uint32_t p = part[turn][w];
            before += w < warp ? p : 0u;
            total += p;
        }
        turn ^= 1;
        return before + inc - mine;
    };

    // ---- s_(b), the picks-th largest key, from below: for the pruning and as the start of top-k's ranks a key that a few more
    // than `picks` rows reach will do
    int reach = 0;
    const uint32_t kb = picks > 0 ? search(similarity ? 14 : 0, picks, similarity ? picks + picks / 4 : kPfRanked, reach) : 0xFFFFFFFFu;
    phase_stamp(id.e, 3);
    bool listed = false;   // idx[] holds the kept slots already

    if (!similarity && reach <= kPfRanked) {
        // top-k: the rows that reach kb, in slot order, one per thread; a row's place in the pick order is the number of rows
        // with a larger key (equal keys: lower slot first), and the first `picks` of them are kept
        uint32_t* ck = reinterpret_cast<uint32_t*>(region);       // (positions and ring are no longer needed)
        unsigned short* cj = reinterpret_cast<unsigned short*>(ck + kPfRanked);
        uint32_t c = 0u, total;
#pragma unroll
        for (int i = 0; i < kPfKeys; ++i) c += key[i] >= kb && key[i] != 0u;
        uint32_t pos = scan2(c, total);
#pragma unroll
        for (int i = 0; i < kPfKeys; ++i)
            if (key[i] >= kb && key[i] != 0u) {
                ck[pos] = key[i];
                cj[pos++] = (unsigned short)(j0 + i);
            }
        if (tid >= (int)total) ck[tid] = 0u;
        work_barrier();
        const uint32_t mine = ck[tid];
        int rank = 0;
        for (int o = 0; o < (int)total; o += 4) {
            const uint4 k4 = *reinterpret_cast<const uint4*>(ck + o);
            rank += (k4.x > mine || (k4.x == mine && o < tid)) + (k4.y > mine || (k4.y == mine && o + 1 < tid)) +
                    (k4.z > mine || (k4.z == mine && o + 2 < tid)) + (k4.w > mine || (k4.w == mine && o + 3 < tid));
        }
        const bool kept = tid < (int)total && rank < picks;
        const uint32_t at = scan2(kept ? 1u : 0u, total);
        if (kept) {
            order[rank] = cj[tid];
            gain[rank] = from_orderable(mine);
            idx[at] = cj[tid];
        }
        listed = true;
        phase_stamp(id.e, 4);
    } else if (!similarity) {
        // top-k: every key above the picks-th one, and the lowest slots among those equal to it; kept slots in slot order
        uint32_t c = 0u, total;
#pragma unroll
        for (int i = 0; i < kPfKeys; ++i) c += (key[i] > kb ? 1u : 0u) + (key[i] == kb && kb ? 1u << 16 : 0u);
        const uint32_t before = scan2(c, total);
        const int ties = picks - (int)(total & 0xFFFFu);          // how many of the equal ones are kept
        int eq = (int)(before >> 16), pos = (int)(before & 0xFFFFu) + min(eq, ties);
        float* ps = reinterpret_cast<float*>(region);             // (positions and ring are no longer needed)
#pragma unroll
        for (int i = 0; i < kPfKeys; ++i) {
            const bool above = key[i] > kb, tie = key[i] == kb && kb;
            if (above || (tie && eq < ties)) {
                idx[pos] = j0 + i;
                ps[pos] = from_orderable(key[i]);
                ++pos;
            }
            eq += tie;
        }
        work_barrier();
        // pick order: by score, equal scores by slot
        for (int t = tid; t < picks; t += kStWork) {
            const uint32_t k = orderable(ps[t]);
            int rank = 0;
#pragma unroll 4
            for (int o = 0; o < picks; ++o) {
                const uint32_t ko = orderable(ps[o]);
                rank += ko > k || (ko == k && o < t);
            }
            order[rank] = idx[t];
            gain[rank] = ps[t];
        }
        listed = true;
        phase_stamp(id.e, 4);
    } else {
        const float sb = from_orderable(kb);
        // -inf keeps everyone (also where kb is below every finite value's key)
        const float thr = a.no_prune || kb < 0x00800000u ? -INFINITY : fmaf(-1.001f, a.lam, sb) - 1e-6f * fabsf(sb);
        const uint32_t low = orderable(thr);
        // the slots with keys in the pool above `bound`, in slot order
        auto list = [&](uint32_t bound, unsigned short* out) -> int {
            uint32_t c = 0u, total;
#pragma unroll
            for (int i = 0; i < kPfKeys; ++i) c += key[i] >= low && key[i] > bound;
            uint32_t pos = scan2(c, total);
#pragma unroll
            for (int i = 0; i < kPfKeys; ++i)
                if (key[i] >= low && key[i] > bound) out[pos++] = (unsigned short)(j0 + i);
            work_barrier();
            return (int)total;
        };
        constexpr uint32_t half_bytes = (kPfActive + kPfMaxBudget) * 128u;
        float* tri = reinterpret_cast<float*>(region);
        const uint32_t tbase = *tmem_holder;
        const int quarter = warp & 3, rho = 32 * quarter + lane;            // row of a product this thread reads
        const uint32_t lanes = tbase + ((uint32_t)(32 * quarter) << 16);
        uint32_t phase = 0u;
        int made = 0, idle = 0;   // idle: rounds without a pick since the last one
        // a product of the tile rows from row_a on with those from row_b on, into the columns from col on
        auto product = [&](int row_a, int row_b, int cols, uint32_t col) {
            const uint32_t idesc = umma_idesc_bf16(128, cols);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                const uint32_t koff = (uint32_t)(kk >> 2) * half_bytes + (uint32_t)(kk & 3) * 32u;
                umma_bf16(tbase + col, umma_desc_sw128(region_u32 + (uint32_t)row_a * 128u + koff),
                          umma_desc_sw128(region_u32 + (uint32_t)row_b * 128u + koff), idesc, kk > 0 ? 1u : 0u);
            }
        };
        auto products_done = [&]() {
            if (!mbar_wait_bounded(barM, phase, a.wait_polls)) cnt[0] = 1;
            phase ^= 1u;
            tc_fence_after();
        };
        // A round without a pick makes the values of its rows known, and the next set holds the rows between the best of
        // those and the bound, all of them unknown, until they fit a set: n / 192 + 1 such rounds at most. (The limit is a
        // safeguard.)
        while (made < picks && idle <= n / kPfActive + 2) {
            // ---- the active set: at most 192 rows (bound 0: the pool is no larger)
            int pool_size, unused1, unused2;
            count3(low, 0xFFFFFFFFu, 0xFFFFFFFFu, pool_size, unused1, unused2);
            ActiveBound found{0u, 0};
            if (pool_size > kPfActive) found = active_bound(low, kb, kPfActive, kPfEnough, kPfLeast, count3);
            // (through shared memory: held in a register over the rest of the round, it costs this kernel 88 bytes of spills and
            // 0.8 % of 384 us for 896 events of 4096 rows)
            if (tid == 0) {
                cnt[5] = 0;
                cnt[6] = (int)found.key;
            }
            work_barrier();
            const uint32_t bound = (uint32_t)*(volatile int*)(cnt + 6);
            if (found.ties) {
                // the lowest slots of those that equal the bound move above it (a key may lie above its row's value)
                uint32_t c = 0u, total;
#pragma unroll
                for (int i = 0; i < kPfKeys; ++i) c += key[i] == bound;
                int eq = (int)scan2(c, total);
#pragma unroll
                for (int i = 0; i < kPfKeys; ++i)
                    if (key[i] == bound) {
                        if (eq < found.ties) ++key[i];
                        else if (eq == found.ties) cnt[5] = j0 + i;
                        ++eq;
                    }
            }
            const int R = list(bound, act);
            if (bound == 0u && R < picks - made) break;   // (values lost to overflowed cosines)
            if (made == 0) phase_stamp(id.e, 4);

            // ---- V rows of the active set and of the rows picked as a swizzled operand tile ------------------------------
            for (int x = tid; x < (R + made) * 16; x += kStWork) {
                const int i = x >> 4, c = x & 15;
                const int row = i < R ? i : kPfActive + i - R, j = i < R ? act[i] : order[i - R];
                cp_async16(region_u32 + tile_chunk(row, c, half_bytes), Vg + rowoff(j) + c * 8);
            }
            cp_async_wait_all();
            fence_proxy_async();
            tc_fence_before();
            work_barrier();
            tc_fence_after();
            // rows from 128 on (nb of them) lie in a second block of rows, base2 on
            const int ncols = max((R + 15) & ~15, 16), nb = R > 128 ? R - 128 : 0, base2 = max(ncols - 128, 0);
            const int ra = base2 + rho - 128;   // this thread's row of the second block, counted from row 128
            const bool second = warp >= 4;      // warps 4..7 read the second block
            if (made > 0) {
                // maxima over the rows picked so far
                const int pcols = (made + 15) & ~15;
                if (tid == 0) {
                    product(0, kPfActive, pcols, 0u);
                    if (nb > 0) product(base2, kPfActive, pcols, 128u);
                    umma_commit(barM);
                }
                products_done();
                float m = 0.f;
                if (!second || nb > 0) {
                    for (int cb = 0; cb < (made + 31) >> 5; ++cb) {
                        uint32_t v[32];
                        tmem_ld32(lanes + (second ? 128u : 0u) + (uint32_t)(32 * cb), v);
                        tmem_ld_wait();
#pragma unroll
                        for (int k = 0; k < 32; ++k)
                            if (32 * cb + k < made) m = fmaxf(m, pr[32 * cb + k] * __uint_as_float(v[k]));
                    }
                }
                if (!second && rho < R) am[rho] = m;
                if (second && ra >= 0 && ra < nb) am[128 + ra] = m;
                tc_fence_before();
                work_barrier();   // the columns have been read
                tc_fence_after();
            }
            if (tid == 0 && (FUSED || !a.starve)) {
                product(0, 0, ncols, 0u);
                // the second block against rows 128.. gives their cosines against one another; those against rows < 128
                // are those rows' columns from 128 on
                if (nb > 0) product(base2, 128, ncols - 128, (uint32_t)ncols);
                umma_commit(barM);
            }
            products_done();
            work_barrier();   // the products have read the whole tile before the triangle lands on it
            if (cnt[0]) {
                if (warp == 0) tmem_dealloc(tbase, kPfCols);
                if (tid == 0 && a.status) a.status[id.e] = 3;
                if (!FUSED) select_gave_up(a, id.e, kStWork);
                if (TAIL && SPLIT > 1 && tid == 0) wait_for_launch_ahead();
                return;
            }
            // lower triangle -> shared memory: warps 0..3 the first product's columns up to the row itself, warps 4..7 its
            // columns from 128 on (to the rows from 128 on, transposed) and the second product
            if (!second) {
                const int trow = tri_row(rho);
                if (32 * quarter < R) {
                    for (int cb = 0; cb < quarter; ++cb) {
                        uint32_t v[32];
                        tmem_ld32(lanes + (uint32_t)(32 * cb), v);
                        tmem_ld_wait();
                        if (rho < R) {
#pragma unroll
                            for (int k = 0; k < 32; ++k) tri[trow + 32 * cb + k] = __uint_as_float(v[k]);
                        }
                    }
                    uint32_t v[32];
                    tmem_ld32(lanes + (uint32_t)(32 * quarter), v);
                    tmem_ld_wait();
                    if (rho < R) {
#pragma unroll
                        for (int k = 0; k < 32; ++k)
                            if (k <= lane) tri[trow + 32 * quarter + k] = __uint_as_float(v[k]);
                        ar[rho] = 1.f / (sqrtf(tri[trow + rho]) + a.eps);  // read back: this thread stored it
                    }
                }
            } else if (nb > 0) {
                for (int cb = 0; cb < (nb + 31) >> 5; ++cb) {
                    uint32_t v[32];
                    tmem_ld32(lanes + 128u + (uint32_t)(32 * cb), v);
                    tmem_ld_wait();
#pragma unroll
                    for (int k = 0; k < 32; ++k)
                        if (32 * cb + k < nb) tri[tri_row(128 + 32 * cb + k) + rho] = __uint_as_float(v[k]);
                }
                float diag = 0.f;
                for (int cb = 0; cb < (nb + 31) >> 5; ++cb) {
                    uint32_t v[32];
                    tmem_ld32(lanes + (uint32_t)ncols + (uint32_t)(32 * cb), v);
                    tmem_ld_wait();
                    if (ra >= 0 && ra < nb) {
#pragma unroll
                        for (int k = 0; k < 32; ++k) {
                            if (32 * cb + k <= ra) tri[tri_row(128 + ra) + 128 + 32 * cb + k] = __uint_as_float(v[k]);
                            diag = (32 * cb + k == ra) ? __uint_as_float(v[k]) : diag;
                        }
                    }
                }
                if (ra >= 0 && ra < nb) ar[128 + ra] = 1.f / (sqrtf(diag) + a.eps);
            }
            tc_fence_before();
            work_barrier();
            tc_fence_after();
            if (made == 0) phase_stamp(id.e, 5);

            // ---- Algorithm 1 over the active set in warp 0 -----------------------------------------------------------
            if (warp == 0) {
                const bool ok = picks_cosine<kPfActive / 32, true>(lane, R, picks - made, s, act, ar, a.lam, tri,
                                                                   reinterpret_cast<uint32_t*>(gain) + made, order + made, bound, am,
                                                                   cnt + 4, made > 0 ? am : nullptr, cnt + 5);
                if (lane == 0) cnt[3] = ok ? picks - made : cnt[4];
            }
            work_barrier();
            const int got = cnt[3];
            uint32_t* upper = reinterpret_cast<uint32_t*>(region);   // by slot: what is known of the active set now
            const bool more = made + got < picks;
            if (more) {
                for (int j = tid; j < n; j += kStWork) upper[j] = 0xFFFFFFFFu;
                work_barrier();
                if (tid < R) {
                    const float m = am[tid];
                    upper[act[tid]] = m == __int_as_float(0x7f800000) ? 0u
                                                                      : orderable(fmaf(-fmaxf(penalty_rate(a.lam, ar[tid]), 1e-30f), m, fmaxf(s[act[tid]], kLowestScore)));
                }
            }
            for (int t = made + tid; t < made + got; t += kStWork) {
                gain[t] = from_orderable(reinterpret_cast<uint32_t*>(gain)[t]);
                pr[t] = ar[order[t]];
                order[t] = act[order[t]];
            }
            work_barrier();
            if (more) {
#pragma unroll
                for (int i = 0; i < kPfKeys; ++i) {
                    if (i >= run || j0 + i >= n) continue;
                    const uint32_t u = upper[j0 + i];
                    if (u != 0xFFFFFFFFu) key[i] = u;
                }
                work_barrier();
            }
            made += got;
            idle = got ? 0 : idle + 1;
        }
        tc_fence_before();
        work_barrier();
        if (warp == 0) tmem_dealloc(tbase, kPfCols);
        if (made < picks) {
            // ---- plain-dot route: the whole pool from the start; V rows read in place, state in the region ----------------
            auto vchunk = [&](int j, int c) -> uint4 { return *reinterpret_cast<const uint4*>(Vg + rowoff(j) + c * 8); };
            auto vdot = [&](int i, int j) -> float {   // of two slots' V rows
                float2 acc = make_float2(0.f, 0.f);
#pragma unroll 4
                for (int c = 0; c < 16; ++c) dot8_bf16(vchunk(i, c), vchunk(j, c), acc);
                return acc.x + acc.y;
            };
            const unsigned np = (unsigned)((N + 3) & ~3);
            float* ps = reinterpret_cast<float*>(region);
            float* m = ps + np;
            float* r = m + np;
            unsigned short* pool = reinterpret_cast<unsigned short*>(r + np);
            unsigned char* gone = reinterpret_cast<unsigned char*>(pool) + align16(np * 2);
#pragma unroll
            for (int i = 0; i < kPfKeys; ++i) key[i] = i < run && j0 + i < n ? orderable(s[j0 + i]) : 0u;
            const int P = list(0u, pool);
            for (int q = tid; q < P; q += kStWork) {
                ps[q] = fmaxf(s[pool[q]], kLowestScore);
                m[q] = 0.f;
                gone[q] = 0;
                r[q] = fmaxf(1.f / (sqrtf(vdot(pool[q], pool[q])) + a.eps), 1e-30f);
            }
            work_barrier();
            int last = -1;
            // Pass t folds the cosines of pick t - 1 into every candidate's running maximum and, in the same sweep,
            // finds the arg-max of Eq. 2 for pick t. The first pass (no pick yet) is the plain arg-max of the scores.
            for (int t = 0; t < picks; ++t) {
                uint32_t hi = 0u, lo = 0u, row = 0u;
                for (int q = tid; q < P; q += kStWork) {
                    if (gone[q] || q == last) continue;   // (the last pick's flag may not be visible yet)
                    float mm = m[q];
                    if (last >= 0) {
                        mm = fmaxf(mm, fminf(r[last] * vdot(pool[q], pool[last]), 1e30f));
                        m[q] = mm;
                    }
                    const uint32_t k = orderable(fmaf(-penalty_rate(a.lam, r[q]), mm, ps[q]));
                    if (k > hi) { hi = k; lo = 0xFFFFFFFFu - (uint32_t)pool[q]; row = (uint32_t)q; }
                }
                // block-wide arg-max, ties to the lower slot; the row travels with it
                const uint32_t whi = __reduce_max_sync(0xFFFFFFFFu, hi);
                const uint32_t wlo = __reduce_max_sync(0xFFFFFFFFu, hi == whi ? lo : 0u);
                if (hi == whi && lo == wlo) best_of[t & 1][warp] = make_uint4(hi, lo, row, 0u);   // (none left: any lane's zeros)
                work_barrier();
                uint4 best = best_of[t & 1][0];
#pragma unroll
                for (int w = 1; w < kStWarps; ++w) {
                    const uint4 o = best_of[t & 1][w];
                    if (o.x > best.x || (o.x == best.x && o.y > best.y)) best = o;
                }
                last = (int)best.z;
                if (tid == 0) {
                    const float g = from_orderable(best.x);
                    gain[t] = g <= -2.9e38f ? -INFINITY : g;
                    order[t] = pool[last];
                    gone[last] = 1;
                }
            }
            work_barrier();
        }
    }
    bad = __any_sync(0xFFFFFFFFu, bad);
    if (lane == 0 && bad) cnt[2] = 2;   // (the positions' flag, 0 or 1, has been read long since)
    work_barrier();

    phase_stamp(id.e, 6);
    // ---- sort(S) and outputs -------------------------------------------------------------------------
    if (!listed) {
        unsigned char* taken = region;
        for (int j = tid; j < (n + 3) / 4; j += kStWork) reinterpret_cast<uint32_t*>(taken)[j] = 0u;
        work_barrier();
        for (int t = tid; t < picks; t += kStWork) taken[order[t]] = 1;
        work_barrier();
        uint32_t c = 0u, total;
        for (int i = 0; i < run && j0 + i < n; ++i) c += taken[j0 + i];
        uint32_t pos = scan2(c, total);
        for (int i = 0; i < run && j0 + i < n; ++i)
            if (taken[j0 + i]) idx[pos++] = j0 + i;
    }
    for (int t = picks + tid; t < a.budget; t += kStWork) idx[t] = -1;
    work_barrier();
    const long long ob = (long long)id.e * a.budget;
    for (int t = tid; t < a.budget; t += kStWork) {
        a.idx_sorted[ob + t] = idx[t];
        if (a.pick_order) a.pick_order[ob + t] = t < picks ? order[t] : -1;
        if (a.pick_gain) a.pick_gain[ob + t] = t < picks ? gain[t] : 0.f;
    }
    if (tid == 0) {
        if (a.n_kept) a.n_kept[id.e] = picks;
        if (a.status) a.status[id.e] = n < bud ? 2 : (cnt[2] == 2 ? 1 : 0);
    }
    if (!FUSED) return;

    phase_stamp(id.e, 7);
    // ---- compaction in place: every kept row is on chip before the first store ---------------------------
    int* wpos = a.pos.p ? a.pos.p + id.b * a.pos.sb + id.l * a.pos.sl + id.h * a.pos.sh : nullptr;
    for (int x = tid; x < picks * 16; x += kStWork) {
        const long long off = rowoff(idx[x >> 4]) + (x & 15) * 8;
        cp_async16(region_u32 + (uint32_t)x * 16u, Kg + off);
        cp_async16(region_u32 + 32768u + (uint32_t)x * 16u, Vg + off);
    }
    int pv = 0;
    if (wpos && tid < picks) pv = gpos[idx[tid]];
    cp_async_wait_all();
    work_barrier();
    for (int x = tid; x < picks * 16; x += kStWork) {
        const long long off = rowoff(x >> 4) + (x & 15) * 8;
        *reinterpret_cast<uint4*>(Kg + off) = *reinterpret_cast<const uint4*>(region + x * 16);
        *reinterpret_cast<uint4*>(Vg + off) = *reinterpret_cast<const uint4*>(region + 32768 + x * 16);
    }
    if (wpos && tid < picks) wpos[tid] = pv;
    if (TAIL && SPLIT > 1 && tid == 0) wait_for_launch_ahead();
    phase_stamp(id.e, 8);
}

}  // namespace akv
