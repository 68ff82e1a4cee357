// Event kernel for bf16, d = 128, per-head signatures, N <= 256 and budgets up to 128 (the shapes of the
// Qwen-7B-shaped batch and of the decode cadence: 256 candidates -> 128). Same structure as event_tri_kernel
// (K rows scored from shared memory, here all of them at once, pool by bisection, cosine matrix on tcgen05, its lower triangle in shared
// memory, Algorithm 1 as a one-warp loop), for an ACTIVE SET instead of the whole pool:
//
//   The picks hardly ever reach beyond the best-scored few dozen rows past the budget. The cosine matrix is
//   therefore formed only for the pool's best-scored rows, 158 to 180 of them (64 KB of triangle: three CTAs
//   per SM; 138 to 158 and 49 KB: four), and only their V rows are read. Every candidate left out scores at most `bound` (see active_bound),
//   and its Eq. 2 value never exceeds its score: the loop over the active set is exact as long as its
//   winning value stays above that bound. In the rare event where it does not, the picks made so far stand and
//   the remaining ones (a few, as a rule) are taken over the whole pool with rows of the cosine matrix as plain
//   dot products, starting from the running maxima the loop had reached.
//
//   Rows 128.. of the active set: a second product (the operand's last 128 rows against rows 128..) gives their
//   cosines against one another; their cosines against rows < 128 are those rows' columns 128.. by symmetry.
#pragma once
#include "akv_event_tri.cuh"
#include "akv_score_order.cuh"

namespace akv {

// Shared memory -> global memory as one bulk copy (16-byte aligned, a multiple of 16 bytes), and the wait that
// must precede leaving the CTA or reusing the source: until the copies issued by this thread have read it.
__device__ __forceinline__ void bulk_s2g(void* dst, uint32_t src, uint32_t bytes) {
    asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_store_wait_read() {
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// FUSED: score + select + compact; otherwise selection only (scores are read from a.scores and
// nothing is rewritten).
// FORM (PoolShape): kPoolWideForm, eight warps for a call of no more events than SMs. Alone on its SM an event is a chain of phases that
// too few warps hide: of 256 rows to 128, 55.2 -> 49.0 thousand cycles (scores 12.5 -> 10.4, picks in pairs 24.7 -> 22.5, triangle 3.2 -> 2.6,
// compaction 5.1 -> 4.4); 112 of them 35.1 -> 31.0 us, in pages 37.1 -> 33.0, top-k 20.7 -> 18.7. Not for what event_tri_kernel takes:
// alone, 112 events of 192 rows to 64 gain 2 us of 27 (in pages 4 of 29), but that kernel has six events on an SM, and four streams with such
// a call each take 41 us there, 50 here (in pages 43 and 80). kPoolThree, four warps and three events per SM. kPoolFour, four events per
// SM: latency bounds a call of many events (34 % of the issue slots used), so what counts is how many an SM holds. For that the last K rows come
// late, the triangle has 158 rows and the last kept V rows wait in registers: 2368 events of 256 rows to 96 191 -> 164 us, in pages
// 198 -> 181 (launch_tri says which calls). PAGED: with the layout known to the compiler 1792 events with a shared matrix take 198 us (all of the
// call) instead of 222. All forms score the rows in the same chains and have the same active set: an event has the same bits in each.
template <bool FUSED, int FORM, bool PAGED>
__global__ void __launch_bounds__(PoolShape<FORM>::kThreads, PoolShape<FORM>::kCtas) event_pool_kernel(const __grid_constant__ EventArgs a, const __grid_constant__ ScoreTab tab) {
    using Shape = PoolShape<FORM>;
    constexpr bool WIDE = FORM == kPoolWideForm, FOUR = FORM == kPoolFour;
    constexpr int NT = Shape::kThreads, NW = NT / 32;
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const DevLayout& lay = a.lay;
    const EventId id = decode_event(lay, blockIdx.x);
    const int n = event_n(a, id.b);
    const int N = lay.N;
    const int bud = event_budget(a, id);
    const int picks = min(bud, n);
    const TriSmem sp = plan_pool_event_smem<FORM>(N, a.budget, PAGED);
    unsigned char* tile = smem + sp.tile;
    float* tri = reinterpret_cast<float*>(tile);  // lower triangle of the cosine matrix, after the product
    float* s = reinterpret_cast<float*>(smem + sp.s);
    uint32_t* key = reinterpret_cast<uint32_t*>(smem + sp.key);
    float* r = reinterpret_cast<float*>(smem + sp.key);  // reuses the score keys' storage
    int* spos = reinterpret_cast<int*>(smem + sp.spos);
    unsigned short* bypool = reinterpret_cast<unsigned short*>(smem + sp.bypool);
    uint32_t* kept = reinterpret_cast<uint32_t*>(smem + sp.taken);
    int* order = reinterpret_cast<int*>(smem + sp.order);
    float* gain = reinterpret_cast<float*>(smem + sp.gain);
    int* idx = reinterpret_cast<int*>(smem + sp.idx);
    float2* sect = reinterpret_cast<float2*>(smem + sp.sect);
    const uint32_t barK = smem_u32(smem + sp.misc);
    const uint32_t barM = barK + 8;
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + sp.misc + 16);
    int* pool_holder = reinterpret_cast<int*>(smem + sp.misc + 20);
    int* pick_holder = reinterpret_cast<int*>(smem + sp.misc + 24);
    int* redi = reinterpret_cast<int*>(smem + sp.misc + 32);
    uint32_t* bound_holder = reinterpret_cast<uint32_t*>(smem + sp.misc + 28);  // key that no candidate outside the active set exceeds
    float* thr_holder = reinterpret_cast<float*>(smem + sp.misc + 56);          // the pool's score threshold
    int* tie_holder = reinterpret_cast<int*>(smem + sp.misc + 60);              // see picks_cosine: tie_slot
    const uint32_t tile_u32 = smem_u32(tile);
    constexpr uint32_t half_bytes = Shape::kOperandRows * 128u;  // the operand's two 128-byte column halves
    const uint32_t barL = barK + 48;  // K rows that wait for a free slot
    const int steps = score_steps(n), second = 16 * steps;   // the second chain's first row
    const int late0 = 16 * (steps - kLateSteps);             // of a chain's rows, the first that comes late
    const int n_late = FOUR && FUSED && n > Shape::kRows ? n - 2 * late0 : 0;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool similarity = a.greedy != 0 && picks > 1;   // (the first pick is the highest score in any case)
    const int np4 = (N + 3) & ~3;
    // row addressing: dense events are one base offset plus a row stride
    // (Three events per SM in pages look at the layout although it is known: with a constant here 16 384 events of 256 rows to 128 take
    // 2007 us a pass instead of 1911. Not for its registers, 138 instead of 106: held to 122 or to 96 of them it takes 2023 and 2118.)
    const bool dense = PAGED && FORM == kPoolThree ? lay.page_size == 0 : !PAGED;
    const long long ev_off = dense ? id.b * lay.sb + id.l * lay.sl + id.h * lay.sh : 0;
    // paged: where the event's pages start, looked up once by as many lanes of warp 0 at the same time (the block table's
    // entries come from L2; looked up row by row and copy by copy: 16 384 events of 256 rows to 128 in pages of 64 1631 us, 1600 so,
    // 8192 in pages of 16 798 and 771). The other warps read them behind the next block-wide barrier.
    long long* page_off = reinterpret_cast<long long*>(smem + sp.pages);
    const int pages = dense ? 0 : event_pages(N, lay.page_shift);
    const bool few_pages = !dense && pages <= kPageOffsets;
    if (few_pages) {
        if (tid < pages) page_off[tid] = row_offset(lay, id.b, id.l, id.h, tid << lay.page_shift);
        __syncwarp();
    }
    auto rowoff = [&](int j) -> long long {
        if (dense) return ev_off + (long long)j * lay.sn;
        return few_pages ? page_off[j >> lay.page_shift] + (long long)(j & (lay.page_size - 1)) * lay.s_page_n : row_offset(lay, id.b, id.l, id.h, j);
    };
    __nv_bfloat16* Kg = reinterpret_cast<__nv_bfloat16*>(a.K);
    __nv_bfloat16* Vg = reinterpret_cast<__nv_bfloat16*>(a.V);
    // shared signatures (Eq. 1, or its per-layer variant): the cosines come from the matrix formed once per
    // sequence (or per sequence and layer) instead of from this head's V rows
    const float* G = a.gram ? a.gram + id.b * a.gram_sb + id.l * a.gram_sl : nullptr;

    phase_stamp(id.e, 0);  // phases: 0 start, 1 tensor memory claimed, 2 K scored, 3 pool, 4 V operand, 5 product, 6 triangle, 7 picks, 8 outputs, 9 end
    // Tensor memory is claimed first and the right to allocate given up at once: the SM starts its
    // next CTA of this kernel only after that, so a late allocation would serialise the CTAs.
    // K rows [r0, r1) -> tile slots from slot0 on: as few bulk copies as the layout allows (whole event
    // when its rows are contiguous, whole pages when pages are, else row by row), all issued by one
    // thread (a bulk copy is a per-warp instruction)
    auto request_k_rows = [&](int r0, int r1, int slot0, uint32_t bar) {
        for (int row = r0; row < r1 && !a.starve;) {  // starve (testing aid): nothing is requested, the waits run out
            int run = 1;
            if (dense && lay.sn == kTcD) run = min(r1 - row, 128);
            else if (!dense && lay.s_page_n == kTcD) run = min(r1 - row, lay.page_size - (row & (lay.page_size - 1)));
            bulk_g2s(tile_u32 + (uint32_t)(slot0 + row - r0) * 256u, Kg + rowoff(row), (uint32_t)run * 256u, bar);
            row += run;
        }
    };
    if (tid == 0) {
        mbar_init(barK, 1);
        mbar_init(barM, 1);
        if (FOUR) mbar_init(barL, 1);
        mbar_init_fence();
        // the K rows are asked for before anything else: the wait for tensor memory below overlaps their flight
        if (FUSED) {
            mbar_expect_tx(barK, (uint32_t)(n - n_late) * 256u);
            if (n_late > 0) {
                request_k_rows(0, late0, 0, barK);
                request_k_rows(second, second + late0, kChainSlots, barK);
            } else {
                request_k_rows(0, n, 0, barK);
            }
        }
    }
    if (FUSED && warp == 1) fill_sector_table(sect, lane);
    // (this kernel claims half of the SM's columns: two of the CTAs on an SM hold theirs at a time, the others wait in the
    // allocation until one has moved its triangle out; claiming late instead measured 2 % slower)
    const bool have_tmem = similarity && !G;
    if (!have_tmem && warp == 0) tmem_relinquish();  // this event takes no tensor memory
    if (have_tmem && warp == 0) tmem_alloc(smem_u32(tmem_holder), kPoolCols);
    tc_fence_before();
    // The address of the columns is read after the next block-wide barrier: in the fused kernel that is the one
    // that follows the position and statistic loads, so that warps 1..3 do those while warp 0 may still be
    // waiting for columns.
    uint32_t tbase = 0u;
    if (!FUSED) {
        __syncthreads();
        tc_fence_after();
        tbase = have_tmem ? *tmem_holder : 0u;
    }

    phase_stamp(id.e, 1);
    // ---- scores ---------------------------------------------------------------------------------
    int bad = 0;
    int timeout = 0;
    if (FUSED) {
        const int* gpos = event_pos(a.pos, id);
        const bool rotate = gpos != nullptr;
        int pmax = INT_MIN;
        for (int j = tid; j < n; j += NT) {
            const int p = rotate ? gpos[j] : 0;
            spos[j] = p;
            pmax = max(pmax, p);
        }
        // folded statistic g_f = c_f z(q)_f / sqrt(d) and the frequencies' phase steps, once per event, in
        // shared memory (storage that the selection uses later)
        float2* gtab = reinterpret_cast<float2*>(smem + sp.bypool);
        unsigned long long* phitab = reinterpret_cast<unsigned long long*>(gtab + 64);
        fill_statistic_tables(a, id.l * lay.H + id.h, tab, tid, gtab, phitab);
        if (rotate) {
#pragma unroll
            for (int off = 16; off > 0; off >>= 1) pmax = max(pmax, __shfl_xor_sync(0xFFFFFFFFu, pmax, off));
            if (lane == 0) redi[warp] = pmax;
        }
        __syncthreads();
        tc_fence_after();
        tbase = have_tmem ? *tmem_holder : 0u;
        long long pref = 0;
        if (rotate) {
            int top = redi[0];
#pragma unroll
            for (int w = 1; w < NW; ++w) top = max(top, redi[w]);
            pref = a.p_ref ? (long long)a.p_ref[id.b] : (long long)top + 1;
        }
        // lane covers frequencies f0..f0+7 of the row handled by its group of eight lanes
        const int grp = lane >> 3, f0 = (lane & 7) * 8;
        // spacing of rows 16 slots apart at the newest end of the event: what a token-by-token cache has everywhere
        const long long D16 = n > 16 ? (long long)spos[n - 1] - (long long)spos[n - 17] : 0;
        ChainScore cs;
        cs.set_step(D16, phitab + f0, sect);
        // whether every row sits D16 after the row 16 slots before it (found once; the chains then need no look at
        // the positions)
        bool uni = true;
        for (int j = 16 + tid; j < n; j += NT) uni &= (long long)spos[j] - (long long)spos[j - 16] == D16;
        const bool uniform = __syncthreads_and(uni);
        // A lane group scores two rows side by side, so that one's dependent arithmetic fills the other's latency: a row of each chain (see
        // score_steps), or, with four of the eight warps on a chain each, a row and the next one of the same chain.
        const int row = 4 * (warp & 3) + grp;
        auto spaced = [&](int j) { return j >= n || (long long)spos[j] - (long long)spos[j - 16] == D16; };
        timeout = !mbar_wait_bounded(barK, 0, a.wait_polls);
        phase_stamp(id.e, 10);  // (K rows have arrived)
        {
            ChainScore cb;
            AKV_PHASE_ACC_DECL(cyc_anchor);
#pragma unroll 1
            for (int i = 0; i < steps; i += WIDE ? 2 : 1) {
                const int ja = 16 * i + row + (WIDE ? (warp >> 2) * second : 0), jb = ja + (WIDE ? 16 : second);
                const bool la = ja < n, lb = jb < n && (!WIDE || i + 1 < steps);
                if (FOUR && n_late > 0) {
                    if (i == kLateSteps) {   // the slots are free
                        __syncthreads();
                        if (tid == 0) {
                            mbar_expect_tx(barL, (uint32_t)n_late * 256u);
                            request_k_rows(late0, second, 0, barL);
                            request_k_rows(second + late0, n, kChainSlots, barL);
                        }
                    }
                    if (i == steps - kLateSteps) timeout |= !mbar_wait_bounded(barL, 0, a.wait_polls);
                }
                // each chain on its own: after an event the kept rows' positions are irregular (fresh rotation every
                // step) while the rows appended since are consecutive (chained)
                bool fa = i == 0 || a.no_chain, fb = WIDE ? a.no_chain != 0 : fa;
                if (!(WIDE ? fb : fa) && !uniform) {
                    if (!WIDE || i > 0) fa = !__all_sync(0xFFFFFFFFu, spaced(ja));
                    fb = !__all_sync(0xFFFFFFFFu, spaced(jb));
                }
                AKV_PHASE_ACC_BEGIN(cyc_anchor);
                if (fa) {
                    if (la) cs.anchor(pref - (long long)spos[ja], gtab + f0, phitab + f0, sect);
                } else {
                    if (WIDE) cs.turn_to(cb);
                    cs.advance();
                }
                if (fb) {
                    if (lb) cb.anchor(pref - (long long)spos[jb], gtab + f0, phitab + f0, sect);
                } else {
                    if (WIDE) cb.turn_to(cs);
                    cb.advance_by(cs);
                }
                AKV_PHASE_ACC_END(cyc_anchor);
                float acca = 0.f, accb = 0.f;
                if (la) {
                    const unsigned char* krow = tile + (FOUR && n_late > 0 ? ja + late_slot_shift(i, steps, 0) : ja) * 256 + (lane & 7) * 16;
                    acca = cs.dot(*reinterpret_cast<const uint4*>(krow), *reinterpret_cast<const uint4*>(krow + 128));
                }
                if (lb) {
                    const unsigned char* krow = tile + (FOUR && n_late > 0 ? jb + late_slot_shift(i, steps, 1) : jb) * 256 + (lane & 7) * 16;
                    accb = cb.dot(*reinterpret_cast<const uint4*>(krow), *reinterpret_cast<const uint4*>(krow + 128));
                }
#pragma unroll
                for (int off = 4; off > 0; off >>= 1) {
                    acca += __shfl_xor_sync(0xFFFFFFFFu, acca, off);
                    accb += __shfl_xor_sync(0xFFFFFFFFu, accb, off);
                }
                if ((lane & 7) == 0) {
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        const int j = h ? jb : ja;
                        const float acc = h ? accb : acca;
                        if (h ? lb : la) {
                            if (a.scores) a.scores[(long long)id.e * N + j] = acc;
                            const bool fin = isfinite(acc);
                            bad |= !fin;
                            const float sj = fin ? acc : -INFINITY;
                            s[j] = sj;
                            key[j] = orderable(sj);
                        }
                    }
                }
            }
            AKV_PHASE_ACC_STORE(id.e, 11, cyc_anchor);
            phase_stamp(id.e, 12);  // (scoring loop left)
        }
    } else {
        for (int j = tid; j < n; j += NT) {
            const float sc = a.scores[(long long)id.e * N + j];
            const bool fin = isfinite(sc);
            bad |= !fin;
            const float sj = fin ? sc : -INFINITY;
            s[j] = sj;
            key[j] = orderable(sj);
        }
    }
    for (int j = n + tid; j < np4; j += NT) key[j] = 0u;  // below every real key
    timeout = __syncthreads_or(timeout);
    if (timeout) {
        if (tid == 0 && a.status) a.status[id.e] = 3;
        mbar_wait_bounded(barK, 0, a.wait_polls);  // give copies still in flight another bounded chance to land
        if (n_late > 0) mbar_wait_bounded(barL, 0, a.wait_polls);
        if (have_tmem && warp == 0) tmem_dealloc(tbase, kPoolCols);
        return;
    }
    bad = __syncthreads_or(bad);
    // (only now: while scoring, this storage holds the statistic's table, which slower warps may still read)
    if (!WIDE && tid < 8) kept[tid] = 0u;

    phase_stamp(id.e, 2);
    // ---- s_(b) by bisection over the score keys, then the pool in slot order (warp 0) -------------
    if constexpr (WIDE) {
        // A key per thread, counts by the barrier itself: a bit per round. (One warp with eight keys per lane: 3.7 thousand cycles
        // of an event, these 3.3.)
        const uint32_t kj = tid < np4 ? key[tid] : 0u;
        uint32_t kb = 0u;
        if (picks > 0)
            for (int lo = 31; lo >= (similarity ? 14 : 0); --lo)
                if (__syncthreads_count(kj >= (kb | (1u << lo))) >= picks) kb |= 1u << lo;
        const float sb = from_orderable(kb);
        const float thr = a.no_prune || kb < 0x00800000u ? -INFINITY : fmaf(-1.001f, a.lam, sb) - 1e-6f * fabsf(sb);
        const bool pooled = kj != 0u && !(from_orderable(kj) < thr);
        ActiveBound bound{0u, 0};
        if (similarity && __syncthreads_count(pooled) > a.active)
            bound = active_bound(orderable(thr), kb, a.active, a.active + 1, a.active - a.active / 8, [&](uint32_t v1, uint32_t v2, uint32_t v3, int& c1, int& c2, int& c3) {
                c1 = __syncthreads_count(kj >= v1);
                c2 = __syncthreads_count(kj >= v2);
                c3 = __syncthreads_count(kj >= v3);
            });
        if (tid == 0) {
            *tie_holder = 0;
            *bound_holder = bound.key;
            *thr_holder = thr;
        }
        if (bound.ties) {
            __syncthreads();
            if (warp == 0) {
                const int base = list_with_ties(key, np4, bound.key, bound.ties, bypool, tie_holder);
                if (lane == 0) *pool_holder = base;
            }
        } else {
            // in slot order: a bit per slot, a row's place is the number of bits below
            const bool in = similarity ? pooled && kj > bound.key : kj != 0u && kj >= kb;
            const uint32_t mask = __ballot_sync(0xFFFFFFFFu, in);
            if (lane == 0) kept[warp] = mask;
            __syncthreads();
            if (in) bypool[kept_below(kept, tid)] = (unsigned short)tid;
            if (tid == 0) {
                int base = 0;
#pragma unroll
                for (int w = 0; w < NW; ++w) base += __popc(kept[w]);
                *pool_holder = base;
            }
        }
    } else if (warp == 0) {
        uint32_t kk[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int j = lane + 32 * k;
            kk[k] = j < np4 ? key[j] : 0u;
        }
        uint32_t kb = 0u;  // the picks-th largest key: the largest v with at least `picks` keys >= v
        if (picks > 0) {
            // two bits per round: the three counts are independent, so their reductions overlap.
            // Pruning only needs a lower bound of s_(b) (the pool may be a little larger than necessary),
            // so the low 14 key bits (0.2 % of the value) are not resolved; top-k needs the exact key.
            const int lo_end = similarity ? 14 : 0;
            for (int lo = 30; lo >= lo_end; lo -= 2) {
                const uint32_t v1 = kb | (1u << lo), v2 = kb | (2u << lo), v3 = kb | (3u << lo);
                int c1 = 0, c2 = 0, c3 = 0;
#pragma unroll
                for (int k = 0; k < 8; ++k) {
                    c1 += kk[k] >= v1;
                    c2 += kk[k] >= v2;
                    c3 += kk[k] >= v3;
                }
                c1 = __reduce_add_sync(0xFFFFFFFFu, c1);
                c2 = __reduce_add_sync(0xFFFFFFFFu, c2);
                c3 = __reduce_add_sync(0xFFFFFFFFu, c3);
                kb = c3 >= picks ? v3 : (c2 >= picks ? v2 : (c1 >= picks ? v1 : kb));
            }
        }
        const float sb = from_orderable(kb);
        // -inf keeps everyone (also where kb, whose low bits are open, is below every finite value's key)
        const float thr = a.no_prune || kb < 0x00800000u ? -INFINITY : fmaf(-1.001f, a.lam, sb) - 1e-6f * fabsf(sb);
        // Active set: the pool's best-scored rows, at most a.active of them; no key left out is above bound.key (0: none
        // is left out). A candidate's Eq. 2 value never exceeds its score: the loop over the active set is exact as long as
        // its winning value stays above the bound (it nearly always does: with lambda = 0.5 the picks reach a few ranks
        // beyond the budget).
        ActiveBound bound{0u, 0};
        if (similarity) {
            int pool_size = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) pool_size += kk[k] != 0u && !(from_orderable(kk[k]) < thr);
            pool_size = __reduce_add_sync(0xFFFFFFFFu, pool_size);
            if (pool_size > a.active) bound = warp_active_bound(kk, orderable(thr), kb, a.active);
        }
        int base = 0;
        if (lane == 0) *tie_holder = 0;
        __syncwarp();
        if (bound.ties) {
            base = list_with_ties(key, np4, bound.key, bound.ties, bypool, tie_holder);
        } else {
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const bool in = kk[k] != 0u && (similarity ? !(from_orderable(kk[k]) < thr) && kk[k] > bound.key : kk[k] >= kb);
                const uint32_t mask = __ballot_sync(0xFFFFFFFFu, in);
                if (in) bypool[base + __popc(mask & ((1u << lane) - 1u))] = (unsigned short)(lane + 32 * k);
                base += __popc(mask);
            }
        }
        if (lane == 0) {
            *pool_holder = base;
            *bound_holder = bound.key;
            *thr_holder = thr;
        }
    }
    __syncthreads();  // every key has been read: its storage becomes r below
    if (WIDE && tid < 8) kept[tid] = 0u;   // (the pool's bits until now)
    const int P = *pool_holder;

    phase_stamp(id.e, 3);
    // ---- V rows of the pool as the swizzled operand tile ---------------------------------------------
    if (similarity && G) {
        // the active set's cosine matrix, gathered from the shared one: row a of the triangle holds the shared
        // matrix's row of slot a at the slots of rows 0..a; the signatures are unit rows, so there are no norms
        // (a warp per row, its lanes across the row's columns: a lane's columns are the same for every row, so it
        // keeps their slots in registers). Asynchronous 4-byte copies straight into the triangle: nothing waits until all of a
        // warp's rows are under way (1792 events of 256 rows to 128: 18.1 thousand cycles of an event with the loads through registers,
        // four rows at a time, 10.4 thousand so; the call with signatures and matrix 297 -> 271 us).
        int col[Shape::kCpl];
#pragma unroll
        for (int k = 0; k < Shape::kCpl; ++k) col[k] = lane + 32 * k < P ? bypool[lane + 32 * k] : 0;
        for (int ra = warp; ra < P; ra += NT / 32) {
            const float* grow = G + (long long)bypool[ra] * N;
            const uint32_t dst = tile_u32 + 4u * (uint32_t)(tri_row(ra) + lane);
#pragma unroll
            for (int k = 0; k < Shape::kCpl; ++k)
                if (lane + 32 * k <= ra) cp_async4(dst + 128u * (uint32_t)k, grow + col[k]);
        }
        cp_async_wait_all();
        for (int ra = tid; ra < P; ra += NT) r[ra] = 1.f;
    } else if (similarity) {
        // thread -> 16-byte column c of rows r0, r0 + 8 or 16, ...: the swizzle term (c ^ row) & 7 is the same for
        // all of them, so a row costs one pool lookup, one address and one copy
        const int c = tid & 15, r0 = tid >> 4;
        const uint32_t dst0 = tile_u32 + tile_chunk(r0, c, half_bytes);
        if (dense) {
            const __nv_bfloat16* vcol = Vg + ev_off + c * 8;
            for (int rho = r0; rho < P; rho += NT / 16)
                cp_async16(dst0 + (uint32_t)(rho - r0) * 128u, vcol + (long long)bypool[rho] * lay.sn);
        } else {
            for (int rho = r0; rho < P; rho += NT / 16)
                cp_async16(dst0 + (uint32_t)(rho - r0) * 128u, Vg + rowoff(bypool[rho]) + c * 8);
        }

        cp_async_wait_all();
        fence_proxy_async();
        tc_fence_before();
        __syncthreads();
        tc_fence_after();
    }
    phase_stamp(id.e, 4);
    // rows from 128 on (nb of them): a second product, the last 128 rows of the operand against those
    // rows, gives their cosines against one another; what lies left of column 128 comes from the first product
    // by symmetry
    const bool product = similarity && !G;  // the cosine matrix comes off the tensor core
    const int nb = (product && P > 128) ? P - 128 : 0;
    const int ncols = max((P + 15) & ~15, 16), base2 = ncols - 128;   // (a shape with no columns is not allowed)
    if (product) {
        if (tid == 0 && (FUSED || !a.starve)) {
            tc_fence_after();
            const uint32_t idesc = umma_idesc_bf16(128, ncols);
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                const uint32_t koff = (uint32_t)(kk >> 2) * half_bytes + (uint32_t)(kk & 3) * 32u;
                umma_bf16(tbase, umma_desc_sw128(tile_u32 + koff), umma_desc_sw128(tile_u32 + koff), idesc, kk > 0 ? 1u : 0u);
            }
            if (nb > 0) {
                const uint32_t idesc2 = umma_idesc_bf16(128, ncols - 128);
#pragma unroll
                for (int kk = 0; kk < 8; ++kk) {
                    const uint32_t koff = (uint32_t)(kk >> 2) * half_bytes + (uint32_t)(kk & 3) * 32u;
                    umma_bf16(tbase + (uint32_t)ncols, umma_desc_sw128(tile_u32 + (uint32_t)base2 * 128u + koff),
                              umma_desc_sw128(tile_u32 + 128u * 128u + koff), idesc2, kk > 0 ? 1u : 0u);
                }
            }
            umma_commit(barM);
        }
        timeout = !mbar_wait_bounded(barM, 0, a.wait_polls);
        tc_fence_after();
    }
    timeout = __syncthreads_or(timeout);  // also: the product has read the whole tile before the triangle lands on it
    if (timeout) {
        if (tid == 0 && a.status) a.status[id.e] = 3;
        if (!FUSED) select_gave_up(a, id.e, NT);
        if (have_tmem && warp == 0) tmem_dealloc(tbase, kPoolCols);
        return;
    }
    phase_stamp(id.e, 5);
    if (product) {
        // lower triangle -> shared memory; row rho = 32 warp + lane needs columns 0..rho
        // (eight warps: the second four take the rows from 128 on)
        const int quarter = warp & 3, rho = 32 * quarter + lane;
        const uint32_t lanes = tbase + ((uint32_t)(32 * quarter) << 16);
        if (warp < 4 && 32 * quarter < P) {
            const int trow = tri_row(rho);
            // column blocks left of the diagonal one: every column is below the row
            for (int cb = 0; cb < quarter; ++cb) {
                uint32_t v[32];
                tmem_ld32(lanes + (uint32_t)(32 * cb), v);
                tmem_ld_wait();
                if (rho < P) {
#pragma unroll
                    for (int k = 0; k < 32; ++k) tri[trow + 32 * cb + k] = __uint_as_float(v[k]);
                }
            }
            // the diagonal block: columns up to the row itself, whose last entry is the squared norm
            {
                uint32_t v[32];
                tmem_ld32(lanes + (uint32_t)(32 * quarter), v);
                tmem_ld_wait();
                if (rho < P) {
#pragma unroll
                    for (int k = 0; k < 32; ++k)
                        if (k <= lane) tri[trow + 32 * quarter + k] = __uint_as_float(v[k]);
                    r[rho] = 1.f / (sqrtf(tri[trow + rho]) + a.eps);  // read back: this thread stored it
                }
            }
        }
        if (nb > 0 && (!WIDE || warp >= 4)) {
            // rows from 128 on. Left of column 128: row a's entry in column b is row b's entry in column a (every
            // thread moves its own row's columns 128..). From column 128 on: the second product, whose lane L holds
            // row base2 + L against rows 128.. in the columns after the first product's.
            for (int cb = 0; cb < (nb + 31) >> 5; ++cb) {
                uint32_t v[32];
                tmem_ld32(lanes + 128u + (uint32_t)(32 * cb), v);
                tmem_ld_wait();
#pragma unroll
                for (int k = 0; k < 32; ++k)
                    if (32 * cb + k < nb) tri[tri_row(128 + 32 * cb + k) + rho] = __uint_as_float(v[k]);
            }
            const int ra = base2 + rho - 128;  // this thread's row of the second product, counted from row 128
            float diag = 0.f;                  // its squared norm (one square root and one division per thread, after the loop)
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
            if (ra >= 0 && ra < nb) r[128 + ra] = 1.f / (sqrtf(diag) + a.eps);
        }
    }
    tc_fence_before();
    __syncthreads();
    if (have_tmem && warp == 0) tmem_dealloc(tbase, kPoolCols);

    phase_stamp(id.e, 6);
    // ---- Algorithm 1 in warp 0 -------------------------------------------------------------------------
    // The winning key of every pick is parked in gain[] and its pool row in order[]; both are decoded
    // after the loop.
    uint32_t* park_key = reinterpret_cast<uint32_t*>(gain);
    if (!similarity) {
        picks_by_rank<NT>(tid, P, picks, key, bypool, park_key, order);
    } else {
        if (warp == 0) {
            float* m_act = reinterpret_cast<float*>(tile + kContMact);
            const uint32_t bound = *bound_holder;
            bool ok;
            // (eight picks per look at the bound instead of four: 16 384 events of 256 rows to 128 1645 -> 1626 us, 448 of them 76.8 -> 74.7)
            if constexpr (!WIDE)
                ok = picks_cosine<Shape::kCpl, true, 8>(lane, P, picks, s, bypool, r, a.lam, tri, park_key, order, bound, m_act, redi, nullptr, tie_holder);
            else if (P <= 128)
                ok = picks_in_pairs<4, true>(lane, P, picks, s, bypool, r, a.lam, tri, park_key, order, bound, m_act, redi, nullptr, tie_holder);
            else
                ok = picks_in_pairs<Shape::kCpl, true>(lane, P, picks, s, bypool, r, a.lam, tri, park_key, order, bound, m_act, redi, nullptr, tie_holder);
            if (lane == 0) *pick_holder = ok ? picks : *redi;
        }
        __syncthreads();
        if (*pick_holder < picks) {
            picks_over_whole_pool<FORM, NT>(a, smem, n, P, picks, *pick_holder);
        }
    }
    __syncthreads();
    int mine = -1;   // the slot of this thread's pick (a budget is at most the threads)
    if (tid < picks) {
        mine = bypool[order[tid]];
        atomicOr(&kept[mine >> 5], 1u << (mine & 31));
    }
    __syncthreads();

    phase_stamp(id.e, 7);
    // ---- sort(S) and outputs -------------------------------------------------------------------------
    const long long ob = (long long)id.e * a.budget;
    if (tid < picks) idx[kept_below(kept, mine)] = mine;
    else if (tid < a.budget) idx[tid] = -1;
    if (tid < a.budget) {
        if (a.pick_order) a.pick_order[ob + tid] = mine;
        if (a.pick_gain) a.pick_gain[ob + tid] = tid < picks ? from_orderable(park_key[tid]) : 0.f;
    }
    __syncthreads();
    if (tid < a.budget) a.idx_sorted[ob + tid] = idx[tid];
    if (tid == 0) {
        if (a.n_kept) a.n_kept[id.e] = picks;
        if (a.status) a.status[id.e] = n < bud ? 2 : (bad ? 1 : 0);
    }
    if (!FUSED) return;

    phase_stamp(id.e, 8);
    // ---- compaction in place ----------------------------------------------------------------------
    // Every kept K and V row and position is on chip before the first store: a destination slot can be
    // another kept row's source. Up to 64 rows: K in registers, V through the (by now free) tile by
    // cp.async, one barrier. Both in registers would make this the kernel's register peak and cost a
    // resident CTA per SM.
    int* wpos = a.pos.p ? a.pos.p + id.b * a.pos.sb + id.l * a.pos.sl + id.h * a.pos.sh : nullptr;
    if (picks <= 64) {
        // thread -> 16-byte column c of kept rows r0, r0 + 8 or 16, ...
        const int c = tid & 15, r0 = tid >> 4;
        const uint32_t slot0 = (uint32_t)(r0 * 256 + c * 16);
        const long long col = (dense ? ev_off : 0) + c * 8;
        for (int t = r0; t < picks; t += NT / 16) {
            const long long off = col + (dense ? (long long)idx[t] * lay.sn : rowoff(idx[t]));
            cp_async16(tile_u32 + slot0 + (uint32_t)(t - r0) * 256u, Kg + off);
            cp_async16(tile_u32 + 16384u + slot0 + (uint32_t)(t - r0) * 256u, Vg + off);
        }
        cp_async_wait_all();
        __syncthreads();  // every load above has been performed
        for (int t = r0; t < picks; t += NT / 16) {
            const long long off = col + (dense ? (long long)t * lay.sn : rowoff(t));
            const unsigned char* src = tile + slot0 + (t - r0) * 256;
            *reinterpret_cast<uint4*>(Kg + off) = *reinterpret_cast<const uint4*>(src);
            *reinterpret_cast<uint4*>(Vg + off) = *reinterpret_cast<const uint4*>(src + 16384);
        }
    } else {
        // The tile holds the kept rows of K and of V side by side: one round of 16-byte gathers, one barrier. (With four CTAs per
        // SM the last V rows that do not fit there wait in registers.)
        // Stores: slots 0..picks-1 are contiguous in a dense cache (and page by page in a paged one), so one
        // thread writes them back with a few bulk copies. (Gathering by one bulk copy per row measured slower.)
        constexpr uint32_t vhalf = 32768u;
        constexpr int kFit = (int)((Shape::kTile - vhalf) / 256u) < 128 ? (int)((Shape::kTile - vhalf) / 256u) : 128;
        constexpr int kHeld = ((128 - kFit) * 16 + NT - 1) / NT;
        const int fit = min(picks, kFit);
        auto gather = [&](int x, bool v) {
            const long long off = rowoff(idx[x >> 4]) + (x & 15) * 8;
            cp_async16(tile_u32 + (uint32_t)x * 16u, Kg + off);
            if (v) cp_async16(tile_u32 + vhalf + (uint32_t)x * 16u, Vg + off);
        };
        if constexpr (WIDE) {
            for (int x = tid; x < picks * 16; x += NT) gather(x, true);
        } else {
#pragma unroll 4
            for (int x = tid; x < picks * 16; x += NT) gather(x, !FOUR || x < fit * 16);   // (several rows' look-ups at once; with one event per SM no gain)
        }
        uint4 held[kHeld > 0 ? kHeld : 1];
#pragma unroll
        for (int i = 0; i < kHeld; ++i) {
            const int x = fit * 16 + tid + i * NT;
            held[i] = x < picks * 16 ? *reinterpret_cast<const uint4*>(Vg + rowoff(idx[x >> 4]) + (x & 15) * 8) : make_uint4(0u, 0u, 0u, 0u);
        }
        cp_async_wait_all();
        fence_proxy_async();  // the bulk stores below read what these copies wrote
        // every kept row is on chip before the first store (those in registers too: the barrier's operand depends on them)
        if constexpr (kHeld > 0) {
            uint32_t arrived = 0u;
#pragma unroll
            for (int i = 0; i < kHeld; ++i) arrived |= held[i].x | held[i].w;
            __syncthreads_or(arrived == 0x7FC07FC1u);
        } else {
            __syncthreads();
        }
        const bool runs = dense ? lay.sn == kTcD : lay.s_page_n == kTcD;
        if (runs) {
            if (tid == 0) {
                for (int row = 0; row < picks;) {
                    const int run = dense ? picks - row : min(picks - row, lay.page_size - (row & (lay.page_size - 1)));
                    const long long off = rowoff(row);
                    const int vrun = min(run, fit - row);
                    bulk_s2g(Kg + off, tile_u32 + (uint32_t)row * 256u, (uint32_t)run * 256u);
                    if (!FOUR || vrun > 0) bulk_s2g(Vg + off, tile_u32 + vhalf + (uint32_t)row * 256u, (uint32_t)vrun * 256u);
                    row += run;
                }
                bulk_store_wait_read();  // shared memory is read out before the CTA may leave
            }
        } else {
            for (int x = tid; x < picks * 16; x += NT) {
                const long long off = rowoff(x >> 4) + (x & 15) * 8;
                copy16(reinterpret_cast<char*>(Kg + off), tile + x * 16);
                if (!FOUR || x < fit * 16) copy16(reinterpret_cast<char*>(Vg + off), tile + vhalf + x * 16);
            }
        }
#pragma unroll
        for (int i = 0; i < kHeld; ++i) {
            const int x = fit * 16 + tid + i * NT;
            if (x < picks * 16) *reinterpret_cast<uint4*>(Vg + rowoff(x >> 4) + (x & 15) * 8) = held[i];
        }
    }
    if (wpos)
        for (int t = tid; t < picks; t += NT) wpos[t] = spos[idx[t]];
    phase_stamp(id.e, 9);
}

}  // namespace akv
