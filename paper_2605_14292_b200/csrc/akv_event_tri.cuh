// Fast event kernel for bf16, d = 128, per-head signatures, N <= 256, used when the pool that
// survives pruning is expected to stay within 127 rows (N <= 128 or budget <= 64). One CTA of four
// warps per event, six CTAs resident per SM (37 KB of shared memory and 80 registers each).
//
//   1. K rows arrive in shared memory by bulk copies (cp.async.bulk + mbarrier) and are scored there
//      (fused RoPE rotate-and-dot against the folded query statistic). The tile holds 128 rows: rows
//      from 128 on arrive later, in the slots of the first rows once those have been scored.
//   2. Only candidates with  s_i >= s_(b) - lambda * (1 + slack)  can ever be an argmax of Eq. 2
//      (the running maximum m never exceeds 1, so every still unchosen member of the top-b scores
//      beats the others). s_(b) comes from a bisection over the score keys; that pool of P rows,
//      in slot order, is the only part of V that is read for the selection.
//      A pool of more than 127 rows (a strong penalty) is cut to its best-scored ones, the active set (112 to 127 rows);
//      no candidate left out scores above `bound`, so the loop is exact while its winning values stay above that, and
//      the rare event where one does not is finished by picks_over_whole_pool.
//   3. The pool's V rows form a K-major, 128-byte-swizzled operand tile, one
//      tcgen05.mma sequence writes the pool's cosine matrix (raw dot products, fp32) into tensor
//      memory, and the four warps move its lower triangle to shared memory (tcgen05.ld), taking
//      the squared norms of Eq. 1 from the diagonal on the way.
//   4. Algorithm 1 runs in ONE warp: every lane owns up to P/32 candidates and keeps s, the
//      running maximum and lambda/norm in registers; the argmax is two warp reductions, the picked
//      row of the cosine matrix is read from the triangle without bank conflicts.
//   5. Kept rows are written back in place: K and V rows are re-read (L2) into the tile, which is
//      free by then, and stored after a barrier; positions come from their shared-memory copy.
#pragma once
#include "akv_active_set.cuh"
#include "akv_event_tc.cuh"
#include "akv_pages.cuh"

namespace akv {

constexpr int kTriTileRows = 128;           // K rows resident at a time = rows of the V operand tile
constexpr unsigned kTriTileBytes = 32768u;  // 128 rows of 256 bytes; holds the triangle of up to 127 rows
constexpr int kTriMaxPool = 127;            // largest pool whose cosine matrix goes through the tile

struct TriSmem {
    unsigned tile, s, key, spos, bypool, taken, order, gain, idx, sect, misc, pages, total;   // taken: a flag per slot, or (event_pool_kernel) a bit
};
// Layout after the 1024-byte aligned base. `key` (score keys) and `r` (reciprocal norms) share storage.
constexpr int kPageOffsets = 16;   // pages of an event whose offsets are kept on chip
__host__ __device__ inline TriSmem plan_event_smem(int N, int budget, unsigned tile_bytes, bool paged, unsigned taken_bytes) {
    TriSmem p;
    const unsigned np = (unsigned)((N + 3) & ~3);
    unsigned o = 0;
    p.tile = o;   o += tile_bytes;
    p.s = o;      o += align16(np * 4);
    p.key = o;    o += align16(np * 4);
    p.spos = o;   o += align16(np * 4);
    p.bypool = o; o += align16(np * 2);
    p.taken = o;  o += align16(taken_bytes);
    p.order = o;  o += align16((unsigned)budget * 4);
    p.gain = o;   o += align16((unsigned)budget * 4);
    p.idx = o;    o += align16((unsigned)budget * 4);
    if (o - p.bypool < 1024u) o = p.bypool + 1024u;  // bypool..idx also hold the folded statistic and the phase steps (1 KB) while scoring
    p.sect = o;   o += 256;       // cosine and sine of the 32 sector angles
    p.misc = o;   o += 64;        // mbarriers (K, product, late K rows), tmem base, pool size, bound, threshold, block-max scratch
    p.pages = o;  o += paged ? 8 * kPageOffsets : 0;
    p.total = o + 1024;           // room to align the base to 1024 bytes
    return p;
}
__host__ __device__ inline TriSmem plan_tri_smem(int N, int budget, bool paged) { return plan_event_smem(N, budget, kTriTileBytes, paged, N < 32 ? 32u : (unsigned)((N + 3) & ~3)); }

// event_pool_kernel's (akv_event_pool.cuh) forms: how many of an event's rows a CTA has on chip, and with how many threads.
enum PoolForm { kPoolThree, kPoolWideForm, kPoolFour };
constexpr uint32_t kPoolCols = 256u;        // tensor-memory columns (a power of two >= the matrix's columns)
constexpr int kPoolWide = 256;              // threads of a CTA that has an SM to itself
template <int FORM>
struct PoolShape {
    // a whole event's K rows, then the triangle of an active set of up to 180 rows; three CTAs per SM, or two of eight warps (a call
    // puts one on an SM, but calls in other streams come beside it: with registers for one only, two streams with 112 events of 256 rows
    // to 128 in pages each took 63 us instead of 41, four 121 instead of 74; for three, one such call alone took 41 instead of 33)
    static constexpr int kThreads = FORM == kPoolWideForm ? kPoolWide : kTcThreads, kCtas = FORM == kPoolWideForm ? 2 : 3;
    static constexpr unsigned kTile = 65536u;
    static constexpr int kActive = 180, kCpl = 6, kRows = 256, kOperandRows = 256;
};
template <>
struct PoolShape<kPoolFour> {
    // 192 K rows (the others arrive in the slots of the first, see late_slot_shift), then the triangle of up to 158 rows; four CTAs per SM: 57 312 bytes for
    // 256 rows in pages to 128, of the 57 344 that four leave each
    static constexpr int kThreads = kTcThreads, kCtas = 4;
    static constexpr unsigned kTile = 50688u;
    static constexpr int kActive = 158, kCpl = 5, kRows = 192, kOperandRows = 160;
};
template <int FORM>
__host__ __device__ inline TriSmem plan_pool_event_smem(int N, int budget, bool paged) { return plan_event_smem(N, budget, PoolShape<FORM>::kTile, paged, 32u); }

// 32 consecutive columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
        "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
          "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
          "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
          "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
        : "r"(taddr)
        : "memory");
}

// entry (a, b), a >= b, of a lower triangle stored row by row; rows a = lane + 32 k of one warp
// fall into 32 different banks for a fixed b, and so do consecutive b for a fixed a
__device__ __forceinline__ int tri_row(int a) { return (a * (a + 1)) >> 1; }

// Per-lane state of the single-warp greedy loop: candidates rho = lane + 32 k, k < CPL.
template <int CPL>
struct GreedyLane {
    float sv[CPL], lr[CPL], M[CPL];
    uint32_t am[CPL];  // all ones while the candidate competes; 0 once chosen, or when the row is empty
    __device__ __forceinline__ void init(int lane, int P, const float* s, const unsigned short* bypool, const float* r, float lam,
                                         bool use_r) {
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const int rho = lane + 32 * k;
            sv[k] = 0.f; lr[k] = 0.f; M[k] = 0.f; am[k] = 0u;
            if (rho < P) {
                sv[k] = s[bypool[rho]];
                lr[k] = use_r ? penalty_rate(lam, r[rho]) : 0.f;
                am[k] = 0xFFFFFFFFu;
            }
        }
    }
    // a = s - lambda m over the candidates still competing; returns the key of the best one and its
    // pool row (ties to the lower row, which is the lower slot) and retires it
    __device__ __forceinline__ int pick(int lane, uint32_t& best_key) {
        uint32_t key[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            const uint32_t u = __float_as_uint(fmaf(-lr[k], M[k], sv[k]));
            key[k] = (u ^ ((uint32_t)((int32_t)u >> 31) | 0x80000000u)) & am[k];  // orderable(a), 0 when retired
        }
        uint32_t bk = key[0];
#pragma unroll
        for (int k = 1; k < CPL; ++k) bk = max(bk, key[k]);
        const uint32_t whi = __reduce_max_sync(0xFFFFFFFFu, bk);
        // lowest row among the candidates that reach the maximum (0xFFFF - row, so that max picks the lowest)
        uint32_t cand = 0u;
#pragma unroll
        for (int k = 0; k < CPL; ++k) cand = max(cand, key[k] == whi ? 0xFFFFu - (uint32_t)(lane + 32 * k) : 0u);
        const uint32_t wlo = __reduce_max_sync(0xFFFFFFFFu, cand);
        const int irho = (int)(0xFFFFu - wlo);
#pragma unroll
        for (int k = 0; k < CPL; ++k) am[k] = (lane + 32 * k == irho) ? 0u : am[k];
        best_key = whi;
        return irho;
    }
};

// One float of shared memory, as a volatile load: a group of these is issued back to back and in
// program order, where plain loads get strung out one per use (a picked row's four entries cost four
// exposed latencies that way).
__device__ __forceinline__ float lds_in_order(uint32_t addr) {
    float v;
    asm volatile("ld.volatile.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr));
    return v;
}

// Top-k in pick order by the whole CTA: a row's place is the number of rows with a larger key (equal keys: lower row
// first). key: by slot; P: rows that reach the picks-th largest key.
template <int NT>
__device__ __forceinline__ void picks_by_rank(int tid, int P, int picks, const uint32_t* key, const unsigned short* bypool,
                                              uint32_t* park_key, int* park_row) {
    for (int rho = tid; rho < P; rho += NT) {
        const uint32_t mine = key[bypool[rho]];
        int rank = 0;
#pragma unroll 4
        for (int o = 0; o < P; ++o) {
            const uint32_t k = key[bypool[o]];
            rank += k > mine || (k == mine && o < rho);
        }
        if (rank < picks) {
            park_key[rank] = mine;
            park_row[rank] = rho;
        }
    }
}

// active_bound for a warp's keys (8 per lane, 0: no row). (A row fewer than the set could hold costs nothing; from an eighth
// fewer on the search goes on to the last bit.)
__device__ __forceinline__ ActiveBound warp_active_bound(const uint32_t (&kk)[8], uint32_t low, uint32_t kb, int cap) {
    return active_bound(low, kb, cap, cap + 1, cap - cap / 8, [&](uint32_t v1, uint32_t v2, uint32_t v3, int& c1, int& c2, int& c3) {
        c1 = c2 = c3 = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            c1 += kk[k] >= v1;
            c2 += kk[k] >= v2;
            c3 += kk[k] >= v3;
        }
        c1 = __reduce_add_sync(0xFFFFFFFFu, c1);
        c2 = __reduce_add_sync(0xFFFFFFFFu, c2);
        c3 = __reduce_add_sync(0xFFFFFFFFu, c3);
    });
}

// The active set in slot order where keys equal to its bound belong to it, by one warp: the keys above the bound and the
// `ties` lowest slots of those equal to it. Returns its size; *tie_slot: the lowest slot that equals the bound and is left
// out. Out of line: few events come here.
__device__ __noinline__ int list_with_ties(const uint32_t* key, int np4, uint32_t bound, int ties, unsigned short* bypool, int* tie_slot) {
    const int lane = threadIdx.x & 31;
    const uint32_t below = (1u << lane) - 1u;
    int base = 0, seen = 0;
    for (int j0 = 0; j0 < np4; j0 += 32) {
        const int j = j0 + lane;
        const uint32_t kj = j < np4 ? key[j] : 0u;
        const bool tie = kj == bound;
        const uint32_t tmask = __ballot_sync(0xFFFFFFFFu, tie);
        const int rank = seen + __popc(tmask & below);
        const bool in = kj > bound || (tie && rank < ties);
        const uint32_t mask = __ballot_sync(0xFFFFFFFFu, in);
        if (in) bypool[base + __popc(mask & below)] = (unsigned short)j;
        if (tie && rank == ties) *tie_slot = j;
        base += __popc(mask);
        seen += __popc(tmask);
    }
    return base;
}

// A kept slot's place in sorted order: the number of kept slots below it (a bit per slot in eight words). One step for all picks
// at once, where ordered_indices walks the slots in one warp: 1.36 instead of 1.78 thousand cycles of an event with 256 rows to
// 128, 16 384 of them 1994 -> 1966 us. (event_tri_kernel keeps flags: with this its registers no longer fit six CTAs per SM.)
__device__ __forceinline__ int kept_below(const uint32_t* kept, int slot) {
    const uint4 w0 = *reinterpret_cast<const uint4*>(kept), w1 = *reinterpret_cast<const uint4*>(kept + 4);
    const uint32_t w[8] = {w0.x, w0.y, w0.z, w0.w, w1.x, w1.y, w1.z, w1.w};
    int place = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int bits = slot - 32 * q;   // of this word, those below the slot
        place += __popc(bits >= 32 ? w[q] : bits > 0 ? w[q] & ((1u << bits) - 1u) : 0u);
    }
    return place;
}

// Warp-wide maximum of a float (sm_100a has the reduction for f32).
__device__ __forceinline__ float warp_max_f32(float v) {
    float m;
    asm volatile("redux.sync.max.f32 %0, %1, 0xffffffff;" : "=f"(m) : "f"(v));
    return m;
}

// A non-finite score competes as this value: below every real score, above a retired candidate's -inf.
constexpr float kLowestScore = -3.0e38f;

// Lowest pool row that is not among the t picked ones: what is taken when no candidate competes any more although
// picks are missing (cosines of infinite value rows).
__device__ __forceinline__ int lowest_free_row(const int* picked, int t) {
    int row = 0;
    for (int i = 0; i < t; ++i)
        if (picked[i] == row) { ++row; i = -1; }
    return row;
}

// The loop of Algorithm 1 with the cosine penalty, run by one warp over a lower triangle of raw dot products, Eq. 2
// evaluated and compared as floats. A candidate is retired through the triangle itself: the diagonal entries are set to
// +inf before the first pick, so the update m <- max(m, Sims[i, :]) gives the picked row m = +inf and a = -inf from then
// on: no mask, no per-candidate retirement. Winning values are parked as order-preserving keys, like the other loops'.
//
// One warp issues an instruction every 1.8 cycles at best, so what a pick costs is its instructions as much as its chain
// of two reductions and one load. Per candidate and pick: an fma, a max, a compare and a select to find the winner's row,
// two integer instructions for the address (an entry's index is max(tri_row(c) + i, tri_row(i) + c) whichever of c and i
// is the higher), a load, a product with the picked row's norm and a max. The row and its offset travel as one word. A
// branch on the winner costs 50 cycles, so the bound is looked at once per four picks or eight (winners only fall), and
// where it was reached those are taken again one by one. (Norms applied to the whole triangle beforehand instead: 5 cycles
// less a pick, but 2 to 6 thousand more for the triangle.)
//
// BOUNDED: the P rows are only the best-scored part of the pool, and every candidate left out scores at most
// `bound_key` (as an order-preserving key), so its Eq. 2 value can never exceed that. The loop is exact as long as the
// winning value stays above the bound, or equals it at a slot below *tie_slot (null: none), the lowest one of the candidates
// left out that may equal it; at the first pick that does not, it stops and returns false. The picks made so
// far stand; with m_out / t_out given the running maxima (by pool row; +inf for the rows already picked) and the number
// of picks are left for the caller to continue from. m_in: maxima to start from (null: 0). `tri` (its diagonal) and `r` are modified. At most 256 rows.
// kGroup: picks per look at the bound (divides 32).
template <int CPL, bool BOUNDED, int kGroup = 4>
__device__ __forceinline__ bool picks_cosine(int lane, int P, int picks, const float* s, const unsigned short* bypool, float* r, float lam,
                                             float* tri, uint32_t* park_key, int* park_row, uint32_t bound_key = 0u,
                                             float* m_out = nullptr, int* t_out = nullptr, const float* m_in = nullptr,
                                             const int* tie_slot = nullptr) {
    const uint32_t tb = smem_u32(tri), rb = smem_u32(r);
    const float ninf = __int_as_float(0xff800000), pinf = __int_as_float(0x7f800000);
    float sv[CPL], lr[CPL], M[CPL];
    int rc4[CPL], trow[CPL];   // 4 * row, and the shared-memory address of that row of the triangle
    uint32_t tag[CPL];         // the row's offset in the triangle and the row: the lower tag is the lower row
    const int last = max(P - 1, 0);
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        const int rho = lane + 32 * k;
        const bool in = rho < P;
        const int rc = min(rho, last);  // clamped: the loads stay inside the triangle, the loop needs no branch
        sv[k] = in ? fmaxf(s[bypool[rc]], kLowestScore) : ninf;
        M[k] = m_in && in ? m_in[rc] : 0.f;
        const float rk = fmaxf(r[rc], 1e-30f);   // positive, so that a maximum of +inf and a value of -inf come about
        lr[k] = in ? fmaxf(penalty_rate(lam, rk), 1e-30f) : 1.f;   // (finite: no value below is ever NaN, so a winner's row is always found)
        rc4[k] = 4 * rc;
        trow[k] = (int)(tb + 4u * (uint32_t)tri_row(rc));
        tag[k] = ((4u * (uint32_t)tri_row(rc)) << 8) | (uint32_t)rc;
        if (in) {
            tri[tri_row(rho) + rho] = pinf;
            r[rho] = rk;
        }
    }
    __syncwarp();
    const float bound = BOUNDED && bound_key ? from_orderable(bound_key) : ninf;
    // the winner: its value, its row and the row's offset (all lanes)
    auto winner = [&](float& whi, uint32_t& w) {
        float v[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) v[k] = fmaf(-lr[k], M[k], sv[k]);
        float lm = v[0];
#pragma unroll
        for (int k = 1; k < CPL; ++k) lm = fmaxf(lm, v[k]);
        whi = warp_max_f32(lm);
        uint32_t best = 0xFFFFFFFFu;
#pragma unroll
        for (int k = CPL - 1; k >= 0; --k) best = v[k] == whi ? tag[k] : best;
        w = __reduce_min_sync(0xFFFFFFFFu, best);
    };
    // m <- max(m, Sims[i, :])
    auto fold = [&](uint32_t w) {
        const int i4 = (int)((w & 255u) << 2), irow = (int)(tb + (w >> 8));
        const float ri = lds_in_order(rb + (uint32_t)i4);
        float x[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) x[k] = lds_in_order((uint32_t)__viaddmax_s32(trow[k], i4, irow + rc4[k]));
#pragma unroll
        for (int k = 0; k < CPL; ++k) M[k] = fmaxf(M[k], ri * x[k]);
    };
    for (int t0 = 0; t0 < picks; t0 += 32) {
        float my_val = 0.f;
        uint32_t my_row = 0u;
        const int t1 = min(t0 + 32, picks);
        bool at_bound = false;
        int t = t0;
#pragma unroll 1
        for (; t < t1 && !at_bound; t += kGroup) {
            float M0[CPL];
#pragma unroll
            for (int k = 0; k < CPL; ++k) M0[k] = M[k];
            float whi = 0.f;
#pragma unroll
            for (int u = 0; u < kGroup; ++u) {   // (picks beyond the last one are not parked)
                uint32_t w;
                winner(whi, w);
                const bool mine = lane == t + u - t0;
                my_val = mine ? whi : my_val;
                my_row = mine ? w & 255u : my_row;
                fold(w);
            }
            if (!(whi > bound)) {
                // one of the group, or one beyond the last pick, was not above the bound (or nothing is left to pick)
#pragma unroll
                for (int k = 0; k < CPL; ++k) M[k] = M0[k];
#pragma unroll 1
                for (int u = 0; u < kGroup && t < t1; ++u, ++t) {
                    uint32_t w;
                    winner(whi, w);
                    at_bound = !(whi > bound || (BOUNDED && tie_slot && whi == bound && whi > ninf && (int)bypool[w & 255u] < *tie_slot));
                    if (at_bound) break;
                    const bool mine = lane == t - t0;
                    my_val = mine ? whi : my_val;
                    my_row = mine ? w & 255u : my_row;
                    fold(w);
                }
                t -= kGroup;   // (the loop adds it)
            }
        }
        t = min(t, t1);
        if (t0 + lane < t) {
            park_key[t0 + lane] = orderable(my_val <= -2.9e38f ? ninf : my_val);
            park_row[t0 + lane] = (int)my_row;
        }
        if (at_bound) {
            __syncwarp();
            if (!BOUNDED || bound_key == 0u) {
                // no bound: every value left is -inf (cosines overflowed)
                if (lane == 0) {
                    for (; t < picks; ++t) {
                        park_key[t] = orderable(ninf);
                        park_row[t] = lowest_free_row(park_row, t);
                    }
                }
                return true;
            }
            if (m_out) {
#pragma unroll
                for (int k = 0; k < CPL; ++k)
                    if (lane + 32 * k < P) m_out[lane + 32 * k] = M[k];
            }
            if (t_out && lane == 0) *t_out = t;
            return false;
        }
    }
    return true;
}

// The same loop where few events share an SM and the chain of one pick after another counts more than its instructions. A step
// finds the best two candidates before either is folded in: the second is the next pick exactly if the first leaves its own maximum
// as it is, for all other values only fall (after t picks it does in all but one step of t, roughly); a step that finds it raised
// takes the first alone. 174 cycles a pick with six candidates per lane where picks_cosine takes 193, 160 with four where it takes 190, one event per SM;
// but about 1.1 times the instructions: with six of the small kernel's events per SM a call is 1 to 4 % slower for it, and in the
// prefill kernel 4 to 7 %. (Moving the candidates that are left to fewer per lane, with a loop for each number: slower everywhere,
// 22.3 -> 25.5 thousand cycles of an event alone on its SM, 358 -> 415 us for 896 events of 4096 rows: code that is not yet in the
// instruction caches costs more than the candidates saved.)
template <int CPL, bool BOUNDED>
__device__ __forceinline__ bool picks_in_pairs(int lane, int P, int picks, const float* s, const unsigned short* bypool, float* r, float lam,
                                               float* tri, uint32_t* park_key, int* park_row, uint32_t bound_key = 0u,
                                               float* m_out = nullptr, int* t_out = nullptr, const float* m_in = nullptr,
                                               const int* tie_slot = nullptr) {
    constexpr int kSteps = 2;   // steps per look at the bound
    const uint32_t tb = smem_u32(tri), rb = smem_u32(r);
    const float ninf = __int_as_float(0xff800000), pinf = __int_as_float(0x7f800000);
    float sv[CPL], lr[CPL], M[CPL];
    int rc4[CPL], trow[CPL];   // 4 * row, and the shared-memory address of that row of the triangle
    uint32_t tag[CPL];         // the row's offset in the triangle and the row: the lower tag is the lower row
    const int last = max(P - 1, 0);
#pragma unroll
    for (int k = 0; k < CPL; ++k) {
        const int rho = lane + 32 * k;
        const bool in = rho < P;
        const int rc = min(rho, last);  // clamped: the loads stay inside the triangle, the loop needs no branch
        sv[k] = in ? fmaxf(s[bypool[rc]], kLowestScore) : ninf;
        M[k] = m_in && in ? m_in[rc] : 0.f;
        const float rk = fmaxf(r[rc], 1e-30f);   // positive, so that a maximum of +inf and a value of -inf come about
        lr[k] = in ? fmaxf(penalty_rate(lam, rk), 1e-30f) : 1.f;   // (finite: no value below is ever NaN, so a winner's row is always found)
        rc4[k] = 4 * rc;
        trow[k] = (int)(tb + 4u * (uint32_t)tri_row(rc));
        tag[k] = ((4u * (uint32_t)tri_row(rc)) << 8) | (uint32_t)rc;
        if (in) {
            tri[tri_row(rho) + rho] = pinf;
            r[rho] = rk;
        }
    }
    __syncwarp();
    const float bound = BOUNDED && bound_key ? from_orderable(bound_key) : ninf;
    // the winner: its value, its row and the row's offset (all lanes)
    auto winner = [&](float& whi, uint32_t& w) {
        float v[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) v[k] = fmaf(-lr[k], M[k], sv[k]);
        float lm = v[0];
#pragma unroll
        for (int k = 1; k < CPL; ++k) lm = fmaxf(lm, v[k]);
        whi = warp_max_f32(lm);
        uint32_t best = 0xFFFFFFFFu;
#pragma unroll
        for (int k = CPL - 1; k >= 0; --k) best = v[k] == whi ? tag[k] : best;
        w = __reduce_min_sync(0xFFFFFFFFu, best);
    };
    // row i of the triangle at this lane's candidates, and its norm
    auto load_row = [&](uint32_t w, float& ri, float (&x)[CPL]) {
        const int i4 = (int)((w & 255u) << 2), irow = (int)(tb + (w >> 8));
        ri = lds_in_order(rb + (uint32_t)i4);
#pragma unroll
        for (int k = 0; k < CPL; ++k) x[k] = lds_in_order((uint32_t)__viaddmax_s32(trow[k], i4, irow + rc4[k]));
    };
    auto park = [&](int t, float val, uint32_t w) {
        park_key[t] = __float_as_uint(val);   // (as a key once the loop is left)
        park_row[t] = (int)(w & 255u);
    };
    // One pick, or two: the best two candidates are found before either is folded in. The second is the next pick exactly if
    // the first leaves its own maximum as it is, for all other values only fall. Returns the lowest value taken.
    auto step = [&](int& t) -> float {
        float v[CPL], u[CPL], x[CPL], y[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) v[k] = fmaf(-lr[k], M[k], sv[k]);
        float lm = v[0];
#pragma unroll
        for (int k = 1; k < CPL; ++k) lm = fmaxf(lm, v[k]);
        const float w1hi = warp_max_f32(lm);
        // the lane's best two (while the reduction is under way)
        uint32_t lt = tag[CPL - 1];
#pragma unroll
        for (int k = CPL - 2; k >= 0; --k) lt = v[k] == lm ? tag[k] : lt;
#pragma unroll
        for (int k = 0; k < CPL; ++k) u[k] = tag[k] == lt ? ninf : v[k];
        float lm2 = u[0];
#pragma unroll
        for (int k = 1; k < CPL; ++k) lm2 = fmaxf(lm2, u[k]);
        uint32_t lt2 = tag[CPL - 1];
#pragma unroll
        for (int k = CPL - 2; k >= 0; --k) lt2 = u[k] == lm2 ? tag[k] : lt2;
        const uint32_t w1 = __reduce_min_sync(0xFFFFFFFFu, lm == w1hi ? lt : 0xFFFFFFFFu);
        const bool own = lt == w1;
        const float lmB = own ? lm2 : lm;
        const uint32_t ltB = own ? lt2 : lt;
        const float w2hi = warp_max_f32(lmB);
        float ri, rj;
        load_row(w1, ri, x);
        const uint32_t w2 = __reduce_min_sync(0xFFFFFFFFu, lmB == w2hi ? ltB : 0xFFFFFFFFu);
        bool raised = false;   // the first raises the maximum of this lane's best other candidate
#pragma unroll
        for (int k = 0; k < CPL; ++k) {
            x[k] *= ri;
            raised |= tag[k] == ltB && x[k] > M[k];
        }
        load_row(w2, rj, y);
        const bool two = !__any_sync(0xFFFFFFFFu, ltB == w2 && raised);
        rj = two ? rj : 0.f;
#pragma unroll
        for (int k = 0; k < CPL; ++k) M[k] = fmaxf(fmaxf(M[k], x[k]), rj * y[k]);   // (0 * inf: NaN, which fmaxf drops)
        if (lane == 0 && t < picks) park(t, w1hi, w1);
        if (lane == 0 && two && t + 1 < picks) park(t + 1, w2hi, w2);
        t += two ? 2 : 1;
        return two ? w2hi : w1hi;
    };
    int t = 0;
    bool at_bound = false;
#pragma unroll 1
    while (t < picks && !at_bound) {
        float M0[CPL];
#pragma unroll
        for (int k = 0; k < CPL; ++k) M0[k] = M[k];
        const int t0 = t;
        float low = 0.f;
#pragma unroll
        for (int u = 0; u < kSteps; ++u) low = step(t);   // (picks beyond the last one are not parked)
        if (!(low > bound)) {
            // one of them, or one beyond the last pick, was not above the bound (or nothing is left to pick)
#pragma unroll
            for (int k = 0; k < CPL; ++k) M[k] = M0[k];
            t = t0;
#pragma unroll 1
            for (int u = 0; u < 2 * kSteps && t < picks; ++u, ++t) {
                float whi;
                uint32_t w;
                winner(whi, w);
                at_bound = !(whi > bound || (BOUNDED && tie_slot && whi == bound && whi > ninf && (int)bypool[w & 255u] < *tie_slot));
                if (at_bound) break;
                if (lane == 0) park(t, whi, w);
                float ri, x[CPL];
                load_row(w, ri, x);
#pragma unroll
                for (int k = 0; k < CPL; ++k) M[k] = fmaxf(M[k], ri * x[k]);
            }
        }
    }
    t = min(t, picks);
    __syncwarp();
    for (int i = lane; i < t; i += 32) {
        const float val = __uint_as_float(park_key[i]);
        park_key[i] = orderable(val <= -2.9e38f ? ninf : val);
    }
    if (at_bound) {
        __syncwarp();
        if (!BOUNDED || bound_key == 0u) {
            // no bound: every value left is -inf (cosines overflowed)
            if (lane == 0) {
                for (; t < picks; ++t) {
                    park_key[t] = orderable(ninf);
                    park_row[t] = lowest_free_row(park_row, t);
                }
            }
            return true;
        }
        if (m_out) {
#pragma unroll
            for (int k = 0; k < CPL; ++k)
                if (lane + 32 * k < P) m_out[lane + 32 * k] = M[k];
        }
        if (t_out && lane == 0) *t_out = t;
        return false;
    }
    return true;
}

// The picks that are missing after the loop over an active set reached its bound with `made` picks done. Those stand (no
// left-out candidate could have won them). The rest, a few as a rule, are taken over the whole pool with rows of the cosine
// matrix as plain dot products, from the state the loop left: its running maxima for the rows it had (m_act), and for the
// rows it had left out the maximum over the picks made, formed here. All threads call, after a barrier; the arrays are the
// event kernels' (the tile is free).
constexpr unsigned kContScratch = 2048u;   // behind the row of the cosine matrix: 2 x 1 KB + 2 x 512 B + 512 B + 256 B + 4 B
constexpr unsigned kContMact = 8192u;      // m_act, 1 KB
//
// Out of line and with few arguments (the rest is found again from them), so that it costs the kernels that call it
// neither registers nor a stretch of cold code between the phases (inlined: 2.5 % of event_tri_kernel).
template <int FORM, int NT>
__device__ __noinline__ void picks_over_whole_pool(const EventArgs& a, unsigned char* smem, int n, int active, int picks, int made) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const DevLayout& lay = a.lay;
    const EventId id = decode_event(lay, blockIdx.x);
    constexpr bool POOL = FORM >= 0;   // (below 0: event_tri_kernel)
    const TriSmem sp = POOL ? plan_pool_event_smem<POOL ? FORM : 0>(lay.N, a.budget, lay.page_size != 0) : plan_tri_smem(lay.N, a.budget, lay.page_size != 0);
    const float* G = POOL && a.gram ? a.gram + id.b * a.gram_sb + id.l * a.gram_sl : nullptr;
    const float* s = reinterpret_cast<const float*>(smem + sp.s);
    unsigned short* bypool = reinterpret_cast<unsigned short*>(smem + sp.bypool);
    float* r = reinterpret_cast<float*>(smem + sp.key);
    int* order = reinterpret_cast<int*>(smem + sp.order);
    uint32_t* park_key = reinterpret_cast<uint32_t*>(smem + sp.gain);
    unsigned char* tile = smem + sp.tile;
    int* holders = reinterpret_cast<int*>(smem + sp.misc + 32);
    const float thr = *reinterpret_cast<const float*>(smem + sp.misc + 56);
    const __nv_bfloat16* Vg = reinterpret_cast<const __nv_bfloat16*>(a.V);
    const bool dense = lay.page_size == 0;
    const __nv_bfloat16* Ve = Vg + (dense ? id.b * lay.sb + id.l * lay.sl + id.h * lay.sh : 0);
    auto vrow_of = [&](int j) { return dense ? Ve + (long long)j * lay.sn : Vg + row_offset(lay, id.b, id.l, id.h, j); };
    float* rowbuf = reinterpret_cast<float*>(tile);
    const float* m_act = reinterpret_cast<const float*>(tile + kContMact);   // by old pool row (from the loop)
    float* m_slot = reinterpret_cast<float*>(tile + kContScratch);           // by slot
    float* m_init = m_slot + 256;                                              // by new pool row
    unsigned short* inv = reinterpret_cast<unsigned short*>(m_init + 256);     // slot -> new pool row
    unsigned short* left = inv + 256;                                          // new pool rows the loop had left out
    int* chosen = reinterpret_cast<int*>(left + 256);                          // slots of the picks made
    unsigned char* state = reinterpret_cast<unsigned char*>(chosen + 128);     // by slot: 1 in the old active set
    int* n_left = reinterpret_cast<int*>(state + 256);
    for (int j = tid; j < 256; j += NT) state[j] = 0;
    if (tid == 0) *n_left = 0;
    __syncthreads();
    for (int rho = tid; rho < active; rho += NT) {
        const int j = bypool[rho];
        state[j] = 1;
        m_slot[j] = m_act[rho];
    }
    for (int t = tid; t < made; t += NT) chosen[t] = bypool[order[t]];
    __syncthreads();
    if (warp == 0) {
        int base = 0;
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int j = lane + 32 * k;
            const bool in = j < n && !(s[j] < thr);
            const uint32_t mask = __ballot_sync(0xFFFFFFFFu, in);
            if (in) bypool[base + __popc(mask & ((1u << lane) - 1u))] = (unsigned short)j;
            base += __popc(mask);
        }
        if (lane == 0) holders[0] = base;
    }
    __syncthreads();
    const int P = holders[0];
    for (int rho = tid; rho < P; rho += NT) {
        const int j = bypool[rho];
        inv[j] = (unsigned short)rho;
        if (state[j]) {
            m_init[rho] = m_slot[j];
        } else {
            m_init[rho] = 0.f;
            left[atomicAdd(n_left, 1)] = (unsigned short)rho;
        }
        if (G) { r[rho] = 1.f; continue; }
        const __nv_bfloat16* vrow = vrow_of(j);
        float ss = 0.f;
#pragma unroll
        for (int c = 0; c < 16; ++c) {
            float x[8];
            load8(vrow + c * 8, x);
#pragma unroll
            for (int e = 0; e < 8; ++e) ss = fmaf(x[e], x[e], ss);
        }
        r[rho] = 1.f / (sqrtf(ss) + a.eps);
    }
    __syncthreads();
    for (int t = tid; t < made; t += NT) order[t] = inv[chosen[t]];
    __syncthreads();
    auto dot = [&](int i, const __nv_bfloat16* vi, int c) -> float {   // of two pool rows (vi: row i's values)
        if (G) return G[(long long)bypool[i] * lay.N + bypool[c]];
        const __nv_bfloat16* vc = vrow_of(bypool[c]);
        float acc = 0.f;
#pragma unroll 4
        for (int q = 0; q < 16; ++q) {
            float xi[8], xc[8];
            load8(vi + q * 8, xi);
            load8(vc + q * 8, xc);
#pragma unroll
            for (int e = 0; e < 8; ++e) acc = fmaf(xi[e], xc[e], acc);
        }
        return acc;
    };
    // left-out rows against the picks made: m = max(0, max_t r_t <V_c, V_t>), every (row, pick) pair its own dot
    // product, the maximum by an integer atomic (the values are non-negative floats)
    const int pairs = *n_left * made;
    for (int x = tid; x < pairs; x += NT) {
        const int c = left[x / made], i = order[x % made];
        const float v = fmaxf(r[i] * dot(i, vrow_of(bypool[i]), c), 0.f);
        atomicMax(reinterpret_cast<int*>(m_init) + c, __float_as_int(v));
    }
    __syncthreads();
    GreedyLane<8> g;
    if (warp == 0) {
        g.init(lane, P, s, bypool, r, a.lam, true);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
            const int rho = lane + 32 * k;
            if (rho < P) {
                const float m0 = m_init[rho];
                g.M[k] = m0;
                if (m0 == __int_as_float(0x7f800000)) g.am[k] = 0u;  // picked already (the loop's +inf)
            }
        }
    }
    for (int t = made; t < picks; ++t) {
        if (warp == 0) {
            uint32_t bk;
            int irho = g.pick(lane, bk);
            if (lane == 0) {
                if (bk == 0u) { irho = lowest_free_row(order, t); bk = orderable(-INFINITY); }
                park_key[t] = bk; order[t] = irho; holders[1] = irho;
            }
        }
        if (t + 1 == picks) break;
        __syncthreads();
        const int irho = holders[1];
        // row irho of the cosine matrix
        const __nv_bfloat16* vpick = vrow_of(bypool[irho]);
        for (int rho = tid; rho < P; rho += NT) rowbuf[rho] = dot(irho, vpick, rho);
        __syncthreads();
        if (warp == 0) {
            const float ri = r[irho];
#pragma unroll
            for (int k = 0; k < 8; ++k) {
                const int rho = lane + 32 * k;
                if (rho < P) g.M[k] = fmaxf(g.M[k], ri * rowbuf[rho]);
            }
        }
    }
}

// FUSED: score + select + compact; otherwise selection only (scores are read from a.scores and
// nothing is rewritten). (The dense form looks at the layout although it is known: a constant there costs four bytes of spills at the 80
// registers of six CTAs per SM, and 4096 events of 192 rows to 64 198.0 us a pass instead of 196.5.)
template <bool FUSED, bool PAGED>
__global__ void __launch_bounds__(kTcThreads) event_tri_kernel(const __grid_constant__ EventArgs a, const __grid_constant__ ScoreTab tab) {
    extern __shared__ unsigned char smem_raw[];
    unsigned char* smem = smem_raw + ((1024u - (smem_u32(smem_raw) & 1023u)) & 1023u);
    const DevLayout& lay = a.lay;
    const EventId id = decode_event(lay, blockIdx.x);
    const int n = event_n(a, id.b);
    const int N = lay.N;
    const int bud = event_budget(a, id);
    const int picks = min(bud, n);
    const TriSmem sp = plan_tri_smem(N, a.budget, PAGED);
    unsigned char* tile = smem + sp.tile;
    float* tri = reinterpret_cast<float*>(tile);  // lower triangle of the cosine matrix, after the product
    float* s = reinterpret_cast<float*>(smem + sp.s);
    uint32_t* key = reinterpret_cast<uint32_t*>(smem + sp.key);
    float* r = reinterpret_cast<float*>(smem + sp.key);  // reuses the score keys' storage
    int* spos = reinterpret_cast<int*>(smem + sp.spos);
    unsigned short* bypool = reinterpret_cast<unsigned short*>(smem + sp.bypool);
    unsigned char* taken = smem + sp.taken;
    int* order = reinterpret_cast<int*>(smem + sp.order);
    float* gain = reinterpret_cast<float*>(smem + sp.gain);
    int* idx = reinterpret_cast<int*>(smem + sp.idx);
    float2* sect = reinterpret_cast<float2*>(smem + sp.sect);
    const uint32_t barK = smem_u32(smem + sp.misc);
    const uint32_t barM = barK + 8;
    const uint32_t barL = barK + 48;  // K rows from 128 on
    uint32_t* tmem_holder = reinterpret_cast<uint32_t*>(smem + sp.misc + 16);
    int* pool_holder = reinterpret_cast<int*>(smem + sp.misc + 20);
    int* pick_holder = reinterpret_cast<int*>(smem + sp.misc + 24);
    uint32_t* bound_holder = reinterpret_cast<uint32_t*>(smem + sp.misc + 28);  // key that no candidate outside the active set exceeds
    float* thr_holder = reinterpret_cast<float*>(smem + sp.misc + 56);          // the pool's score threshold
    int* tie_holder = reinterpret_cast<int*>(smem + sp.misc + 60);              // see picks_cosine: tie_slot
    int* redi = reinterpret_cast<int*>(smem + sp.misc + 32);
    const uint32_t tile_u32 = smem_u32(tile);
    const uint32_t half_bytes = (uint32_t)kTriTileRows * 128u;

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const bool similarity = a.greedy != 0 && picks > 1;   // (the first pick is the highest score in any case)
    const int np4 = (N + 3) & ~3;
    // row addressing: dense events are one base offset plus a row stride
    const bool dense = !PAGED && lay.page_size == 0;
    const long long ev_off = dense ? id.b * lay.sb + id.l * lay.sl + id.h * lay.sh : 0;
    // paged: where the event's pages start, looked up once by as many lanes of warp 0 at the same time (the block table's entries come from L2;
    // looked up row by row and copy by copy: 4096 events of 192 rows to 64 in pages of 64 191 us, 182 so). The other warps read
    // them behind the next block-wide barrier.
    long long* page_off = reinterpret_cast<long long*>(smem + sp.pages);
    const int pages = PAGED ? event_pages(N, lay.page_shift) : 0;
    const bool few_pages = PAGED && pages <= kPageOffsets;
    if (PAGED && few_pages) {
        if (tid < pages) page_off[tid] = row_offset(lay, id.b, id.l, id.h, tid << lay.page_shift);
        __syncwarp();
    }
    auto rowoff = [&](int j) -> long long {
        if (PAGED && few_pages) return page_off[j >> lay.page_shift] + (long long)(j & (lay.page_size - 1)) * lay.s_page_n;
        return dense ? ev_off + (long long)j * lay.sn : row_offset(lay, id.b, id.l, id.h, j);
    };
    __nv_bfloat16* Kg = reinterpret_cast<__nv_bfloat16*>(a.K);
    __nv_bfloat16* Vg = reinterpret_cast<__nv_bfloat16*>(a.V);

    phase_stamp(id.e, 0);  // phases: 0 start, 1 tensor memory claimed, 2 K scored, 3 pool, 4 V operand, 5 product, 6 triangle, 7 picks, 8 outputs, 9 end
    // Tensor memory is claimed first and the right to allocate given up at once: the SM starts its
    // next CTA of this kernel only after that, so a late allocation would serialise the CTAs.
    const bool use_tc = similarity;
    // K rows [r0, r1) -> tile slots from slot0 on: as few bulk copies as the layout allows (whole event
    // when its rows are contiguous, whole pages when pages are, else row by row), all issued by one
    // thread (a bulk copy is a per-warp instruction)
    auto request_k_rows = [&](int r0, int r1, int slot0, uint32_t bar) {
        mbar_expect_tx(bar, (uint32_t)(r1 - r0) * 256u);
        for (int row = r0; row < r1 && !a.starve;) {  // starve (testing aid): nothing is requested, the waits run out
            int run = 1;
            if (dense && lay.sn == kTcD) run = min(r1 - row, 128);
            else if (!dense && lay.s_page_n == kTcD) run = min(r1 - row, lay.page_size - (row & (lay.page_size - 1)));
            bulk_g2s(tile_u32 + (uint32_t)(slot0 + row - r0) * 256u, Kg + rowoff(row), (uint32_t)run * 256u, bar);
            row += run;
        }
    };
    const int n_late = FUSED && n > kTriTileRows ? n - kTriTileRows : 0;  // rows that wait for a free slot
    if (tid == 0) {
        mbar_init(barK, 1);
        mbar_init(barM, 1);
        mbar_init(barL, 1);
        mbar_init_fence();
    }
    if (FUSED && tid >= 32 && tid < 64) {
        float sn, cs;
        sincospif((float)(tid - 32) * 0.0625f, &sn, &cs);  // angle 2 pi h / 32
        sect[tid - 32] = make_float2(cs, sn);
    }
    if (warp == 0) {
        if (use_tc) tmem_alloc(smem_u32(tmem_holder), kTcCols);
        else tmem_relinquish();  // top-k events take no tensor memory, and must not hold up the next CTA's start
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tbase = use_tc ? *tmem_holder : 0u;

    phase_stamp(id.e, 1);
    // ---- scores ---------------------------------------------------------------------------------
    int bad = 0;
    int timeout = 0;
    if (FUSED) {
        if (tid == 0) request_k_rows(0, n - n_late, 0, barK);
        const int* gpos = event_pos(a.pos, id);
        const bool rotate = gpos != nullptr;
        int pmax = INT_MIN;
        for (int j = tid; j < n; j += kTcThreads) {
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
        long long pref = 0;
        if (rotate) pref = a.p_ref ? (long long)a.p_ref[id.b] : (long long)max(max(redi[0], redi[1]), max(redi[2], redi[3])) + 1;
        // lane covers frequencies f0..f0+7 of the row handled by its group of eight lanes
        const int grp = lane >> 3, f0 = (lane & 7) * 8;
        // spacing of rows 16 slots apart at the newest end of the event: what a token-by-token cache has everywhere
        const long long D16 = n > 16 ? (long long)spos[n - 1] - (long long)spos[n - 17] : 0;
        ChainScore cs;
        cs.set_step(D16, phitab + f0, sect);
        const int rounds = (n + 15) >> 4, late_round = (n_late + 15) >> 4;
        // 16 rows per round (4 per warp), in three stretches. Rows from 128 on reuse the slots of rows
        // 0..n_late-1: they are requested after the first stretch, once every warp is past those rows,
        // and awaited before the third. The rounds also run after a timeout (over whatever the tile
        // holds), so that the barrier between them is reached by every thread.
        auto score_rounds = [&](int round0, int round1) {
            for (int round = round0; round < round1; ++round) {
                const int j = 16 * round + 4 * warp + grp;
                const bool live = j < n;
                // G follows from the previous round's by the constant turn when all four rows of the warp sit
                // D16 after the rows 16 slots before them
                bool fresh = (round & (kChainRoundsShort - 1)) == 0 || a.no_chain;
                if (!fresh) fresh = !__all_sync(0xFFFFFFFFu, !live || (long long)spos[j] - (long long)spos[j - 16] == D16);
                if (fresh) {
                    if (live) cs.anchor(pref - (long long)spos[j], gtab + f0, phitab + f0, sect);
                } else {
                    cs.advance();
                }
                float acc = 0.f;
                if (live) {
                    const unsigned char* krow = tile + (j & (kTriTileRows - 1)) * 256 + (lane & 7) * 16;
                    acc = cs.dot(*reinterpret_cast<const uint4*>(krow), *reinterpret_cast<const uint4*>(krow + 128));
                }
#pragma unroll
                for (int off = 4; off > 0; off >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, off);
                if (live && (lane & 7) == 0) {
                    if (a.scores) a.scores[(long long)id.e * N + j] = acc;
                    const bool fin = isfinite(acc);
                    bad |= !fin;
                    const float sj = fin ? acc : -INFINITY;
                    s[j] = sj;
                    key[j] = orderable(sj);
                }
            }
        };
        timeout = !mbar_wait_polls(barK, 0, a.wait_polls);
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            // first and third stretch share one copy of the loop (the kernel's code should stay small)
            if (pass && n_late > 0) timeout |= !mbar_wait_polls(barL, 0, a.wait_polls);
            score_rounds(pass ? kTriTileRows / 16 : 0, pass ? rounds : late_round);
            if (!pass) {
                if (n_late > 0) {
                    __syncthreads();
                    if (tid == 0) request_k_rows(kTriTileRows, n, 0, barL);
                }
                score_rounds(late_round, min(rounds, kTriTileRows / 16));
            }
        }
    } else {
        for (int j = tid; j < n; j += kTcThreads) {
            const float sc = a.scores[(long long)id.e * N + j];
            const bool fin = isfinite(sc);
            bad |= !fin;
            const float sj = fin ? sc : -INFINITY;
            s[j] = sj;
            key[j] = orderable(sj);
        }
    }
    for (int j = n + tid; j < np4; j += kTcThreads) key[j] = 0u;  // below every real key
    timeout = __syncthreads_or(timeout);
    if (timeout) {
        if (tid == 0 && a.status) a.status[id.e] = 3;
        mbar_wait_polls(barK, 0, a.wait_polls);  // give copies still in flight another bounded chance to land
        if (n_late > 0) mbar_wait_polls(barL, 0, a.wait_polls);
        if (use_tc && warp == 0) tmem_dealloc(tbase, kTcCols);
        return;
    }
    bad = __syncthreads_or(bad);
    // (only now: while scoring, this storage holds the statistic's table, which slower warps may still read)
    for (int j = tid; j < np4; j += kTcThreads) taken[j] = 0;

    phase_stamp(id.e, 2);
    // ---- s_(b) by bisection over the score keys, then the pool in slot order (warp 0) -------------
    if (warp == 0) {
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
        // active set: no key left out is above bound.key (0: none is left out)
        ActiveBound bound{0u, 0};
        if (similarity) {
            int pool_size = 0;
#pragma unroll
            for (int k = 0; k < 8; ++k) pool_size += kk[k] != 0u && !(from_orderable(kk[k]) < thr);
            pool_size = __reduce_add_sync(0xFFFFFFFFu, pool_size);
            if (pool_size > kTriMaxPool) bound = warp_active_bound(kk, orderable(thr), kb, kTriMaxPool);
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
    const int P = *pool_holder;

    phase_stamp(id.e, 3);
    // ---- V rows of the pool as the swizzled operand tile ---------------------------------------------
    if (similarity) {
        // thread -> 16-byte column c of rows r0, r0 + 8, ...: the swizzle term (c ^ row) & 7 is the same for
        // all of them, so a row costs one pool lookup, one address and one copy
        const int c = tid & 15, r0 = tid >> 4;
        const uint32_t dst0 = tile_u32 + tile_chunk(r0, c, half_bytes);
        if (dense) {
            const __nv_bfloat16* vcol = Vg + ev_off + c * 8;
            for (int rho = r0; rho < P; rho += 8)
                cp_async16(dst0 + (uint32_t)(rho - r0) * 128u, vcol + (long long)bypool[rho] * lay.sn);
        } else {
            for (int rho = r0; rho < P; rho += 8)
                cp_async16(dst0 + (uint32_t)(rho - r0) * 128u, Vg + rowoff(bypool[rho]) + c * 8);
        }
        cp_async_wait_all();
        fence_proxy_async();
        __syncthreads();
    }
    phase_stamp(id.e, 4);
    if (similarity) {
        if (tid == 0 && (FUSED || !a.starve)) {
            tc_fence_after();
            const uint32_t idesc = umma_idesc_bf16(128, max((P + 15) & ~15, 16));   // (a shape with no columns is not allowed)
#pragma unroll
            for (int kk = 0; kk < 8; ++kk) {
                const uint32_t koff = (uint32_t)(kk >> 2) * half_bytes + (uint32_t)(kk & 3) * 32u;
                umma_bf16(tbase, umma_desc_sw128(tile_u32 + koff), umma_desc_sw128(tile_u32 + koff), idesc, kk > 0 ? 1u : 0u);
            }
            umma_commit(barM);
        }
        timeout = !mbar_wait_polls(barM, 0, a.wait_polls);
        tc_fence_after();
    }
    timeout = __syncthreads_or(timeout);  // also: the product has read the whole tile before the triangle lands on it
    if (timeout) {
        if (tid == 0 && a.status) a.status[id.e] = 3;
        if (!FUSED) select_gave_up(a, id.e, kTcThreads);
        if (use_tc && warp == 0) tmem_dealloc(tbase, kTcCols);
        return;
    }
    phase_stamp(id.e, 5);
    if (similarity) {
        // lower triangle -> shared memory; row rho = 32 warp + lane needs columns 0..rho
        const int rho = 32 * warp + lane;
        if (32 * warp < P) {
            const int trow = tri_row(rho);
            const uint32_t lanes = tbase + ((uint32_t)(warp * 32) << 16);
            // column blocks left of the diagonal one: every column is below the row
            for (int cb = 0; cb < warp; ++cb) {
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
                tmem_ld32(lanes + (uint32_t)(32 * warp), v);
                tmem_ld_wait();
                if (rho < P) {
#pragma unroll
                    for (int k = 0; k < 32; ++k)
                        if (k <= lane) tri[trow + 32 * warp + k] = __uint_as_float(v[k]);
                    r[rho] = 1.f / (sqrtf(tri[trow + rho]) + a.eps);  // read back: this thread stored it
                }
            }
        }
    }
    tc_fence_before();
    __syncthreads();
    if (use_tc && warp == 0) tmem_dealloc(tbase, kTcCols);

    phase_stamp(id.e, 6);
    // ---- Algorithm 1 in warp 0 -------------------------------------------------------------------------
    // The winning key of every pick is parked in gain[] and its pool row in order[]; both are decoded
    // after the loop.
    uint32_t* park_key = reinterpret_cast<uint32_t*>(gain);
    if (!similarity) {
        picks_by_rank<kTcThreads>(tid, P, picks, key, bypool, park_key, order);
    } else {
        if (warp == 0) {
            const bool ok = picks_cosine<4, true>(lane, P, picks, s, bypool, r, a.lam, tri, park_key, order, *bound_holder,
                                                  reinterpret_cast<float*>(tile + kContMact), redi, nullptr, tie_holder);
            if (lane == 0) *pick_holder = ok ? picks : *redi;
        }
        __syncthreads();
        if (*pick_holder < picks) {
            picks_over_whole_pool<-1, kTcThreads>(a, smem, n, P, picks, *pick_holder);
        }
    }
    __syncthreads();
    for (int t = tid; t < picks; t += kTcThreads) {
        const int j = bypool[order[t]];
        gain[t] = from_orderable(park_key[t]);
        order[t] = j;
        taken[j] = 1;
    }
    __syncthreads();

    phase_stamp(id.e, 7);
    // ---- sort(S) and outputs -------------------------------------------------------------------------
    ordered_indices(n, a.budget, taken, idx);
    __syncthreads();
    const long long ob = (long long)id.e * a.budget;
    for (int t = tid; t < a.budget; t += kTcThreads) {
        a.idx_sorted[ob + t] = idx[t];
        if (a.pick_order) a.pick_order[ob + t] = t < picks ? order[t] : -1;
        if (a.pick_gain) a.pick_gain[ob + t] = t < picks ? gain[t] : 0.f;
    }
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
        // thread -> 16-byte column c of kept rows r0, r0 + 8, ...
        const int c = tid & 15, r0 = tid >> 4;
        const uint32_t slot0 = (uint32_t)(r0 * 256 + c * 16);
        const long long col = (dense ? ev_off : 0) + c * 8;
        for (int t = r0; t < picks; t += 8) {
            const long long off = col + (dense ? (long long)idx[t] * lay.sn : rowoff(idx[t]));
            cp_async16(tile_u32 + slot0 + (uint32_t)(t - r0) * 256u, Kg + off);
            cp_async16(tile_u32 + 16384u + slot0 + (uint32_t)(t - r0) * 256u, Vg + off);
        }
        cp_async_wait_all();
        __syncthreads();  // every load above has been performed
        for (int t = r0; t < picks; t += 8) {
            const long long off = col + (dense ? (long long)t * lay.sn : rowoff(t));
            const unsigned char* src = tile + slot0 + (t - r0) * 256;
            *reinterpret_cast<uint4*>(Kg + off) = *reinterpret_cast<const uint4*>(src);
            *reinterpret_cast<uint4*>(Vg + off) = *reinterpret_cast<const uint4*>(src + 16384);
        }
    } else {
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
            __nv_bfloat16* X = pass ? Vg : Kg;
            __syncthreads();  // the tile is free (greedy loop, or the previous pass, is done with it)
            for (int x = tid; x < picks * 16; x += kTcThreads)
                copy16(tile + x * 16, reinterpret_cast<const char*>(X + rowoff(idx[x >> 4])) + (x & 15) * 16);
            __syncthreads();
            for (int x = tid; x < picks * 16; x += kTcThreads)
                copy16(reinterpret_cast<char*>(X + rowoff(x >> 4)) + (x & 15) * 16, tile + x * 16);
        }
    }
    if (wpos)
        for (int t = tid; t < picks; t += kTcThreads) wpos[t] = spos[idx[t]];
    phase_stamp(id.e, 9);
}

}  // namespace akv
