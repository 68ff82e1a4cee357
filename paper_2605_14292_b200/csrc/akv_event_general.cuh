// Fused event for every shape the tensor-memory kernels do not take (fp32, head dimensions other than 128,
// the maximum over grouped query statistics, shared signatures without a cosine matrix), when the event's K and V tiles
// fit in shared memory.
//
// Selection, when lambda > 0: the exact pool (s_i >= s_(b) - lambda (1 + slack), see akv_select_pool.cuh) is
// formed, and when the lower triangle of its cosine matrix fits, into the shared memory left beside the tiles or else over
// the K tile, which scoring is done with (the kept K rows are then read again for the compaction), the triangle is filled
// by plain fp32 dot products and Algorithm 1 runs as the one-warp loop of the tensor-memory kernels. A pool that does not
// fit is taken in rounds of active sets (picks_in_rounds). Otherwise, and for lambda = 0, the CTA-wide loop with rows of the
// cosine matrix on demand (greedy_cta). (896 events of 256 bf16 rows of 64, 128 kept, lambda = 0.5, the
// call alone: 345 us in rounds, 1471 in the CTA-wide loop, 556 with the whole triangle and one CTA per SM.)
//
// The dot products are bound by shared-memory reads, so a thread takes 8 x 4 pairs of rows at a time (12 reads for
// 128 multiply-adds a step instead of 2 for 4), walking the head dimension from its own starting column so that a warp's loads
// fall into different banks.
#pragma once
#include "akv_event_tri.cuh"

namespace akv {

// The rows of one event in the n slots listed (slots null: 0..n-1), from global memory into a dense shared tile by 16-byte
// asynchronous copies, all in flight at once (a lane keeps its column, a row costs one address), as one group of copies; the caller
// waits and synchronises before reading the tile.
template <typename T>
__device__ __forceinline__ void load_rows_async(T* tile, const T* base, const DevLayout& lay, const EventId& id, int n, const int* slots) {
    const int cpr = lay.d * (int)sizeof(T) / 16;  // 16-byte chunks per row
    const int lanes = min(pow2_ceil(cpr), 32), rows = 32 / lanes, lane = threadIdx.x & 31;
    const uint32_t t0 = smem_u32(tile);
    for (int row = (threadIdx.x >> 5) * rows + lane / lanes; row < n; row += kWarps * rows) {
        const char* src = reinterpret_cast<const char*>(base + row_offset(lay, id.b, id.l, id.h, slots ? slots[row] : row));
        for (int c = lane & (lanes - 1); c < cpr; c += lanes) cp_async16(t0 + (uint32_t)(row * cpr + c) * 16u, src + c * 16);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
}
template <int PENDING>
__device__ __forceinline__ void cp_async_wait_pending() {
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}
// Rows that one bulk copy can take: up to 32 KB where rows are contiguous (at most a page, where pages are), else one.
__device__ __forceinline__ int rows_per_copy(const DevLayout& lay, int row_bytes) {
    if (lay.page_size == 0 ? lay.sn != lay.d : lay.s_page_n != lay.d) return 1;
    const int run = max(32768 / row_bytes, 1);
    if (lay.page_size == 0) return run;
    return run > lay.page_size ? lay.page_size : 1 << (31 - __clz(run));   // (a power of two, like pages: no copy crosses one)
}
// Rows 0..n-1 of one event from global memory into a dense shared tile by bulk copies of `run` rows each, which report to `bar`; one
// warp calls, its lanes share the copies. (192 rows of K and V in fp32, d = 128, contiguous: all threads' 16-byte copies took 13.3 of
// an event's 65 thousand cycles to issue; one event 38.9 -> 34.8 us, 896 of them 240 -> 209.)
template <typename T>
__device__ __forceinline__ void load_tile_bulk(T* tile, const T* base, const DevLayout& lay, const EventId& id, int n, uint32_t bar, int run) {
    const uint32_t row_bytes = (uint32_t)lay.d * (uint32_t)sizeof(T), t0 = smem_u32(tile);
    const int lane = threadIdx.x & 31;
    if (lane == 0) mbar_expect_tx(bar, (uint32_t)n * row_bytes);
    __syncwarp();
    for (int row = lane * run; row < n; row += 32 * run)
        bulk_g2s(t0 + (uint32_t)row * row_bytes, base + row_offset(lay, id.b, id.l, id.h, row), (uint32_t)min(run, n - row) * row_bytes, bar);
}
// Smallest copy of a paged cache that is worth a bulk copy; rows that lie apart in a dense one never are. One warp's many small
// copies are slower than all threads' 16-byte ones, whose addresses cost more where they go through a block table. 896 events, us per call
// with bulk copies / 16-byte ones. Pages: copies of 64 bytes 115 / 87 (256 rows of 16 bf16, pages of 2), of 256 130 / 118 (192 of 64 bf16,
// pages of 2), of 512 117 / 117 (pages of 4) and 303 / 297 (192 of 128 fp32, pages of 1), of 1024 111 / 115 (192 of 64 bf16, pages of 8),
// 256 / 281 (192 of 128 fp32, pages of 2) and 242 / 244 (96 of 256 fp32, pages of 1). Rows apart: of 128 bytes 146 / 111, of 512 281 / 242
// (192 of 128 fp32) and 363 / 332 (160 of 256 bf16), of 1024 233 / 223 (96 of 256 fp32).
constexpr int kLeastBulk = 1024;

constexpr int kResidentCtas = 2;       // most CTAs per SM that the registers of the kernel with the penalty allow
constexpr int kResidentCtasTopk = 3;   // ... and of the one without: no triangle (896 events of 128 bf16 rows of 64: 107 us, with the
                                       // other's 128 registers 156)
constexpr int kResidentLeastSet = 64;  // rows from which an active set is worth its triangle

// Where a row's values lie: four at a time from global memory, or from shared memory by 32-bit address (a generic pointer's loads
// and arithmetic cost more).
struct GlobalRow {
    const float* p;
    __device__ __forceinline__ GlobalRow operator+(int n) const { return {p + n}; }
    __device__ __forceinline__ void load(float (&x)[4]) const { load4(p, x); }
};
template <typename T>
struct SharedRow {
    uint32_t at;
    __device__ __forceinline__ SharedRow operator+(int n) const { return {at + (uint32_t)(n * (int)sizeof(T))}; }
    __device__ __forceinline__ void load(float (&x)[4]) const {
        if constexpr (sizeof(T) == 4) {
            asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]) : "r"(at));
        } else {
            uint32_t a, b;
            asm volatile("ld.shared.v2.b32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "r"(at));
            x[0] = bf16lo(a); x[1] = bf16hi(a); x[2] = bf16lo(b); x[3] = bf16hi(b);
        }
    }
};

// Raw dot products of every pair of the R rows listed in `rows` (i >= j) -> the triangle `tri`, 8 x 4 at a time: thread x
// takes blocks x, x + 256, ...; row band b of eight rows has 2 b + 2 blocks, so it starts at block b (b + 1). row_of: slot ->
// values.
template <typename RowOf>
__device__ __forceinline__ void fill_triangle(RowOf row_of, const unsigned short* rows, int R, int d, float* tri) {
    const int tid = threadIdx.x, G4 = d >> 2;   // G4: groups of four elements per row
    const int bands = (R + 7) >> 3, blocks = bands * (bands + 1);
    for (int x = tid; x < blocks; x += kThreads) {
        int bi = (int)sqrtf((float)x);
        while (bi * (bi + 1) > x) --bi;
        while ((bi + 1) * (bi + 2) <= x) ++bi;
        const int bj = x - bi * (bi + 1);
        float acc[8][4] = {};
        decltype(row_of(0)) vi[8], vj[4];
#pragma unroll
        for (int q = 0; q < 8; ++q) vi[q] = row_of(rows[min(8 * bi + q, R - 1)]);
#pragma unroll
        for (int q = 0; q < 4; ++q) vj[q] = row_of(rows[min(4 * bj + q, R - 1)]);
        int gq = tid % G4;
#pragma unroll 1
        for (int c = 0; c < G4; ++c) {
            float xi[8][4], xj[4][4];
#pragma unroll
            for (int q = 0; q < 4; ++q) (vj[q] + 4 * gq).load(xj[q]);
#pragma unroll
            for (int p = 0; p < 8; ++p) (vi[p] + 4 * gq).load(xi[p]);
#pragma unroll
            for (int p = 0; p < 8; ++p)
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int e = 0; e < 4; ++e) acc[p][q] = fmaf(xi[p][e], xj[q][e], acc[p][q]);
            gq = gq + 1 == G4 ? 0 : gq + 1;
        }
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
            for (int q = 0; q < 4; ++q)
                if (8 * bi + p < R && 4 * bj + q <= 8 * bi + p) tri[tri_row(8 * bi + p) + 4 * bj + q] = acc[p][q];
    }
}

// State of the rounds over active sets, in the shared memory beside the tiles or else at the head of the K tile.
struct ResidentState {
    unsigned key, seen, row, in, r, m, total;
};
__host__ __device__ inline ResidentState plan_resident_state(int N) {
    ResidentState p;
    unsigned o = 0;
    p.key = o;  o += align16((unsigned)N * 4);   // by slot: the most that the row's value can be, 0 once it is picked
    p.seen = o; o += align16((unsigned)N * 2);   // by slot: how many picks its running maximum covers
    p.row = o;  o += align16((unsigned)N * 2);   // the active set's slots
    p.in = o;   o += align16((unsigned)N);       // by slot: 1 in the active set
    p.r = o;    o += 1024;                       // the set's norms
    p.m = o;    o += 1024;                       // and running maxima
    p.total = o;
    return p;
}

// Algorithm 1 in rounds over the best rows of a pool whose triangle does not fit (`low`: the pool's threshold, as a key).
// At the bound of an active set the picks made stand, and the next set is formed from what is known of every row's value,
// as in akv_event_prefill.cuh. All threads call, after a barrier; s and r by slot, taken 0. Leaves order[], gain[] and
// taken[] and returns kRoundsDone; leaves taken 0 and returns without that bit where a set would be too small or values are
// lost to infinite cosines. kRoundsOverK: the K tile was written over. Out of line: registers and code of the kernel stay
// those of the pool that fits.
constexpr int kRoundsDone = 1, kRoundsOverK = 2;
template <typename T>
__device__ __noinline__ int picks_in_rounds(const EventArgs& a, unsigned char* smem, int n, int picks, uint32_t low, int extra_bytes) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int d = a.lay.d, N = a.lay.N, G4 = d >> 2;
    const EventId id = decode_event(a.lay, blockIdx.x);
    const SmemPlan sp = plan_smem(N, d, sizeof(T), a.budget, true, true);
    const T* Vt = reinterpret_cast<const T*>(smem + sp.tileV);
    const float* s = reinterpret_cast<const float*>(smem + sp.s);
    const float* r = reinterpret_cast<const float*>(smem + sp.r);
    float* m = reinterpret_cast<float*>(smem + sp.m);
    int* order = reinterpret_cast<int*>(smem + sp.order);
    float* gain = reinterpret_cast<float*>(smem + sp.gain);
    uint32_t* park_key = reinterpret_cast<uint32_t*>(gain);
    unsigned char* taken = smem + sp.taken;
    const float* sig = a.flat_sig ? event_sig(a, id) : nullptr;
    // state and triangle: beside the tiles what fits there, the rest over the K tile
    const ResidentState rs = plan_resident_state(N);
    const bool state_beside = (int)rs.total <= extra_bytes;
    unsigned char* state = state_beside ? smem + sp.total : smem + sp.tileK;
    const int room_beside = extra_bytes - (state_beside ? (int)rs.total : 0);
    const int room_over = N * d * (int)sizeof(T) - (state_beside ? 0 : (int)rs.total);
    const int room = max(room_beside, room_over);
    int cap = min((int)sqrtf((float)room * 0.5f), 256);   // rows whose triangle fits
    while (2 * cap * (cap + 1) > room) --cap;
    if (cap < kResidentLeastSet) return 0;
    int over_k = state_beside ? 0 : kRoundsOverK;
    uint32_t* key = reinterpret_cast<uint32_t*>(state + rs.key);
    unsigned short* seen = reinterpret_cast<unsigned short*>(state + rs.seen);
    unsigned short* act = reinterpret_cast<unsigned short*>(state + rs.row);
    unsigned char* in_set = state + rs.in;
    float* ar = reinterpret_cast<float*>(state + rs.r);
    float* am = reinterpret_cast<float*>(state + rs.m);
    uint32_t* bound_holder = reinterpret_cast<uint32_t*>(smem + sp.red);
    int* tie_holder = reinterpret_cast<int*>(smem + sp.red) + 1;    // see picks_cosine: tie_slot
    int* made_holder = reinterpret_cast<int*>(smem + sp.red) + 2;
    for (int j = tid; j < n; j += kThreads) {
        key[j] = orderable(s[j]);
        seen[j] = 0;
        m[j] = 0.f;
    }
    __syncthreads();
    int made = 0, idle = 0;   // idle: rounds without a pick since the last one (the limit is a safeguard)
    while (made < picks && idle <= n / cap + 2) {
        // ---- the active set: the pool's rows with the largest keys, equal ones by slot
        int P = 0;
        for (int j0 = 0; j0 < n; j0 += kThreads) P += __syncthreads_count(j0 + tid < n && key[j0 + tid] >= low);
        for (int j = tid; j < n; j += kThreads) {
            const uint32_t kj = key[j];
            bool in = kj >= low;
            if (in && P > cap) {
                int rank = 0;
                for (int i = 0; i < n; ++i) {
                    const uint32_t ki = key[i];
                    rank += ki > kj || (ki == kj && i < j);
                }
                in = rank < cap;
                if (rank == cap) {   // the best row left out
                    *bound_holder = kj;
                    *tie_holder = j;
                }
            }
            in_set[j] = in;
        }
        __syncthreads();
        const int R = min(P, cap);
        const uint32_t bound = P > cap ? *bound_holder : 0u;
        if (bound == 0u && R < picks - made) break;   // (values lost to overflowed cosines)
        if (warp == 0) {
            int base = 0;
            for (int j0 = 0; j0 < n; j0 += 32) {
                const int j = j0 + lane;
                const bool in = j < n && in_set[j];
                const uint32_t mask = __ballot_sync(0xFFFFFFFFu, in);
                if (in) act[base + __popc(mask & ((1u << lane) - 1u))] = (unsigned short)j;
                base += __popc(mask);
            }
        }
        __syncthreads();
        if (tid < R) {
            ar[tid] = sig ? 1.f : r[act[tid]];
            am[tid] = m[act[tid]];
        }
        __syncthreads();
        // running maxima over the picks that a row has not seen yet: a dot product per (row, pick), the maximum by an integer
        // atomic (the values are non-negative floats)
        for (int x = tid; x < R * made; x += kThreads) {
            const int row = x / made, t = x - row * made, j = act[row], i = order[t];
            if (t < seen[j]) continue;
            float acc = 0.f;
            int gq = tid % G4;
            for (int c = 0; c < G4; ++c) {
                float xi[4], xj[4];
                if (sig) {
                    load4(sig + (long long)i * d + 4 * gq, xi);
                    load4(sig + (long long)j * d + 4 * gq, xj);
                } else {
                    load4(Vt + (size_t)i * d + 4 * gq, xi);
                    load4(Vt + (size_t)j * d + 4 * gq, xj);
                }
#pragma unroll
                for (int e = 0; e < 4; ++e) acc = fmaf(xi[e], xj[e], acc);
                gq = gq + 1 == G4 ? 0 : gq + 1;
            }
            atomicMax(reinterpret_cast<int*>(am) + row, __float_as_int(fmaxf((sig ? 1.f : r[i]) * acc, 0.f)));
        }
        const bool beside = 2 * R * (R + 1) <= room_beside;
        if (!beside) over_k = kRoundsOverK;
        float* tri = reinterpret_cast<float*>(beside ? smem + sp.total + (state_beside ? rs.total : 0u) : smem + sp.tileK + (state_beside ? 0u : rs.total));
        if (sig) fill_triangle([&](int j) { return GlobalRow{sig + (long long)j * d}; }, act, R, d, tri);
        else fill_triangle([&](int j) { return SharedRow<T>{smem_u32(Vt) + (uint32_t)(j * d * (int)sizeof(T))}; }, act, R, d, tri);
        __syncthreads();
        if (warp == 0) {
            const bool ok = picks_cosine<8, true>(lane, R, picks - made, s, act, ar, a.lam, tri, park_key + made, order + made, bound, am, made_holder, am,
                                                  tie_holder);
            if (ok && lane == 0) *made_holder = picks - made;
        }
        __syncthreads();
        const int got = *made_holder;
        for (int t = made + tid; t < made + got; t += kThreads) {
            const int j = act[order[t]];
            gain[t] = from_orderable(park_key[t]);
            order[t] = j;
            taken[j] = 1;
        }
        __syncthreads();
        made += got;
        if (made < picks && tid < R) {
            const int j = act[tid];
            m[j] = am[tid];
            seen[j] = (unsigned short)made;
            key[j] = taken[j] ? 0u : orderable(fmaf(-fmaxf(penalty_rate(a.lam, ar[tid]), 1e-30f), am[tid], fmaxf(s[j], kLowestScore)));
        }
        idle = got ? 0 : idle + 1;
        __syncthreads();
    }
    if (made == picks) return kRoundsDone | over_k;
    for (int j = tid; j < n; j += kThreads) taken[j] = 0;
    return over_k;
}

// ---------------------------------------------------------------------------------------------
// Fused event, tiles resident in shared memory: K and V are read from HBM once and the kept rows
// are written once. One CTA per (sequence, layer, KV head).
// ---------------------------------------------------------------------------------------------
template <typename T, bool PENALTY>
__global__ void __launch_bounds__(kThreads, PENALTY ? kResidentCtas : kResidentCtasTopk) event_resident_kernel(const __grid_constant__ EventArgs a, const __grid_constant__ ScoreTab tab, int extra_bytes) {
    extern __shared__ __align__(16) unsigned char smem[];
    const DevLayout& lay = a.lay;
    const EventId id = decode_event(lay, blockIdx.x);
    const int n = event_n(a, id.b);
    const int d = lay.d, N = lay.N;
    const SmemPlan sp = plan_smem(N, d, sizeof(T), a.budget, true, true);
    T* Kt = reinterpret_cast<T*>(smem + sp.tileK);
    T* Vt = reinterpret_cast<T*>(smem + sp.tileV);
    unsigned long long* phi = reinterpret_cast<unsigned long long*>(smem + sp.phi);
    float2* g = reinterpret_cast<float2*>(smem + sp.g);
    int* spos = reinterpret_cast<int*>(smem + sp.pos);
    float* s = reinterpret_cast<float*>(smem + sp.s);
    float* r = reinterpret_cast<float*>(smem + sp.r);
    float* m = reinterpret_cast<float*>(smem + sp.m);
    int* order = reinterpret_cast<int*>(smem + sp.order);
    float* gain = reinterpret_cast<float*>(smem + sp.gain);
    int* idx = reinterpret_cast<int*>(smem + sp.idx);
    unsigned char* taken = smem + sp.taken;
    unsigned long long* red = reinterpret_cast<unsigned long long*>(smem + sp.red);
    int* redi = reinterpret_cast<int*>(smem + sp.red + 2 * kWarps * 8);

    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int* gpos = event_pos(a.pos, id);
    T* Kg = reinterpret_cast<T*>(a.K);
    T* Vg = reinterpret_cast<T*>(a.V);

    phase_stamp(id.e, 0);  // phases: 0 start, 1 K landed, 2 scores, V landed, 3 norms, 4 pool, 5 triangle, 6 picks, 7 outputs, 8 end
    // stage the event on chip (the barriers' place is the reductions', which come later)
    const uint32_t bar_k = smem_u32(red), bar_v = bar_k + 8;
    volatile int* late = reinterpret_cast<volatile int*>(red) + 4;   // a wait for them ran out
    if (warp == 0) {
        if (lane == 0) {
            mbar_init(bar_k, 1);
            mbar_init(bar_v, 1);
            *late = 0;
            mbar_init_fence();
        }
        __syncwarp();
    }
    const int run = rows_per_copy(lay, d * (int)sizeof(T));
    if (a.starve) {
        // (a testing aid: nothing is requested and nobody reports to the barriers, the waits for them run out)
    } else if (lay.page_size ? run * d * (int)sizeof(T) >= kLeastBulk : run > 1) {
        if (warp == 0) {
            load_tile_bulk(Kt, Kg, lay, id, n, bar_k, run);
            load_tile_bulk(Vt, Vg, lay, id, n, bar_v, run);
        }
    } else {
        if (tid == 0) {   // (the copies are awaited as groups)
            mbar_expect_tx(bar_k, 0);
            mbar_expect_tx(bar_v, 0);
        }
        load_rows_async(Kt, Kg, lay, id, n, nullptr);
        load_rows_async(Vt, Vg, lay, id, n, nullptr);
    }
    int pmax = INT_MIN;
    for (int j = tid; j < n; j += kThreads) {
        const int p = gpos ? gpos[j] : 0;
        spos[j] = p;
        pmax = max(pmax, p);
        taken[j] = 0;
        m[j] = 0.f;
    }
    for (int f = tid; f < d / 2; f += kThreads) phi[f] = tab.phi[f];
    const int members = fold_group(a, id, tab, d, g);
    long long pref = 0;
    if (gpos) pref = a.p_ref ? (long long)a.p_ref[id.b] : (long long)block_max_int(pmax, redi) + 1;
    cp_async_wait_pending<1>();
    __syncthreads();
    if (!mbar_wait_bounded(bar_k, 0, a.wait_polls)) *late = 1;   // K has landed; V may still be under way
    phase_stamp(id.e, 1);

    // scores: four rows of a lane group at a time, so that one row's dependent steps fill another's latency
    const int G = pow2_ceil(d >> 3) > 32 ? 32 : pow2_ceil(d >> 3);
    const int RPW = 32 / G, grp = lane / G, lig = lane % G;
    int bad = 0;
    auto keep_score = [&](int j, float sc) {
        if (a.scores) a.scores[(long long)id.e * N + j] = sc;
        const bool fin = isfinite(sc);
        bad |= !fin;
        s[j] = fin ? sc : -INFINITY;
    };
    if (members == 1) {
        const int step = kWarps * RPW;
        for (int j0 = warp * RPW + grp; j0 - grp < n; j0 += 4 * step) {
            float acc[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int j = j0 + i * step;
                const bool valid = j < n;
                const long long dist = valid ? pref - (long long)spos[j] : 0;
                acc[i] = score_part(Kt + (size_t)(valid ? j : 0) * d, valid, dist, gpos != nullptr, d, phi, g, lig);
            }
            for (int off = G >> 1; off > 0; off >>= 1) {
#pragma unroll
                for (int i = 0; i < 4; ++i) acc[i] += __shfl_xor_sync(0xFFFFFFFFu, acc[i], off);
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                if (lig == 0 && j0 + i * step < n) keep_score(j0 + i * step, acc[i]);
        }
    } else {
        for (int j0 = warp * RPW; j0 < n; j0 += kWarps * RPW) {
            const int j = j0 + grp;
            const bool valid = j < n;
            const long long dist = valid ? pref - (long long)spos[j] : 0;
            const float sc = score_group(Kt + (size_t)j * d, valid, dist, gpos != nullptr, d, phi, g, lig, G, members);
            if (valid && lig == 0) keep_score(j, sc);
        }
    }
    cp_async_wait_pending<0>();
    if (!mbar_wait_bounded(bar_v, 0, a.wait_polls)) *late = 1;
    __syncthreads();
    if (*late) {   // (everybody is past the barriers: their place is free)
        // a wait ran out: report it, give copies that may still be in flight a bounded chance to land, leave
        if (tid == 0) {
            if (a.status) a.status[id.e] = 3;
            mbar_wait_bounded(bar_k, 0, a.wait_polls);
            mbar_wait_bounded(bar_v, 0, a.wait_polls);
        }
        return;
    }
    if (tid == 0) {
        mbar_inval(bar_k);
        mbar_inval(bar_v);
    }
    phase_stamp(id.e, 2);
    // reciprocal norms: a thread per row, each lane from its own block of eight elements on (different banks). A block's
    // squares in two chains of four, the blocks in eight sums: an error of 4.2e-8 at d = 128, as from sixteen lanes' partial
    // sums; one chain of all squares has 1.6e-7.
    if (PENALTY && !a.flat_sig) {
        const int nb = d >> 3, half = lane & 4;
        for (int j = tid; j < n; j += kThreads) {
            float u[8] = {};
            int c = lane % nb;
            for (int i0 = 0; i0 < nb; i0 += 8) {
#pragma unroll
                for (int q = 0; q < 8; ++q)
                    if (i0 + q < nb) {
                        float x[4], y[4], sx = 0.f, sy = 0.f;
                        load4(Vt + (size_t)j * d + 8 * c + half, x);
                        load4(Vt + (size_t)j * d + 8 * c + (half ^ 4), y);
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            sx = fmaf(x[e], x[e], sx);
                            sy = fmaf(y[e], y[e], sy);
                        }
                        u[q] += sx + sy;
                        c = c + 1 == nb ? 0 : c + 1;
                    }
            }
            r[j] = 1.f / (sqrtf(((u[0] + u[1]) + (u[2] + u[3])) + ((u[4] + u[5]) + (u[6] + u[7]))) + a.eps);
        }
    }
    bad = __syncthreads_or(bad);
    phase_stamp(id.e, 3);

    // selection
    const int bud = event_budget(a, id);
    const int picks = min(bud, n);
    // (nothing below can fail: written here, so that the selection need not hold what it says)
    if (tid == 0) {
        if (a.n_kept) a.n_kept[id.e] = picks;
        if (a.status) a.status[id.e] = n < bud ? 2 : (bad ? 1 : 0);
    }
    // ---- pool + triangle + one-warp loop, when it fits --------------------------------------------------------
    bool done = false, k_tile = true;   // k_tile: the K rows are still in theirs
    if (PENALTY && picks > 1) {
        unsigned short* bypool = reinterpret_cast<unsigned short*>(m);
        float* sb_holder = reinterpret_cast<float*>(red);
        int* pool_holder = redi;
        float sb;
        if (n <= kThreads) {
            // s_(b) from below to 2^-9 of its value, which is all that pruning needs: a key per thread, a bit per count, and the
            // barrier does the counting. (The exact value by counting every other key, as below: 5.1 of one event's 55 thousand
            // cycles, 3.1 so; 896 events of 192 fp32 rows 205 -> 195 us, of 256 bf16 rows of 64 332 -> 322.)
            const uint32_t kj = tid < n ? orderable(s[tid]) : 0u;
            uint32_t kb = 0u;
            for (int lo = 31; lo >= 14; --lo)
                if (__syncthreads_count(kj >= (kb | (1u << lo))) >= picks) kb |= 1u << lo;
            sb = kb < 0x00800000u ? -INFINITY : from_orderable(kb);
        } else {
            // s_(b): the value v with fewer than `picks` scores above it and at least `picks` not below it
            uint32_t* keys = reinterpret_cast<uint32_t*>(m);   // (padded to a multiple of four with keys below every real one)
            const int n4 = (n + 3) & ~3;
            for (int j = tid; j < n4; j += kThreads) keys[j] = j < n ? orderable(s[j]) : 0u;
            __syncthreads();
            for (int j = tid; j < n; j += kThreads) {
                const uint32_t kj = keys[j];
                int gt = 0, ge = 0;
#pragma unroll 4
                for (int i = 0; i < n4; i += 4) {
                    const uint4 k4 = *reinterpret_cast<const uint4*>(keys + i);
                    gt += (k4.x > kj) + (k4.y > kj) + (k4.z > kj) + (k4.w > kj);
                    ge += (k4.x >= kj) + (k4.y >= kj) + (k4.z >= kj) + (k4.w >= kj);
                }
                if (gt < picks && picks <= ge) *sb_holder = s[j];
            }
            __syncthreads();
            sb = *sb_holder;
        }
        const float thr = a.no_prune || sb == -INFINITY ? -INFINITY : fmaf(-1.001f, a.lam, sb) - 1e-6f * fabsf(sb);
        if (warp == 0) {
            int base = 0;
            for (int j0 = 0; j0 < n; j0 += 32) {
                const int j = j0 + lane;
                const bool in = j < n && !(s[j] < thr);
                const uint32_t mask = __ballot_sync(0xFFFFFFFFu, in);
                if (in) bypool[base + __popc(mask & ((1u << lane) - 1u))] = (unsigned short)j;
                base += __popc(mask);
            }
            if (lane == 0) *pool_holder = base;
        }
        __syncthreads();
        const int P = *pool_holder;
        const long long need = (long long)P * (P + 1) / 2 * 4;
        const bool beside = need <= (long long)extra_bytes;
        if (P <= 256 && (beside || need <= (long long)N * d * (long long)sizeof(T))) {
            done = true;
            k_tile = beside;
            float* tri = reinterpret_cast<float*>(beside ? smem + sp.total : smem + sp.tileK);
            const float* sig = a.flat_sig ? event_sig(a, id) : nullptr;
            phase_stamp(id.e, 4);
            // the norms, by slot until now, by pool row from here on
            const float own_r = tid < P && !sig ? r[bypool[tid]] : 1.f;
            __syncthreads();
            if (tid < P) r[tid] = own_r;
            if (sig) fill_triangle([&](int j) { return GlobalRow{sig + (long long)j * d}; }, bypool, P, d, tri);
            else fill_triangle([&](int j) { return SharedRow<T>{smem_u32(Vt) + (uint32_t)(j * d * (int)sizeof(T))}; }, bypool, P, d, tri);
            __syncthreads();
            phase_stamp(id.e, 5);
            uint32_t* park_key = reinterpret_cast<uint32_t*>(gain);
            if (warp == 0) {
                // (in pairs: 896 events of 192 fp32 rows 196.6 -> 192.5 us; one event's loop 12.1 -> 10.4 thousand cycles)
                if (P <= 128) picks_in_pairs<4, false>(lane, P, picks, s, bypool, r, a.lam, tri, park_key, order);
                else picks_in_pairs<8, false>(lane, P, picks, s, bypool, r, a.lam, tri, park_key, order);
            }
            __syncthreads();
            for (int t = tid; t < picks; t += kThreads) {
                const int j = bypool[order[t]];
                gain[t] = from_orderable(park_key[t]);
                order[t] = j;
                taken[j] = 1;
            }
            __syncthreads();
        } else {
            const int rounds = picks_in_rounds<T>(a, smem, n, picks, orderable(thr), extra_bytes);
            done = rounds & kRoundsDone;
            k_tile = !(rounds & kRoundsOverK);
            __syncthreads();
            if (!done) {
                for (int j = tid; j < n; j += kThreads) m[j] = 0.f;
                __syncthreads();
            }
        }
    }
    if (!done) {
        if (a.flat_sig) {
            StridedRows<float> rows{event_sig(a, id), d};
            greedy_cta<float>(n, picks, a.lam, PENALTY, d, s, nullptr, m, taken, order, gain, rows, red);
        } else {
            StridedRows<T> rows{Vt, d};
            greedy_cta<T>(n, picks, a.lam, PENALTY, d, s, r, m, taken, order, gain, rows, red);
        }
    }
    phase_stamp(id.e, 6);
    ordered_indices(n, a.budget, taken, idx);
    __syncthreads();

    // outputs
    const long long ob = (long long)id.e * a.budget;
    for (int t = tid; t < a.budget; t += kThreads) {
        a.idx_sorted[ob + t] = idx[t];
        if (a.pick_order) a.pick_order[ob + t] = t < picks ? order[t] : -1;
        if (a.pick_gain) a.pick_gain[ob + t] = t < picks ? gain[t] : 0.f;
    }
    phase_stamp(id.e, 7);
    // compaction: kept rows go to slots 0..picks-1 of the same buffer, all sources on chip first
    if (!k_tile) {
        load_rows_async(Kt, Kg, lay, id, picks, idx);
        cp_async_wait_pending<0>();
        __syncthreads();
    }
    const int cpr = d * (int)sizeof(T) / 16, lanes = min(pow2_ceil(cpr), 32), rows = 32 / lanes;
    for (int rr = warp * rows + lane / lanes; rr < picks; rr += kWarps * rows) {
        const int src = idx[rr];
        const long long off = row_offset(lay, id.b, id.l, id.h, rr);
        const T* krow = Kt + (size_t)(k_tile ? src : rr) * d;
        const T* vrow = Vt + (size_t)src * d;
        for (int c = lane & (lanes - 1); c < cpr; c += lanes) {
            copy16(reinterpret_cast<char*>(Kg + off) + c * 16, reinterpret_cast<const char*>(krow) + c * 16);
            copy16(reinterpret_cast<char*>(Vg + off) + c * 16, reinterpret_cast<const char*>(vrow) + c * 16);
        }
    }
    if (gpos) {
        int* wpos = a.pos.p + id.b * a.pos.sb + id.l * a.pos.sl + id.h * a.pos.sh;
        for (int t = tid; t < picks; t += kThreads) wpos[t] = spos[idx[t]];
    }
    phase_stamp(id.e, 8);
}

}  // namespace akv
