// Scores of the fused on-chip kernels (bf16, d = 128): eight lanes per key row, eight frequencies per
// lane, the rotation of the query statistic carried from row to row.
#pragma once
#include "akv_kernels.cuh"

namespace akv {

// (cos, sin) of the angle 2 pi ph / 2^32: nearest of the 32 sector angles from the shared-memory table,
// remainder (in units of 2 pi / 2^37, to the last place: with 4.5716245e-11, 1.2e-6 off, a carried turn was off by up to 1.2e-7,
// and scores by 3.1e-7 of their size, 2-norm over 2-norm, instead of 1.8e-7 at chains of eight) by the short polynomials of score_lane8
__device__ __forceinline__ float2 phase_cos_sin(uint32_t ph, const float2* sect) {
    const float2 e = sect[(ph + 0x04000000u) >> 27];
    const float w = (float)(int32_t)(ph << 5) * 4.571619e-11f, z = w * w;
    const float sw = w * fmaf(z, fmaf(z, 8.3333333e-3f, -0.16666667f), 1.f);
    const float cw = fmaf(z, fmaf(z, 4.1666667e-2f, -0.5f), 1.f);
    return make_float2(e.x * cw - e.y * sw, e.y * cw + e.x * sw);
}
// bits 32..63 of dist * phi (mod 2^64) for a signed 64-bit distance: the angle dist * theta_f in 2^-32 turns
__device__ __forceinline__ uint32_t phase_of(long long dist, unsigned long long phi) {
    const uint32_t dl = (uint32_t)dist, dh = (uint32_t)((unsigned long long)dist >> 32);
    const uint32_t pl = (uint32_t)phi, ph = (uint32_t)(phi >> 32);
    return __umulhi(dl, pl) + dl * ph + dh * pl;
}

// Scoring state of a lane: the folded statistic already turned to the row at hand,
// G_f = g_f e^{i dist theta_f} for the lane's eight frequencies, so that a row's score is
// sum_f Re(G_f conj(k_f)); and the turn S_f = e^{-i D theta_f} that takes G from one row of a lane
// group to its next one when the two rows' positions differ by D (rows 16 slots apart: D = 16 for a
// cache filled token by token). G is taken afresh (sector table + polynomials) whenever the spacing is
// not D, and every kChainRounds-th (kChainRoundsShort-th) round in any case: a chained complex product adds
// about 3e-9 of the score's scale to the error (fp32 summation of the 64 terms gives 4e-8 by itself; a chain
// of twelve products measured 8e-8 in all).
struct ChainScore {
    float2 Gx[4], Gy[4], Sx[4], Sy[4], nSy[4];
    // S from D (any sign); phitab: phi_f for the lane's frequencies (shared memory)
    __device__ __forceinline__ void set_step(long long D, const unsigned long long* phitab, const float2* sect) {
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float2 e = phase_cos_sin(phase_of(-D, phitab[u]), sect);
            if (u & 1) { Sx[u >> 1].y = e.x; Sy[u >> 1].y = e.y; nSy[u >> 1].y = -e.y; }
            else { Sx[u >> 1].x = e.x; Sy[u >> 1].x = e.y; nSy[u >> 1].x = -e.y; }
        }
    }
    // G afresh for a row at distance dist (any sign); gtab: folded statistic g_f for the lane's frequencies
    __device__ __forceinline__ void anchor(long long dist, const float2* gtab, const unsigned long long* phitab,
                                           const float2* sect) {
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const float4 g2 = *reinterpret_cast<const float4*>(gtab + 2 * p);       // g of frequencies 2p, 2p + 1
            const ulonglong2 ph = *reinterpret_cast<const ulonglong2*>(phitab + 2 * p);
            const float2 ea = phase_cos_sin(phase_of(dist, ph.x), sect), eb = phase_cos_sin(phase_of(dist, ph.y), sect);
            Gx[p] = make_float2(g2.x * ea.x - g2.y * ea.y, g2.z * eb.x - g2.w * eb.y);
            Gy[p] = make_float2(g2.x * ea.y + g2.y * ea.x, g2.z * eb.y + g2.w * eb.x);
        }
    }
    __device__ __forceinline__ void advance() {
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const float2 nx = __ffma2_rn(Gy[p], nSy[p], __fmul2_rn(Gx[p], Sx[p]));
            const float2 ny = __ffma2_rn(Gy[p], Sx[p], __fmul2_rn(Gx[p], Sy[p]));
            Gx[p] = nx; Gy[p] = ny;
        }
    }
    // the same turn, taken from another state's S (two rows of a lane group chained side by side share one S)
    __device__ __forceinline__ void advance_by(const ChainScore& o) {
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            const float2 nx = __ffma2_rn(Gy[p], o.nSy[p], __fmul2_rn(Gx[p], o.Sx[p]));
            const float2 ny = __ffma2_rn(Gy[p], o.Sx[p], __fmul2_rn(Gx[p], o.Sy[p]));
            Gx[p] = nx; Gy[p] = ny;
        }
    }
    // the row that another state is at
    __device__ __forceinline__ void turn_to(const ChainScore& o) {
#pragma unroll
        for (int p = 0; p < 4; ++p) { Gx[p] = o.Gx[p]; Gy[p] = o.Gy[p]; }
    }
    // the lane's partial sum of Re(G conj(k)) over its 8 frequencies
    __device__ __forceinline__ float dot(const uint4& wr, const uint4& wi) const {
        const uint32_t wre[4] = {wr.x, wr.y, wr.z, wr.w}, wim[4] = {wi.x, wi.y, wi.z, wi.w};
        float2 acc2 = make_float2(0.f, 0.f);
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            acc2 = __ffma2_rn(Gx[p], make_float2(bf16lo(wre[p]), bf16hi(wre[p])), acc2);
            acc2 = __ffma2_rn(Gy[p], make_float2(bf16lo(wim[p]), bf16hi(wim[p])), acc2);
        }
        return acc2.x + acc2.y;
    }
    // the same sum with four independent accumulators (a chain of two dependent products instead of eight)
    __device__ __forceinline__ float dot4(const uint4& wr, const uint4& wi) const {
        const uint32_t wre[4] = {wr.x, wr.y, wr.z, wr.w}, wim[4] = {wi.x, wi.y, wi.z, wi.w};
        float2 acc[4];
#pragma unroll
        for (int p = 0; p < 4; ++p)
            acc[p] = __ffma2_rn(Gy[p], make_float2(bf16lo(wim[p]), bf16hi(wim[p])),
                                __fmul2_rn(Gx[p], make_float2(bf16lo(wre[p]), bf16hi(wre[p]))));
        const float2 a01 = __fadd2_rn(acc[0], acc[1]), a23 = __fadd2_rn(acc[2], acc[3]);
        const float2 a = __fadd2_rn(a01, a23);
        return a.x + a.y;
    }
};
constexpr int kChainRounds = 8;        // rounds between two fresh computations of G (long events, streamed)
constexpr int kChainRoundsShort = 16;  // the same for events of at most 256 rows: one or two fresh computations per lane
                                       // group; fifteen chained products add 1e-7 of the score's scale at most

// The 32 sector angles' cosines and sines, written by one warp: sect[h] = (cos, sin)(2 pi h / 32)
__device__ __forceinline__ void fill_sector_table(float2* sect, int lane) {
    float sn, cs;
    sincospif((float)lane * 0.0625f, &sn, &cs);
    sect[lane] = make_float2(cs, sn);
}
// Folded statistic g_f = c_f z(q)_f / sqrt(d) of (layer, KV head) lh and the frequencies' phase steps for d = 128, written
// by threads 0..63 into gtab[64] and phitab[64]. Several query heads per KV head: the statistic is their mean (the score
// is linear in it, so this is the mean of their scores; the maximum of them has no such form and takes other kernels).
__device__ __forceinline__ void fill_statistic_tables(const EventArgs& a, int lh, const ScoreTab& tab, int tid, float2* gtab,
                                                      unsigned long long* phitab) {
    if (tid < 64) {
        const int G = a.gqa_group;
        const float* q = a.qstat + (long long)lh * G * 128;
        float qr = q[tid], qi = q[tid + 64];
        for (int m = 1; m < G; ++m) {
            qr += q[m * 128 + tid];
            qi += q[m * 128 + tid + 64];
        }
        const float inv = rsqrtf(128.f) / (float)max(G, 1);
        qr *= inv;
        qi *= inv;
        const float2 c = tab.cw[tid];
        gtab[tid] = make_float2(c.x * qr - c.y * qi, c.x * qi + c.y * qr);
        phitab[tid] = tab.phi[tid];
    }
}

// ---------------------------------------------------------------------------------------------
// Stand-alone score for bf16, d = 128 (score_kernel, akv_kernels.cuh, takes the rest): one CTA per (event, block of 256
// rows), K streamed from global memory once, the next 64 rows requested before the present ones are scored. A lane group
// scores two rows of every 64 side by side, rotations from the sector table. They are taken afresh for every row: carried on
// over four rows they cost 7 us less of 137 (448 events of 1000 rows, score, selection and compaction), but the scores' error
// rises by half (from 1.2e-7 to 1.8e-7 when that was measured, with the remainder's constant of then; 9.6e-8 as they are now, score_kernel,
// which took 44 us more, 1.4e-7).
// Dense and paged layouts are instantiations of their own (58.3 -> 57.7 us of those calls).
// ---------------------------------------------------------------------------------------------
constexpr int kScoreRows128 = 256;
template <bool PAGED>
__global__ void __launch_bounds__(kThreads, 3) score_rows_kernel(const EventArgs a, const __grid_constant__ ScoreTab tab) {
    __shared__ __align__(16) float2 gtab[64];
    __shared__ __align__(16) unsigned long long phitab[64];
    __shared__ float2 sect[32];
    __shared__ int spos[kScoreRows128];
    __shared__ int redi[kWarps];
    const DevLayout& lay = a.lay;
    const int row_blocks = (lay.N + kScoreRows128 - 1) / kScoreRows128;
    const EventId id = decode_event(lay, blockIdx.x / row_blocks);
    const int n = event_n(a, id.b);
    const int row0 = (blockIdx.x % row_blocks) * kScoreRows128;
    if (row0 >= n) return;
    const int rows = min(kScoreRows128, n - row0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int* gpos = event_pos(a.pos, id);
    const bool rotate = gpos != nullptr;
    constexpr bool dense = !PAGED;
    const __nv_bfloat16* Kg = reinterpret_cast<const __nv_bfloat16*>(a.K) + (lane & 7) * 8;
    const long long ev_off = dense ? id.b * lay.sb + id.l * lay.sl + id.h * lay.sh : 0;
    // this lane's pieces of rows j and j + 32 of a stage (rows beyond the block read its last one, which is not used)
    const int ja0 = 4 * warp + (lane >> 3);
    auto request = [&](int st, uint4 (&k)[4]) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int j = row0 + min(64 * st + ja0 + 32 * h, rows - 1);
            const __nv_bfloat16* p = Kg + (dense ? ev_off + (long long)j * lay.sn : row_offset(lay, id.b, id.l, id.h, j));
            k[2 * h] = __ldcs(reinterpret_cast<const uint4*>(p));
            k[2 * h + 1] = __ldcs(reinterpret_cast<const uint4*>(p + 64));
        }
    };
    uint4 cur[4];
    request(0, cur);
    if (warp == 1) fill_sector_table(sect, lane);
    fill_statistic_tables(a, id.l * lay.H + id.h, tab, tid, gtab, phitab);
    if (tid < rows) spos[tid] = rotate ? gpos[row0 + tid] : 0;
    long long pref = 0;
    if (rotate) {
        if (a.p_ref) pref = a.p_ref[id.b];
        else {
            int pmax = INT_MIN;
            for (int j = tid; j < n; j += kThreads) pmax = max(pmax, gpos[j]);
            pref = (long long)block_max_int(pmax, redi) + 1;
        }
    }
    __syncthreads();
    const int f0 = (lane & 7) * 8;
    ChainScore ca, cb;   // (their rotations only, no chain)
    if (!rotate) {       // keys that are rotated already: the statistic itself, for every row
        ca.anchor(0, gtab + f0, phitab + f0, sect);
        cb = ca;
    }
    int bad = 0;
    for (int st = 0; 64 * st < rows; ++st) {
        uint4 next[4];
        if (64 * (st + 1) < rows) request(st + 1, next);
        const int ja = 64 * st + ja0, jb = ja + 32;
        if (rotate) {
            ca.anchor(pref - (long long)spos[min(ja, rows - 1)], gtab + f0, phitab + f0, sect);
            cb.anchor(pref - (long long)spos[min(jb, rows - 1)], gtab + f0, phitab + f0, sect);
        }
        const float acca = ca.dot4(cur[0], cur[1]), accb = cb.dot4(cur[2], cur[3]);
        // both rows' sums in three exchanges: lanes 0..3 of a group go on with the first, lanes 4..7 with the second
        const bool second = lane & 4;
        float acc = (second ? accb : acca) + __shfl_xor_sync(0xFFFFFFFFu, second ? acca : accb, 4);
        acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 2);
        acc += __shfl_xor_sync(0xFFFFFFFFu, acc, 1);
        const int j = second ? jb : ja;
        if ((lane & 3) == 0 && j < rows) {
            a.scores[(long long)id.e * lay.N + row0 + j] = acc;
            bad |= !isfinite(acc);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) cur[i] = next[i];
    }
    if (a.status) {
        bad = __syncthreads_or(bad);
        if (tid == 0 && bad) atomicMax(a.status + id.e, 1);
    }
}

}  // namespace akv
