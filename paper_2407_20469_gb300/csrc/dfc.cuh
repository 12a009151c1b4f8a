// dfc.cuh - darkfield spectrum extension (WSI-APIC Eq. 11-13) of tiles up to 256 pixels
// by a thread-block cluster, with the band grids in the cluster's shared memory.
//
// The method, grids, transforms and the order of every sum are those of kernels_dfr.cu
// (one block per tile), so a tile's result is bit for bit the same; this kernel is for
// batches that leave SMs idle there. A tile is solved by K blocks (3 to 8): block r owns a
// contiguous share of the grid's columns, of the Q rows and of the U rows.
//  * No band grid of the CG leaves the cluster: a pass reads its rows or columns from the
//    block's own shared memory and stores its results straight into the shared memory of
//    the blocks that own them for the next pass (st.shared::cluster), so the transpose
//    between a rows and a columns pass costs one cluster barrier and no round trip
//    through L2. The slabs keep the owner's rows (columns) innermost with an odd
//    stride: a half-warp's 16 stores are 128 consecutive bytes of one or two owners, its
//    16 loads fall in different banks.
//  * The known field of the block's columns stays in tensor memory (no MMA is issued).
//  * Every block keeps the CG vectors whole: the rows pass that gathers w stores it into
//    every block, and all blocks take the same steps, their inner products formed as 16
//    warps of one block form them. No scalar crosses blocks; an iteration has five
//    cluster barriers, one behind each pass.
// What bounds it: the chain of five passes per iteration, each a half-warp's one or two
// transforms deep (about 1.6 k cycles each), and the barriers (about 1 k each). Measured
// (GB300, darkfield stage of one tile, 8 + 16 images): 128 pixels 5.0 -> 2.7 ms, 256 pixels
// 14.6 -> 4.3 ms with 8 blocks. With the grids in L2 instead (the one-block kernel's passes
// split over a cluster) the same tiles took 4.9 and 8.3 ms: the release of every barrier
// waits for the stores to reach L2, and each pass then loads from there. More than 8
// blocks gain nothing: a share is then less than a half-warp's transform each.
#pragma once

#include <math.h>

#include <algorithm>

#include "../../include/apic.h"
#include "cluster.cuh"
#include "internal.cuh"
#include "regfft.cuh"
#include "t4grid.cuh"
#include "tmem.cuh"

namespace apic {

constexpr int kClThreads = 320;                 // 20 half-warps: the 18-20 columns, 16-17 Q rows of a share of 1/8 (256 px)
constexpr int kClHW = kClThreads / 16;
constexpr int kClTmemCols = 512;
constexpr int kClQWords = 8;                    // Q membership words per band row (two 16-bit masks each)
constexpr int kClTmemSlot = 160;                // TMEM columns per thread: 10 warps, three per lane quarter

// Shared memory of one block (byte offsets, 16-aligned). The half-warp areas of the
// camera-grid setup transforms alias the CG's areas, vectors and slabs up to cq; the cq
// slab is apart (it receives the known field's rows, then b's, while the setup runs).
// cu: U rows' columns on their way into C1, then the U rows out of C2; the two are never
// live together. urp, ux, qm: the image's U row pointers, the points' positions on the row
// grid, and the Q masks of the block's rows - the acquire of a cluster barrier drops the
// L1 cache, so tables in global memory cost each pass an L2 round trip or two.
struct ClSmem {
    size_t vec, cu, rq, cq, tw, tab, urp, ux, qm, red, total;
};

__host__ __device__ inline size_t cl_align(size_t b) { return (b + 15) & ~(size_t)15; }
__host__ __device__ inline int cl_share(int n, int K) { return (n + K - 1) / K; }
__host__ __device__ inline size_t cl_max(size_t a, size_t b) { return a > b ? a : b; }

// maxB: largest row or column grid / 16 of the used images; mx: their largest row grid
__host__ __device__ inline ClSmem cl_smem_layout(int BN, int B, int K, int maxB, int mx, int band_u, int band_p,
                                                 int band_q, int max_N) {
    ClSmem L;
    const size_t c = sizeof(float2);
    const int lc = cl_share(mx, K) | 1, lu = cl_share(band_u, K) | 1, lq = cl_share(band_q, K) | 1;
    L.vec = cl_align((size_t)kClHW * hw_single_size(maxB) * c);
    L.cu = L.vec + cl_align((size_t)4 * max_N * c);
    L.rq = L.cu + cl_align(cl_max((size_t)band_u * lc, (size_t)mx * lu) * c);
    const size_t cg_end = L.rq + cl_align((size_t)mx * lq * c);
    const size_t setup = cl_align((size_t)kClHW * hw_single_size(BN > B ? BN : B) * c);
    L.cq = cl_max(cg_end, setup);
    L.tw = L.cq + cl_align((size_t)(band_q > band_p ? band_q : band_p) * lc * c);
    L.tab = L.tw + cl_align((size_t)2 * 16 * (BN + B + 2 * maxB) * c);
    L.urp = L.tab + cl_align((size_t)(mx + band_q + band_u) * sizeof(uint32_t));
    L.ux = L.urp + cl_align((size_t)(band_u + 1) * sizeof(int));
    L.qm = L.ux + cl_align((size_t)max_N * sizeof(uint16_t));
    L.red = L.qm + cl_align((size_t)cl_share(band_q, K) * kClQWords * sizeof(unsigned));
    L.total = L.red + 64 * sizeof(double);
    return L;
}

// Global scratch of a cluster: the known field's rows on the register grid m (tiled), the
// image's column transforms (column by column), P * P's columns (Q rows, tiled), b on Q
struct ClScratch {
    size_t gx, rb, bq, total;       // values
};
__host__ __device__ inline ClScratch cl_scratch_layout(int n, int m, int band_p, int band_q, int max_M) {
    ClScratch S;
    S.gx = (size_t)t4_rows(band_p) * m;
    S.rb = S.gx + (size_t)n * band_q;
    S.bq = (S.rb + 15) / 16 * 16 + (size_t)t4_rows(band_q) * m;
    S.rb = (S.rb + 15) / 16 * 16;
    S.total = S.bq + max_M;
    return S;
}

namespace {

__device__ __forceinline__ int sfreqc(int i, int n) { return i < n / 2 ? i : i - n; }

// the cluster-wide address of a shared-memory address of this block in block `rank`
__device__ __forceinline__ uint32_t cl_map(uint32_t a, uint32_t rank) {
    uint32_t r;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cl_st(uint32_t a, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void cl_sync() { tile_sync<true>(); }

// Half-warp hw of the block, lane t; hs its transform area; tm the thread's TMEM columns.
struct ClLane {
    int t, hw;
    unsigned mask;
    uint32_t tm;
    float2* hs;
    __device__ HalfWarp h() const { return HalfWarp{t, mask, hs}; }
};

// Where a pass stores: element i of the next pass's owners' lists (rows or columns) at
// tab[i] + off, plus a multiple of `step` bytes for the other coordinate.
struct ClDst {
    const uint32_t* tab;
    uint32_t off;
    int step;
};

// ---- per-point functors
struct ClValKnown {      // P(c) = O_known(K) exp(j phi(c)); the spectrum is written by any block: from L2
    const float2* sp;
    const float* ph;
    const int* ap;
    const int* pup;
    __device__ float2 operator()(int e) const {
        float sn, cs;
        sincosf(ph[pup[e]], &sn, &cs);
        return cmul(__ldcg(sp + ap[e]), make_float2(cs, sn));
    }
};
// ---- per-column operations on o[s][k1], the value at y = (t + 16 s) + B k1
template <int B>
struct ClMidStore {      // p s W^(shift y) into the thread's TMEM columns (wt: W_16B^j)
    float scale;
    const float2* wt;
    int shift;
    static constexpr bool kOut = false;
    __device__ void operator()(float2 (&o)[Slots<B>::value][16], int t, uint32_t tm) const {
        constexpr int m = 16 * B;
#pragma unroll
        for (int s = 0; s < Slots<B>::value; ++s) {
            const int u = t + 16 * s < B ? t + 16 * s : 0;
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) o[s][k1] = cscale(cmul(o[s][k1], wt[(shift * (u + B * k1)) % m]), scale);
            tmem_st16(tm + 32 * s, o[s]);
        }
        tmem_wait_st();
    }
};
template <int B, bool CONJ>
struct ClMidTimes {      // o *= p s or conj(p s)
    static constexpr bool kOut = true;
    __device__ void operator()(float2 (&o)[Slots<B>::value][16], int, uint32_t tm) const {
#pragma unroll
        for (int s = 0; s < Slots<B>::value; ++s) {
            float2 p[16];
            tmem_ld16(tm + 32 * s, p);
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) o[s][k1] = CONJ ? cmulc(o[s][k1], p[k1]) : cmul(o[s][k1], p[k1]);
        }
    }
};

// ---- passes

// rows r0 .. r0 + nr - 1 of a band: scatter val(e) at x = px[e], inverse transform along
// x, store to the column owners (column x at row b: dst.tab[x] + dst.off + b dst.step).
template <int B, class Val>
__device__ __noinline__ void cl_rows_in(ClLane w, const float2* tw, int r0, int nr, const int* rp, const int* px,
                                        Val val, ClDst dst) {
    constexpr int m = 16 * B, S = Slots<B>::value;
    const HalfWarp h = w.h();
    for (int b = r0 + w.hw; b < r0 + nr; b += kClHW) {
#pragma unroll
        for (int j = 0; j < B; ++j) w.hs[w.t + 16 * j] = make_float2(0.f, 0.f);
        __syncwarp(w.mask);
        for (int e = rp[b] + w.t; e < rp[b + 1]; e += 16) w.hs[freq_index(px[e], m)] = val(e);
        __syncwarp(w.mask);
        float2 v[B], o[S][16];
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = w.hs[w.t + 16 * j];
        __syncwarp(w.mask);
        fft_a<B, true>(v, o, h, tw);
        const uint32_t at = dst.off + b * dst.step;
#pragma unroll
        for (int s = 0; s < S; ++s)
            if (w.t + 16 * s < B) {
#pragma unroll
                for (int k1 = 0; k1 < 16; ++k1) cl_st(dst.tab[w.t + 16 * s + B * k1] + at, o[s][k1]);
            }
    }
}

// the block's U rows of the direction d: as cl_rows_in with the tables in shared memory
template <int B>
__device__ __noinline__ void cl_rows_dir(ClLane w, const float2* tw, int r0, int nr, const int* urp, const uint16_t* ux,
                                         const float2* dv, ClDst dst) {
    const HalfWarp h = w.h();
    for (int b = r0 + w.hw; b < r0 + nr; b += kClHW) {
#pragma unroll
        for (int j = 0; j < B; ++j) w.hs[w.t + 16 * j] = make_float2(0.f, 0.f);
        __syncwarp(w.mask);
        const int e1 = urp[b + 1];
        for (int e = urp[b] + w.t; e < e1; e += 16) w.hs[ux[e]] = dv[e];
        __syncwarp(w.mask);
        float2 v[B], o[1][16];
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = w.hs[w.t + 16 * j];
        __syncwarp(w.mask);
        fft_a<B, true>(v, o, h, tw);
        const uint32_t at = dst.off + b * dst.step;
        if (w.t < B) {
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) cl_st(dst.tab[w.t + B * k1] + at, o[0][k1]);
        }
    }
}

// the known field's rows on the register grid, into the tiled grid GP in global scratch
// (every block reads its columns from L2)
template <int B>
__device__ __noinline__ void cl_rows_known(ClLane w, const float2* tw, int r0, int nr, const int* rp, const int* px,
                                           ClValKnown val, float2* GP) {
    constexpr int m = 16 * B, S = Slots<B>::value;
    const HalfWarp h = w.h();
    const T4Lane L(w.t);
    for (int b = r0 + w.hw; b < r0 + nr; b += kClHW) {
#pragma unroll
        for (int j = 0; j < B; ++j) w.hs[w.t + 16 * j] = make_float2(0.f, 0.f);
        __syncwarp(w.mask);
        for (int e = rp[b] + w.t; e < rp[b + 1]; e += 16) w.hs[freq_index(px[e], m)] = val(e);
        __syncwarp(w.mask);
        float2 v[B], o[S][16];
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = w.hs[w.t + 16 * j];
        __syncwarp(w.mask);
        fft_a<B, true>(v, o, h, tw);
        float2* row = GP + t4_row(b, m);
#pragma unroll
        for (int s = 0; s < S; ++s)
            if (w.t + 16 * s < B) {
#pragma unroll
                for (int k1 = 0; k1 < 16; ++k1) row[L.at(16 * s + B * k1)] = o[s][k1];
            }
    }
}

// the block's nc columns (grid columns c0 ..; `rounds` rounds of the block's half-warps,
// the same for every warp): the ni band rows of the slab G[row][column] (stride ld) are
// the input at column indices 0..ni - 1, the rest zero; inverse along y, mid, and
// (Mid::kOut) forward along y, column indices 0..no - 1 stored to the row owners
// (row b, column x: dst.tab[b] + dst.off + x dst.step). Bands are taken from row 0;
// the field carries the ramp of their true starts (see wpass_cols in kernels_dfw.cu).
template <int B, class Mid>
__device__ __noinline__ void cl_cols(ClLane w, const float2* tw, int rounds, int c0, int nc, const float2* G, int ld,
                                     int ni, int no, Mid mid, ClDst dst) {
    constexpr int S = Slots<B>::value;
    const HalfWarp h = w.h();
    for (int r = 0; r < rounds; ++r) {
        const int xl = w.hw + r * kClHW;
        const bool mine = xl < nc;
        float2 v[B], o[S][16];
#pragma unroll
        for (int j = 0; j < B; ++j)
            v[j] = mine && w.t + 16 * j < ni ? G[(w.t + 16 * j) * ld + xl] : make_float2(0.f, 0.f);
        fft_a<B, true>(v, o, h, tw);
        __syncwarp();
        mid(o, w.t, w.tm + 32 * S * r);
        if constexpr (Mid::kOut) {
            fft_b<B, false>(o, v, h, tw);
            const uint32_t at = dst.off + (c0 + xl) * dst.step;
#pragma unroll
            for (int k1 = 0; k1 < B; ++k1)
                if (mine && w.t + 16 * k1 < no) cl_st(dst.tab[w.t + 16 * k1] + at, v[k1]);
        }
    }
}

// the block's Q rows: forward along x, keep the Q lags (qmask: per row of the block, words of
// two 16-bit masks, bit k1 of mask t for x index t + B k1), inverse along x.
template <int B>
__device__ __noinline__ void cl_rows_mask(ClLane w, const float2* tw, int r0, int nr, const float2* G, int ld,
                                          const unsigned* qmask, ClDst dst) {
    constexpr int S = Slots<B>::value;
    const HalfWarp h = w.h();
    for (int i = w.hw; i < nr; i += kClHW) {
        const int b = r0 + i;
        unsigned qw[S];
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int ls = w.t + 16 * s;
            qw[s] = ls < B ? qmask[i * kClQWords + (ls >> 1)] >> (16 * (ls & 1)) : 0u;
        }
        float2 v[B], o[S][16];
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = G[(w.t + 16 * j) * ld + i];
        fft_a<B, false>(v, o, h, tw);
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1)
                if (!((qw[s] >> k1) & 1u)) o[s][k1] = make_float2(0.f, 0.f);
        fft_b<B, true>(o, v, h, tw);
        const uint32_t at = dst.off + b * dst.step;
#pragma unroll
        for (int k1 = 0; k1 < B; ++k1) cl_st(dst.tab[w.t + 16 * k1] + at, v[k1]);
    }
}

// the block's U rows: forward along x, the values at the U points into entry e of w in
// every block (wT: w's address in block t's shared memory, lanes t < K)
template <int B>
__device__ __noinline__ void cl_rows_out(ClLane w, const float2* tw, int r0, int nr, const float2* G, int ld,
                                         const int* urp, const uint16_t* ux, uint32_t wa, int K) {
    constexpr int S = Slots<B>::value;
    const HalfWarp h = w.h();
    for (int i = w.hw; i < nr; i += kClHW) {
        const int b = r0 + i;
        float2 v[B], o[S][16];
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = G[(w.t + 16 * j) * ld + i];
        fft_a<B, false>(v, o, h, tw);
#pragma unroll
        for (int s = 0; s < S; ++s)
            if (w.t + 16 * s < B) {
#pragma unroll
                for (int k1 = 0; k1 < 16; ++k1) w.hs[w.t + 16 * s + B * k1] = o[s][k1];
            }
        __syncwarp(w.mask);
        const int e1 = urp[b + 1];
        for (int e = urp[b] + w.t; e < e1; e += 16) {
            const float2 val = w.hs[ux[e]];
            for (int r = 0; r < K; ++r) cl_st(cl_map(wa + 8 * e, r), val);
        }
        __syncwarp(w.mask);
    }
}

// the block's columns x0 .. x0 + nx - 1 of the image (n = 16 BN): forward along y, the Q
// rows to GX[x][row] (nQ rows). The image is read through L1: neighbouring half-warps take
// neighbouring columns, which share sectors (tr: the image transposed, rows are contiguous).
template <int BN>
__device__ __noinline__ void cl_image_cols(ClLane w, const float2* tw, int x0, int nx, const float* __restrict__ img,
                                           int qy0, int nQ, bool tr, float2* GX) {
    constexpr int n = 16 * BN;
    const HalfWarp h = w.h();
    for (int x = x0 + w.hw; x < x0 + nx; x += kClHW) {
        float2 v[BN], o[1][16];
#pragma unroll
        for (int j = 0; j < BN; ++j) {
            const int y = w.t + 16 * j;
            v[j] = make_float2(__ldg(img + (tr ? (size_t)x * n + y : (size_t)y * n + x)), 0.f);
        }
        fft_a<BN, false>(v, o, h, tw);
        if (w.t < BN) {
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) {
                const int b = sfreqc(w.t + BN * k1, n) - qy0;
                if (b >= 0 && b < nQ) GX[(size_t)x * nQ + b] = o[0][k1];
            }
        }
    }
}

// the block's Q rows of the image's spectrum: forward along x, b = value / n^2 at the Q points
template <int BN>
__device__ __noinline__ void cl_image_rows(ClLane w, const float2* tw, int r0, int nr, const float2* GX, int nQ,
                                           const int* qrp, const int* Qx, float2* bq) {
    constexpr int n = 16 * BN;
    const HalfWarp h = w.h();
    const float inv_n2 = 1.f / (float)(n * n);
    for (int b = r0 + w.hw; b < r0 + nr; b += kClHW) {
        float2 v[BN], o[1][16];
#pragma unroll
        for (int j = 0; j < BN; ++j) v[j] = __ldcg(GX + (size_t)(w.t + 16 * j) * nQ + b);
        fft_a<BN, false>(v, o, h, tw);
        if (w.t < BN) {
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) w.hs[w.t + BN * k1] = o[0][k1];
        }
        __syncwarp(w.mask);
        for (int e = qrp[b] + w.t; e < qrp[b + 1]; e += 16) bq[e] = cscale(w.hs[freq_index(Qx[e], n)], inv_n2);
        __syncwarp(w.mask);
    }
}

// the block's columns of |p|^2 on the register grid (m = 16 B): p's column from the nP band
// rows in(b, x), inverse along y, |p|^2 W^(shift y), forward along y, the Q rows to RB (tiled)
template <int B, class In>
__device__ __noinline__ void cl_cols_abs2(ClLane w, const float2* tw, int x0, int nx, In in, int nP, float2* RB, int nQ,
                                          const float2* wt, int shift) {
    constexpr int m = 16 * B;
    const HalfWarp h = w.h();
    for (int xl = w.hw; xl < nx; xl += kClHW) {
        const int x = x0 + xl;
        float2 v[B], o[1][16];
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = w.t + 16 * j < nP ? in(w.t + 16 * j, x, xl) : make_float2(0.f, 0.f);
        fft_a<B, true>(v, o, h, tw);
        if (w.t < B) {
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) o[0][k1] = cscale(wt[(shift * (w.t + B * k1)) % m], cabs2(o[0][k1]));
        }
        fft_b<B, false>(o, v, h, tw);
        float2* go = RB + t4_row(w.t, m) + t4_col(x);
#pragma unroll
        for (int k1 = 0; k1 < B; ++k1)
            if (w.t + 16 * k1 < nQ) go[16 * k1 * m] = v[k1];
    }
}

// the block's Q rows of P * P: forward along x on the register grid (16 B points), b -= value
// / m^2 at the Q points, then b's rows inverse along x on the row grid (16 BX points), stored
// to the column owners
template <int B, int BX>
__device__ __noinline__ void cl_rows_rhs(ClLane w, const float2* tw_m, const float2* tw, int r0, int nr,
                                         const float2* RB, const int* qrp, const int* Qx, const float2* bq, ClDst dst) {
    constexpr int m = 16 * B, mx = 16 * BX;
    const HalfWarp h = w.h();
    const float inv_m2 = 1.f / (float)(m * m);
    for (int b = r0 + w.hw; b < r0 + nr; b += kClHW) {
        {
            const float2* row = RB + t4_row(b, m) + t4_col(w.t);
            float2 v[B], o[1][16];
#pragma unroll
            for (int j = 0; j < B; ++j) v[j] = __ldcg(row + 64 * j);
            fft_a<B, false>(v, o, h, tw_m);
            if (w.t < B) {
#pragma unroll
                for (int k1 = 0; k1 < 16; ++k1) w.hs[w.t + B * k1] = o[0][k1];
            }
        }
        __syncwarp(w.mask);
        // the row's points (at most 16 BX) through registers, then onto the row grid
        const int e0 = qrp[b] + w.t, e1 = qrp[b + 1];
        float2 q[BX];
        int xq[BX];
#pragma unroll
        for (int j = 0; j < BX; ++j) {
            const int e = e0 + 16 * j;
            xq[j] = e < e1 ? Qx[e] : 0;
            q[j] = e < e1 ? csub(bq[e], cscale(w.hs[freq_index(xq[j], m)], inv_m2)) : make_float2(0.f, 0.f);
        }
        __syncwarp(w.mask);
#pragma unroll
        for (int j = 0; j < BX; ++j) w.hs[w.t + 16 * j] = make_float2(0.f, 0.f);
        __syncwarp(w.mask);
#pragma unroll
        for (int j = 0; j < BX; ++j)
            if (e0 + 16 * j < e1) w.hs[freq_index(xq[j], mx)] = q[j];
        __syncwarp(w.mask);
        float2 v[BX], o[1][16];
#pragma unroll
        for (int j = 0; j < BX; ++j) v[j] = w.hs[w.t + 16 * j];
        __syncwarp(w.mask);
        fft_a<BX, true>(v, o, h, tw);
        const uint32_t at = dst.off + b * dst.step;
        if (w.t < BX) {
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) cl_st(dst.tab[w.t + BX * k1] + at, o[0][k1]);
        }
    }
}

// Inner products in the order of a block of 512 threads (kernels_dfr.cu): part(v, lane) is
// the FP32 sum of lane `lane` of its warp v; each warp's 32 lanes in FP32, the 16 warps in
// FP64 (warp 0). The quotient of the sum and `num` (OVER: sum / num, else num / sum)
// rounded to FP32. Every thread gets both; red: 64 doubles, used in turns (parity).
constexpr int kRefWarps = 16;

template <bool OVER, class Part>
__device__ __forceinline__ double cl_sum_ratio(Part part, double num, double* red, int& parity, float& ratio) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    double* r = red + parity * 32;
    for (int v = warp; v < kRefWarps; v += kClThreads / 32) {
        float p = part(v, lane);
        for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
        if (lane == 0) r[v] = (double)p;
    }
    __syncthreads();
    if (warp == 0) {
        double t = r[lane & (kRefWarps - 1)];
        for (int o = kRefWarps / 2; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (lane == 0) {
            r[31] = t;
            r[30] = OVER ? t / num : num / t;
        }
    }
    __syncthreads();
    const double total = r[31];
    ratio = (float)r[30];
    parity ^= 1;
    return total;
}

// Lane's part of a sum over the U rows, rows hw, hw + 32, ... of half-warp hw = 2 v + lane / 16
template <class Term>
__device__ __forceinline__ float cl_rows_part(int v, int lane, int nU, const int* urp, Term term) {
    float acc = 0.f;
    for (int b = 2 * v + (lane >> 4); b < nU; b += 2 * kRefWarps)
        for (int e = urp[b] + (lane & 15); e < urp[b + 1]; e += 16) acc += term(e);
    return acc;
}

// Block-wide context of a tile's solves.
struct ClCtx {
    ClLane w, ws;            // half-warp areas of the CG grids and of the setup passes
    char* smem;
    uint32_t base;           // shared-memory address of smem
    int K, rank;
    ClSmem L;
    float2 *tw_n, *tw_m;     // step twiddles: camera grid, register grid, the image's row and column grids
    float2 *tw_x, *tw_y;
    float2 *GP, *GX, *RB, *bq;   // global scratch of the cluster
};

// plain twiddle table of a 16 G-point grid of a solve on the 16 B-point register grid
__device__ __forceinline__ const float2* cl_table(const DevPlan& P, int G, int B) {
    return G == B ? P.tw_r : G == 6 ? P.tw_y6 : G == 8 ? P.tw_y8 : G == 9 ? P.tw_y9 : P.tw_y10;
}

// Solve of one darkfield image by the cluster, on a grid of 16 BX row points x 16 BY
// column points (P * P on 16 B x 16 B). Returns the CG iterations (negative: did not converge).
template <int BN, int B, int BX, int BY>
__device__ __forceinline__ int cl_solve(const ClCtx& c, const DevPlan& P, const DevDF& D, const float* img, float2* sp,
                                        const float* ph, int iters, float tol) {
    constexpr int n = 16 * BN, m = 16 * B, mx = 16 * BX, my = 16 * BY;
    const int K = c.K, rank = c.rank;
    const int u_off = D.u_off, p_off = D.p_off, q_off = D.q_off;
    const int uy0 = D.uy0, qy0 = D.qy0, py0 = D.py0;
    const int N = D.N, nU = D.uy1 - uy0 + 1, nQ = D.qy1 - qy0 + 1, nP = D.py1 - py0 + 1;
    const int *qrp = P.d_rowptr + D.qrp, *prp = P.d_rowptr + D.prp;
    // shares: columns, U rows, Q rows, P rows, camera-grid and register-grid columns
    const int sc = cl_share(mx, K), su = cl_share(nU, K), sq = cl_share(nQ, K), spn = cl_share(nP, K);
    const int sn = cl_share(n, K), sm = cl_share(m, K);
    const int c0 = min(rank * sc, mx), nc = min(sc, mx - c0), rounds = cl_share(sc, kClHW);
    const int u0 = min(rank * su, nU), nu = min(su, nU - u0), q0 = min(rank * sq, nQ), nq = min(sq, nQ - q0);
    const int p0 = min(rank * spn, nP), np = min(spn, nP - p0);
    const int x0 = min(rank * sn, n), nx = min(sn, n - x0), m0 = min(rank * sm, m), nm = min(sm, m - m0);
    const int lc = sc | 1, lu = su | 1, lq = sq | 1;
    uint32_t* tabC = reinterpret_cast<uint32_t*>(c.smem + c.L.tab);
    uint32_t *tabQ = tabC + mx, *tabU = tabQ + nQ;
    for (int i = threadIdx.x; i < mx; i += kClThreads) tabC[i] = cl_map(c.base, i / sc) + 8 * (i % sc);
    for (int i = threadIdx.x; i < nQ; i += kClThreads) tabQ[i] = cl_map(c.base, i / sq) + 8 * (i % sq);
    for (int i = threadIdx.x; i < nU; i += kClThreads) tabU[i] = cl_map(c.base, i / su) + 8 * (i % su);
    int* urp = reinterpret_cast<int*>(c.smem + c.L.urp);
    uint16_t* ux = reinterpret_cast<uint16_t*>(c.smem + c.L.ux);
    unsigned* qm = reinterpret_cast<unsigned*>(c.smem + c.L.qm);
    for (int i = threadIdx.x; i <= nU; i += kClThreads) urp[i] = P.d_rowptr[D.urp + i];
    for (int i = threadIdx.x; i < N; i += kClThreads) ux[i] = (uint16_t)freq_index(P.dU_x[u_off + i], mx);
    for (int i = threadIdx.x; i < nq * kClQWords; i += kClThreads) qm[i] = P.d_qmask[D.qmask_off + q0 * kClQWords + i];
    const float2 *wx = cl_table(P, BX, B), *wy = cl_table(P, BY, B);
    make_step_twiddles(c.tw_x, wx, BX);
    make_step_twiddles(c.tw_y, wy, BY);
    __syncthreads();
    const ClDst toCU{tabC, (uint32_t)c.L.cu, 8 * lc}, toCQ{tabC, (uint32_t)c.L.cq, 8 * lc};
    const ClDst toRQ{tabQ, (uint32_t)c.L.rq, 8 * lq}, toRU{tabU, (uint32_t)c.L.cu, 8 * lu};
    const float2* CU = reinterpret_cast<const float2*>(c.smem + c.L.cu);
    const float2* CQ = reinterpret_cast<const float2*>(c.smem + c.L.cq);
    const float2* RQ = reinterpret_cast<const float2*>(c.smem + c.L.rq);
    float2* xv = reinterpret_cast<float2*>(c.smem + c.L.vec);
    float2 *dv = xv + P.max_N, *sv = dv + P.max_N, *wv = sv + P.max_N;
    const uint32_t wa = c.base + (uint32_t)c.L.vec + 24 * P.max_N;
    double* red = reinterpret_cast<double*>(c.smem + c.L.red);

    // the known field's rows (Eq. 11) on the row grid and (where it differs) the register
    // grid, the image's columns
    const ClValKnown pval{sp, ph, P.dP_ap + p_off, P.dP_pup + p_off};
    cl_rows_in<BX>(c.ws, c.tw_x, p0, np, prp, P.dP_x + p_off, pval, toCQ);
    if constexpr (BX != B) cl_rows_known<B>(c.ws, c.tw_m, p0, np, prp, P.dP_x + p_off, pval, c.GP);
    cl_image_cols<BN>(c.ws, c.tw_n, x0, nx, img, qy0, nQ, D.tr != 0, c.GX);
    cl_sync();
    // p s with the ramp of the U <-> Q column passes into TMEM; |p|^2; F(I) on Q
    const int shift = (((uy0 - qy0 - py0) % my) + my) % my, shift2 = ((qy0 % m) + m) % m;
    cl_cols<BY>(c.ws, c.tw_y, rounds, c0, nc, CQ, lc, nP, 0,
                ClMidStore<BY>{1.f / ((float)mx * (float)my), wy, shift}, toRU);
    if constexpr (BX != B) {
        const float2* GP = c.GP;
        cl_cols_abs2<B>(c.ws, c.tw_m, m0, nm, [GP](int b, int x, int) { return __ldcg(GP + t4_index(b, x, m)); }, nP,
                        c.RB, nQ, P.tw_r, shift2);
    } else {
        cl_cols_abs2<B>(c.ws, c.tw_m, c0, nc, [CQ, lc](int b, int, int xl) { return CQ[b * lc + xl]; }, nP, c.RB, nQ,
                        P.tw_r, shift2);
    }
    cl_image_rows<BN>(c.ws, c.tw_n, q0, nq, c.GX, nQ, qrp, P.dQ_x + q_off, c.bq);
    cl_sync();
    // b = F(I) - P * P on Q (Eq. 13), its rows on the row grid; s = d = C^H b
    cl_rows_rhs<B, BX>(c.ws, c.tw_m, c.tw_x, q0, nq, c.RB, qrp, P.dQ_x + q_off, c.bq, toCQ);
    cl_sync();
    cl_cols<BY>(c.w, c.tw_y, rounds, c0, nc, CQ, lc, nQ, nU, ClMidTimes<BY, false>{}, toRU);
    cl_sync();
    cl_rows_out<BX>(c.w, c.tw_x, u0, nu, CU, lu, urp, ux, wa, K);
    cl_sync();
    for (int e = threadIdx.x; e < N; e += kClThreads) {
        const float2 v = wv[e];
        sv[e] = v;
        dv[e] = v;
        xv[e] = make_float2(0.f, 0.f);
    }
    __syncthreads();
    int par = 0;
    float bf = 0.f;
    double gamma = cl_sum_ratio<true>(
        [&](int v, int lane) {
            return cl_rows_part(v, lane, nU, urp, [&](int e) {
                const float2 q = sv[e];
                return q.x * q.x + q.y * q.y;
            });
        },
        1.0, red, par, bf);
    // CGNR
    bool conv = !(gamma > 1e-300);
    const double stop = (double)tol * (double)tol * gamma;
    int it = 0;
    bf = 0.f;                        // first direction: d = s
    for (; it < iters && !conv; ++it) {
        for (int e = threadIdx.x; e < N; e += kClThreads) dv[e] = cadd(sv[e], cscale(dv[e], bf));
        __syncthreads();
        cl_rows_dir<BX>(c.w, c.tw_x, u0, nu, urp, ux, dv, toCU);
        cl_sync();
        cl_cols<BY>(c.w, c.tw_y, rounds, c0, nc, CU, lc, nU, nQ, ClMidTimes<BY, true>{}, toRQ);
        cl_sync();
        cl_rows_mask<BX>(c.w, c.tw_x, q0, nq, RQ, lq, qm, toCQ);
        cl_sync();
        cl_cols<BY>(c.w, c.tw_y, rounds, c0, nc, CQ, lc, nQ, nU, ClMidTimes<BY, false>{}, toRU);
        cl_sync();
        cl_rows_out<BX>(c.w, c.tw_x, u0, nu, CU, lu, urp, ux, wa, K);
        cl_sync();
        float af;
        const double delta = cl_sum_ratio<false>(
            [&](int v, int lane) {
                return cl_rows_part(v, lane, nU, urp, [&](int e) {
                    const float2 d = dv[e], q = wv[e];
                    return d.x * q.x + d.y * q.y;
                });
            },
            gamma, red, par, af);
        if (!(delta > 0)) break;
        const double gnew = cl_sum_ratio<true>(
            [&](int v, int lane) {
                float g2 = 0.f;
                for (int e = 32 * v + lane; e < N; e += 32 * kRefWarps) {
                    const float2 d = dv[e];
                    float2 x = xv[e];
                    x.x += af * d.x;
                    x.y += af * d.y;
                    xv[e] = x;
                    const float2 s = csub(sv[e], cscale(wv[e], af));
                    sv[e] = s;
                    g2 += s.x * s.x + s.y * s.y;
                }
                return g2;
            },
            gamma, red, par, bf);
        gamma = gnew;
        conv = gnew <= stop;
    }
    // corrected unknown spectrum into the tile's spectrum
    const int* Upup = P.dU_pup + u_off;
    const int* Uap = P.dU_ap + u_off;
    __syncthreads();
    for (int e = rank * kClThreads + threadIdx.x; e < N; e += K * kClThreads) {
        float sn, cs;
        sincosf(ph[Upup[e]], &sn, &cs);
        sp[Uap[e]] = cmul(xv[e], make_float2(cs, -sn));
    }
    cl_sync();
    return conv ? it : -1 - it;
}

// The (row, column) grids the plan chooses from, per tile size and register grid.
template <int BN, int B>
__device__ __forceinline__ int cl_dispatch(const ClCtx& c, const DevPlan& P, const DevDF& D,
                                           const float* img, float2* sp, const float* ph, int iters, float tol) {
#define APIC_CL_GRID(X, Y) \
    case 32 * X + Y: return cl_solve<BN, B, X, Y>(c, P, D, img, sp, ph, iters, tol);
    if constexpr (B == 12) {
        switch (32 * D.bx + D.by) {
            APIC_CL_GRID(12, 6)
            APIC_CL_GRID(12, 8)
            APIC_CL_GRID(12, 9)
            APIC_CL_GRID(10, 6)
            APIC_CL_GRID(10, 8)
            APIC_CL_GRID(9, 9)
            default: return cl_solve<BN, B, 12, 12>(c, P, D, img, sp, ph, iters, tol);
        }
    } else {
        return cl_solve<BN, B, B, B>(c, P, D, img, sp, ph, iters, tol);
    }
#undef APIC_CL_GRID
}

template <int BN, int B>
__global__ void __launch_bounds__(kClThreads, 1)
k_darkfield_cluster(DevPlan P, ClSmem L, int n_tiles, const float* __restrict__ I, const float* __restrict__ phi,
                    float2* __restrict__ spec, char* __restrict__ scratch, size_t per_slot, int iters, float tol,
                    int32_t* __restrict__ status, unsigned long long* __restrict__ counters, DfTiles T) {
    constexpr int n = 16 * BN;
    n_tiles = T.count(n_tiles);
    if (n_tiles <= 0) return;
    extern __shared__ float4 smem4[];
    __shared__ uint32_t tmem_base;
    ClCtx c;
    c.smem = reinterpret_cast<char*>(smem4);
    c.base = (uint32_t)__cvta_generic_to_shared(c.smem);
    c.L = L;
    c.K = (int)cta_count();
    c.rank = (int)cta_rank();
    const int slot = blockIdx.x / c.K, nslots = gridDim.x / c.K;
    c.tw_n = reinterpret_cast<float2*>(c.smem + L.tw);
    c.tw_m = c.tw_n + 2 * 16 * BN;
    c.tw_x = c.tw_m + 2 * 16 * B;
    c.tw_y = c.tw_x + 2 * 16 * P.cl_maxB;
    const ClScratch S = cl_scratch_layout(n, 16 * B, P.band_p, P.band_q, P.max_M);
    c.GP = reinterpret_cast<float2*>(scratch + (size_t)slot * per_slot);
    c.GX = c.GP + S.gx;
    c.RB = c.GP + S.rb;
    c.bq = c.GP + S.bq;
    // all TMEM columns: the launch's shared memory admits one block per SM, so no other
    // block of these kernels holds TMEM there
    const int warp = threadIdx.x >> 5;
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"((uint32_t)__cvta_generic_to_shared(&tmem_base)), "r"(kClTmemCols) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    make_step_twiddles(c.tw_n, P.tw_n, BN);
    make_step_twiddles(c.tw_m, P.tw_r, B);
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    c.w.t = c.ws.t = threadIdx.x & 15;
    c.w.hw = c.ws.hw = threadIdx.x >> 4;
    c.w.mask = c.ws.mask = (threadIdx.x & 16) ? 0xFFFF0000u : 0x0000FFFFu;
    c.w.tm = c.ws.tm = tmem_base + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(kClTmemSlot * (warp >> 2));
    c.w.hs = reinterpret_cast<float2*>(c.smem) + c.w.hw * hw_single_size(P.cl_maxB);
    c.ws.hs = reinterpret_cast<float2*>(c.smem) + c.ws.hw * hw_single_size(BN > B ? BN : B);
    cl_sync();           // every block of the cluster runs before any stores into another's shared memory

    for (int i = slot; i < n_tiles; i += nslots) {
        const int tile = T.tile(i);
        if (status && (status[tile] & (APIC_TILE_BACKGROUND | APIC_TILE_BADINPUT))) continue;
        const float* ph = phi + (size_t)tile * P.npup;
        float2* sp = spec + (size_t)tile * P.nap;
        bool notconv = false;
        for (int di = 0; di < P.n_used; ++di) {
            const DevDF& D = P.df[di];
            const float* img = I + ((size_t)tile * P.n_img + D.led) * n * n;
            const int r = cl_dispatch<BN, B>(c, P, D, img, sp, ph, iters, tol);
            if (r < 0) notconv = true;
            if (threadIdx.x == 0 && c.rank == 0 && counters) {
                atomicAdd(counters + 1, (unsigned long long)(r < 0 ? -1 - r : r));
                atomicAdd(counters + 2, 1ull);
                if (di < kCountedImages) atomicAdd(counters + 4 + di, (unsigned long long)(r < 0 ? -1 - r : r));
            }
        }
        if (threadIdx.x == 0 && c.rank == 0 && notconv && status) atomicOr(status + tile, APIC_TILE_NOTCONV);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    cl_sync();           // no block leaves while another may still store into its shared memory
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kClTmemCols)
                     : "memory");
    }
}

}  // namespace

using ClKernel = void (*)(DevPlan, ClSmem, int, const float*, const float*, float2*, char*, size_t, int, float,
                          int32_t*, unsigned long long*, DfTiles);

// The kernel of 256-pixel tiles for a register grid of 16 B points (NULL: none); a translation unit of its own.
ClKernel cl_kernel_256(int B);

}  // namespace apic
