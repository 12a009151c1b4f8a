// kernels_dfw.cu - darkfield spectrum extension (WSI-APIC Eq. 11-13) for 512-pixel
// tiles, with the wide register FFTs (16 B points, 16 < B <= 32, two step-B rows
// per lane).
//
// The method is the one of kernels_dfr.cu (CG on the normal equations of Eq. 13,
// five passes per iteration over a band-row grid; see there), at the sizes of a
// 512 x 512 tile (pupil radius ~85 grid points, up to ~2.8 k unknowns and ~36 k
// equations per image):
//  * the right-hand side b = F(I_j) - P * P on Q is formed on the camera grid,
//    n = 512 = 16 x 32, as the spectrum of I_j - |p|^2 with p the known field's
//    inverse transform (exact: the lags of P * P reach 2 R < n / 2);
//  * each image's CG runs on its own (row, column) grid chosen with the plan,
//    rows of 288 or 320 points and columns of 192, 256, 288 or 320 points, the
//    smallest on which both correlations are free of aliasing;
//  * the band grids GU, GQ, the column-major known field p and b on Q live in the
//    block's global scratch (L2 / HBM): a 512-pixel tile's GU alone (up to 94 rows
//    of 320 points) exceeds what shared memory can hold beside the transform
//    areas. The band grids are stored in 4 x 4 tiles (t4_index), so that the column
//    passes' loads and stores use whole sectors and few cache lines, like the rows
//    passes'. Shared memory holds the half-warp transform areas and the CG vectors;
//    the setup transforms (512-point areas, the column stage) alias both, since no
//    CG vector is live while an image is being set up.
// A tile is solved by a cluster of K blocks of 512 threads (persistent over tiles;
// images of a tile in order): every pass splits its rows or columns over the K x 32
// half-warps of the cluster, each block owning a fixed share (and with it the CG
// vector entries of its U rows); passes end at cluster barriers and inner products
// are summed across the blocks through distributed shared memory, in rank order, so
// every block takes the same steps. With K blocks per tile only 1/K as many tiles are
// in flight, so their band grids stay in L2 instead of going to HBM. Data another
// block wrote is read with L2-only loads (no stale L1 lines).
// Transforms, vectors and the sums within a row FP32; the sums across rows and the CG's
// scalars to more than FP64's precision (rowsum.cuh).
#define APIC_PACKED_ADDS 1
#include <math.h>

#include <algorithm>

#include "../../include/apic.h"
#include "cluster.cuh"
#include "internal.cuh"
#include "regfft.cuh"
#include "rowsum.cuh"
#include "t4grid.cuh"

namespace apic {

namespace {

#ifndef APIC_DFW_THREADS
#define APIC_DFW_THREADS 512
#endif
constexpr int kWThreads = APIC_DFW_THREADS;
constexpr int kWHW = kWThreads / 16;       // half-warps per block
constexpr int kWStageLd = 33;              // column stage: 32 columns + 1 pad
constexpr int kWBN = 32;                   // camera grid 16 x 32 = 512
constexpr int kWMaxB = 20;                 // longest CG grid: 16 x 20 = 320 points
constexpr int kWQWords = 16;               // Q membership words per band row (two 16-bit masks each)

__device__ __forceinline__ int sfreqw(int i, int n) { return i < n / 2 ? i : i - n; }

// Half-warp of a cluster: t lane, hw index in the block, gh index in the cluster
// (rank x 32 + hw), ghs half-warps in the cluster.
struct HWw {
    int t, hw, gh, ghs;
    unsigned mask;
    float2* hs;
    __device__ HalfWarp h() const { return HalfWarp{t, mask, hs}; }
};

// The sum of a U row's values over the half-warp, into entry b of the list rs of every
// block of the tile (its own through distributed shared memory as well).
template <bool CL>
__device__ __forceinline__ void wrow_sum(const HWw& w, float v, int b, float* rs) {
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(w.mask, v, o, 16);
    if constexpr (!CL) {
        if (w.t == 0) rs[b] = v;
    } else {
        if (w.t < w.ghs / kWHW) {
            const unsigned a = (unsigned)__cvta_generic_to_shared(rs + b);
            unsigned ra;
            asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"((unsigned)w.t));
            asm volatile("st.shared::cluster.f32 [%0], %1;" :: "r"(ra), "f"(v) : "memory");
        }
    }
}

// ---- per-point functors (as in the 256-pixel kernel)
template <bool CL>
struct WValKnown {      // P(c) = O_known(K) exp(j phi(c)) (the spectrum: written by any block of the tile)
    const float2* sp;
    const float* ph;
    const int* ap;
    const int* pup;
    __device__ float2 operator()(int e) const {
        float sn, cs;
        sincosf(ph[pup[e]], &sn, &cs);
        return cmul(ldx<CL>(sp + ap[e]), make_float2(cs, sn));
    }
};
struct WValNextDir {    // d = s + beta d (stored back)
    const float2* sv;
    float2* dv;
    float beta;
    __device__ float2 operator()(int e) const {
        const float2 d = cadd(sv[e], cscale(dv[e], beta));
        dv[e] = d;
        return d;
    }
};
struct WOutStart {      // s = d = C^H b, x = 0; returns |s|^2
    float2* sv;
    float2* dv;
    float2* xv;
    __device__ float operator()(int e, float2 v) const {
        sv[e] = v;
        dv[e] = v;
        xv[e] = make_float2(0.f, 0.f);
        return v.x * v.x + v.y * v.y;
    }
};
struct WValB {          // b on Q
    const float2* bq;
    __device__ float2 operator()(int e) const { return bq[e]; }
};
struct WOutDot {        // w = C^H C d; returns Re <d, w>
    float2* wv;
    const float2* dv;
    __device__ float operator()(int e, float2 v) const {
        wv[e] = v;
        const float2 d = dv[e];
        return d.x * v.x + d.y * v.y;
    }
};

// ---- per-column operations on a column of 16 B points: slot s of lane t holds
// o[s][k1] = the value at y = (t + 16 s) + B k1 (valid where t + 16 s < B)
template <int B>
struct WMidStoreField {     // column-major p s W^(shift k) (16 B values per column; wt: W_16B^j)
    float2* PF;
    float scale;
    const float2* wt;
    int shift;
    static constexpr bool kOut = false;
    static constexpr bool kPre = false;
    __device__ void operator()(float2 (&o)[Slots<B>::value][16], int x, int t) const {
        constexpr int m = 16 * B;
        float2* col = PF + (size_t)x * m;
#pragma unroll
        for (int s = 0; s < Slots<B>::value; ++s)
            if (t + 16 * s < B) {
#pragma unroll
                for (int k1 = 0; k1 < 16; ++k1) {
                    const int k = t + 16 * s + B * k1;
                    col[k] = cscale(cmul(o[s][k1], wt[(shift * k) % m]), scale);
                }
            }
    }
};
template <int B, bool CONJ>
struct WMidTimesField {     // o *= p s or conj(p s), from the column-major copy
    const float2* PF;
    static constexpr bool kOut = true;
    // 256-point columns: the column's 16 values of this lane are loaded before the
    // forward transform (pre), so that their latency overlaps it (measured on the whole
    // step, same box: 1618 Mpx/s against 1567 with the 192-point columns included;
    // the two-slot columns have no registers for it)
    static constexpr bool kPre = B == 16;
    struct Pre {
        float2 v[16];
    };
    __device__ void load(Pre& p, int x, int t) const {
        const float2* col = PF + (size_t)x * (16 * B) + t;
        if (t < B) {
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) p.v[k1] = col[B * k1];
        }
    }
    __device__ void apply(float2 (&o)[Slots<B>::value][16], const Pre& p) const {
#pragma unroll
        for (int k1 = 0; k1 < 16; ++k1) o[0][k1] = CONJ ? cmulc(o[0][k1], p.v[k1]) : cmul(o[0][k1], p.v[k1]);
    }
    __device__ void operator()(float2 (&o)[Slots<B>::value][16], int x, int t) const {
        const float2* col = PF + (size_t)x * (16 * B);
#pragma unroll
        for (int s = 0; s < Slots<B>::value; ++s)
            if (t + 16 * s < B) {
#pragma unroll
                for (int k1 = 0; k1 < 16; ++k1) {
                    const float2 pf = col[t + 16 * s + B * k1];
                    o[s][k1] = CONJ ? cmulc(o[s][k1], pf) : cmul(o[s][k1], pf);
                }
            }
    }
};

// ---- passes (each a separate function so registers are allocated per pass)

// rows of a band: scatter val(e) at x = px[e], inverse transform along x, store the
// rows of the tiled grid G (ld columns).
template <int B, class Val>
__device__ __noinline__ void wpass_rows_in(HWw w, const float2* tw, float2* G, int ld, int nrows, const int* rp,
                                           const int* px, Val val) {
    constexpr int m = 16 * B, S = Slots<B>::value;
    const HalfWarp h = w.h();
    const T4Lane L(w.t);
    for (int b = w.gh; b < nrows; b += w.ghs) {
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
        float2* row = G + t4_row(b, ld);
#pragma unroll
        for (int s = 0; s < S; ++s)
            if (w.t + 16 * s < B) {
#pragma unroll
                for (int k1 = 0; k1 < 16; ++k1) row[L.at(16 * s + B * k1)] = o[s][k1];
            }
    }
}

// rows of a band of the tiled grid G (ld columns): forward transform along x; the sum of
// out(e, value) over each row into the list rs.
template <int B, bool CL, class Out>
__device__ __noinline__ void wpass_rows_out(HWw w, const float2* tw, const float2* G, int ld, int nrows,
                                            const int* rp, const int* px, Out out, float* rs) {
    constexpr int m = 16 * B, S = Slots<B>::value;
    const HalfWarp h = w.h();
    const int c0 = t4_col(w.t);
    for (int b = w.gh; b < nrows; b += w.ghs) {
        const float2* row = G + t4_row(b, ld) + c0;
        float2 v[B], o[S][16];
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = ldx<CL>(row + 64 * j);
        // the row's point range and this lane's first point, loaded before the transform
        const int e0 = rp[b] + w.t, e1 = rp[b + 1];
        int xn = e0 < e1 ? px[e0] : 0;
        fft_a<B, false>(v, o, h, tw);
#pragma unroll
        for (int s = 0; s < S; ++s)
            if (w.t + 16 * s < B) {
#pragma unroll
                for (int k1 = 0; k1 < 16; ++k1) w.hs[w.t + 16 * s + B * k1] = o[s][k1];
            }
        __syncwarp(w.mask);
        float acc = 0.f;
        for (int e = e0; e < e1; e += 16) {
            const int xc = xn;
            if (e + 16 < e1) xn = px[e + 16];
            acc += out(e, w.hs[freq_index(xc, m)]);
        }
        __syncwarp(w.mask);
        wrow_sum<CL>(w, acc, b, rs);
    }
}

// columns x < ncols of a grid whose columns have 16 B points: the ni band rows of the
// tiled grid Gi (ldi columns) are the input at column indices 0..ni - 1, the rest zero;
// inverse along y, mid, and (Mid::kOut) forward along y, column indices 0..no - 1
// stored as the band rows of the tiled grid Go (ldo columns). An input band that
// starts at grid row yi0 and an output band at yo0 are thus transformed as if both
// started at row 0: by the shift theorem that multiplies the inverse transform by
// W^(-yi0 k) and the forward one's input by W^(yo0 k), a ramp W^((yo0 - yi0) k) that
// the stored field (the mid's factor) carries (the column passes of the CG run
// between the U and the Q band in both directions, with the field and its
// conjugate). Each half-warp reads and writes its
// own columns, so Gi and Go may be the same grid. Ends with a tile barrier.
// (Measured and left out: staging strips of 32 columns through shared memory for
// 256-byte row accesses, and issuing the next column's loads before the current
// transform; both slowed the kernel by ~10 %: the first adds block barriers between
// half-warps that otherwise overlap one another's loads and transforms, the second
// spills.)
template <int B, bool CL, class Mid>
__device__ __noinline__ void wpass_cols(HWw w, const float2* tw, int ncols, const float2* Gi, int ldi, int ni,
                                        float2* Go, int ldo, int no, Mid mid) {
    constexpr int S = Slots<B>::value;
    const HalfWarp h = w.h();
    const int ri = t4_row(w.t, ldi), ro = t4_row(w.t, ldo);      // band row t of the lane
    for (int x = w.gh; x < ncols; x += w.ghs) {
        float2 v[B], o[S][16];
        const float2* gi = Gi + ri + t4_col(x);
#pragma unroll
        for (int j = 0; j < B; ++j)                                  // band row t + 16 j
            v[j] = w.t + 16 * j < ni ? ldx<CL>(gi + 16 * j * ldi) : make_float2(0.f, 0.f);
        if constexpr (Mid::kPre) {
            typename Mid::Pre pre;
            mid.load(pre, x, w.t);
            fft_a<B, true>(v, o, h, tw);
            mid.apply(o, pre);
        } else {
            fft_a<B, true>(v, o, h, tw);
            mid(o, x, w.t);
        }
        if constexpr (Mid::kOut) {
            fft_b<B, false>(o, v, h, tw);
            float2* go = Go + ro + t4_col(x);
#pragma unroll
            for (int k1 = 0; k1 < B; ++k1)
                if (w.t + 16 * k1 < no) go[16 * k1 * ldo] = v[k1];
        }
    }
    tile_sync<CL>();
}

// rows of Q in place (tiled grid of 16 B columns): forward along x, keep the Q lags, inverse
// along x. qmask: per band row 16 words; the bit k1 of half (t + 16 s) & 1 of word
// (t + 16 s) >> 1 says whether x index (t + 16 s) + B k1 is in Q. Ends with __syncthreads.
template <int B, bool CL>
__device__ __noinline__ void wpass_rows_mask(HWw w, const float2* tw, float2* G, int nrows, const unsigned* qmask) {
    constexpr int m = 16 * B, S = Slots<B>::value;
    const HalfWarp h = w.h();
    const int c0 = t4_col(w.t);
    for (int b = w.gh; b < nrows; b += w.ghs) {
        float2* row = G + t4_row(b, m) + c0;
        float2 v[B], o[S][16];
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = ldx<CL>(row + 64 * j);
        unsigned qw[S];
#pragma unroll
        for (int s = 0; s < S; ++s) qw[s] = qmask[(size_t)b * kWQWords + ((w.t + 16 * s) >> 1)];
        fft_a<B, false>(v, o, h, tw);
#pragma unroll
        for (int s = 0; s < S; ++s) {
            const int ls = w.t + 16 * s;
            const unsigned bits = qw[s] >> (16 * (ls & 1));
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1)
                if (!((bits >> k1) & 1u)) o[s][k1] = make_float2(0.f, 0.f);
        }
        fft_b<B, true>(o, v, h, tw);
#pragma unroll
        for (int k1 = 0; k1 < B; ++k1) row[64 * k1] = v[k1];
    }
    tile_sync<CL>();
}

// Columns of I - |p|^2 (n = 512; the image read transposed with tr, once, with
// evict-first loads): Eq. 13's right-hand side F(I) - P * P is the spectrum of the
// image minus the intensity of the known field, so p's column x is formed from the
// nP band rows of the tiled grid GP (P's rows transformed along x on the camera grid) by an
// inverse transform along y and |p|^2 kept in registers; then the chunk's 32 image
// columns are staged through shared memory (coalesced reads), the difference is
// formed and transformed forward along y; rows qy0.. (nQ) go to GX (row length n).
// Half-warps 0..31 take one column of a chunk each. The stages alias the half-warp
// areas; barriers separate each use from the transforms. Ends with a tile barrier.
template <bool CL>
__device__ __noinline__ void wpass_image_cols_p(HWw w, const float2* tw, float2* stage, const float* img,
                                                const float2* GP, int nP, float2* GX, int qy0, int nQ,
                                                bool tr) {
    constexpr int BN = kWBN, n = 16 * BN, S = Slots<BN>::value;
    const HalfWarp h = w.h();
    float* stage_f = reinterpret_cast<float*>(stage);
    for (int c0 = 32 * (w.gh / kWHW); c0 < n; c0 += 32 * (w.ghs / kWHW)) {     // this block's chunks of 32 columns
        const int x = c0 + w.hw;
        float2 v[BN], o[S][16];
        float q[S][16];
        // the band as if it started at row 0: that multiplies p by a phase ramp along
        // y, which |p|^2 does not see
        const float2* gp = GP + t4_row(w.t, n) + t4_col(x);
#pragma unroll
        for (int j = 0; j < BN; ++j) v[j] = w.t + 16 * j < nP ? ldx<CL>(gp + 16 * j * n) : make_float2(0.f, 0.f);
        fft_a<BN, true>(v, o, h, tw);               // p(x, y), y = (t + 16 s) + BN k1
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) q[s][k1] = cabs2(o[s][k1]);
        __syncthreads();                            // transforms done: the stage may overwrite the areas
        if (tr) {   // column c of the solve frame is image row c
            for (int idx = threadIdx.x; idx < n * 32; idx += blockDim.x) {
                const int c = idx / n, y = idx - c * n;
                stage_f[y * kWStageLd + c] = __ldcs(img + (size_t)(c0 + c) * n + y);
            }
        } else {
            for (int idx = threadIdx.x; idx < n * 32; idx += blockDim.x) {
                const int y = idx >> 5, c = idx & 31;
                stage_f[y * kWStageLd + c] = __ldcs(img + (size_t)y * n + c0 + c);
            }
        }
        __syncthreads();
#pragma unroll
        for (int s = 0; s < S; ++s)
#pragma unroll
            for (int k1 = 0; k1 < 16; ++k1) {
                const int y = (w.t + 16 * s < BN ? w.t + 16 * s : 0) + BN * k1;
                o[s][k1] = make_float2(stage_f[y * kWStageLd + w.hw] - q[s][k1], 0.f);
            }
        __syncthreads();                            // the stage is consumed
        fft_b<BN, false>(o, v, h, tw);              // along y: v[k1] at ky = t + 16 k1
        __syncthreads();
#pragma unroll
        for (int k1 = 0; k1 < BN; ++k1) {
            const int bb = sfreqw(w.t + 16 * k1, n) - qy0;
            if (bb >= 0 && bb < nQ) stage[bb * kWStageLd + w.hw] = v[k1];
        }
        __syncthreads();
        for (int idx = threadIdx.x; idx < nQ * 32; idx += blockDim.x) {
            const int b = idx >> 5, c = idx & 31;
            GX[(size_t)b * n + c0 + c] = stage[b * kWStageLd + c];
        }
        __syncthreads();
    }
    tile_sync<CL>();
}

// rows of GX (length n): forward along x, bq[e] = value / n^2 at the Q points. Ends
// with __syncthreads.
template <bool CL>
__device__ __noinline__ void wpass_image_rows(HWw w, const float2* tw, const float2* GX, int nQ, const int* qrp,
                                              const int* Qx, float2* bq) {
    constexpr int BN = kWBN, n = 16 * BN, S = Slots<BN>::value;
    const HalfWarp h = w.h();
    const float inv_n2 = 1.f / (float)(n * n);
    for (int b = w.gh; b < nQ; b += w.ghs) {
        const float2* row = GX + (size_t)b * n;
        float2 v[BN], o[S][16];
#pragma unroll
        for (int j = 0; j < BN; ++j) v[j] = ldx<CL>(row + w.t + 16 * j);
        fft_a<BN, false>(v, o, h, tw);
#pragma unroll
        for (int s = 0; s < S; ++s)
            if (w.t + 16 * s < BN) {
#pragma unroll
                for (int k1 = 0; k1 < 16; ++k1) w.hs[w.t + 16 * s + BN * k1] = o[s][k1];
            }
        __syncwarp(w.mask);
        for (int e = qrp[b] + w.t; e < qrp[b + 1]; e += 16) bq[e] = cscale(w.hs[freq_index(Qx[e], n)], inv_n2);
        __syncwarp(w.mask);
    }
    tile_sync<CL>();
}

}  // namespace

// Shared memory of one block (bytes, 16-aligned offsets):
//   [0, vec)          half-warp areas of the CG grids (17 x 20 values each)
//   [vec, vec_end)    CG vectors x, d, s, w (max_N each)
//   [0, setup)        during an image's setup: half-warp areas of the 512-point
//                     transforms (17 x 32 values each), or the 32-column image
//                     stage, or the output stage of the image columns
//   [tw, total)       step twiddles of the camera grid and of the image's row and
//                     column grids. The camera grid's serve an image's setup alone and are
//                     made anew for each image; during the CG its scalars and two lists of the
//                     U rows' sums take their place. (Beside them the lists took 2 KB, and plans whose CG
//                     vectors fill the block lost this kernel: 3967 unknowns fit, 3902 did
//                     then; 8 + 16 images on rings at NA 0.29 and 0.376 have 3933.)
struct DFWSmem {
    size_t vec, tw, total;
};

__host__ __device__ inline size_t walign16(size_t b) { return (b + 15) & ~(size_t)15; }

// band: the most band rows a column pass stages (max of the U, P and Q bands)
__host__ __device__ inline DFWSmem dfw_smem_layout(int max_N, int band) {
    DFWSmem L;
    L.vec = walign16(std::max((size_t)kWHW * hw_single_size(kWMaxB), (size_t)band * kWStageLd) * sizeof(float2));
    const size_t cg_end = L.vec + walign16((size_t)4 * max_N * sizeof(float2));
    const size_t setup_hw = (size_t)kWHW * hw_single_size(kWBN) * sizeof(float2);
    const size_t stage_c = (size_t)band * kWStageLd * sizeof(float2);
    const size_t stage_f = (size_t)16 * kWBN * kWStageLd * sizeof(float);
    const size_t setup = std::max(setup_hw, std::max(stage_c, stage_f));
    L.tw = walign16(std::max(cg_end, setup));
    L.total = walign16(L.tw + (size_t)2 * 16 * (kWBN + 2 * kWMaxB) * sizeof(float2));
    return L;
}

size_t dfw_smem_bytes(int max_N, int band) { return dfw_smem_layout(max_N, band).total; }

// Global scratch of one block: GQ (Q or P band rows on the camera grid), PF (the
// column-major known field of the CG grid, or the image's Q rows), GU (U band rows
// of the CG grid), b on Q.
size_t dfw_scratch_bytes(const DevPlan& P) {
    const int n = P.h;
    size_t s = (size_t)t4_rows(std::max(P.band_q, P.band_p)) * n;                         // GQ (tiled)
    s += std::max((size_t)P.max_mxy, (size_t)P.band_q * n);                               // PF / F(I) rows
    s += (size_t)t4_rows(P.band_u) * P.max_mx;                                            // GU (tiled)
    s += (size_t)P.max_M;                                                                 // b on Q
    return (s * sizeof(float2) + 255) & ~(size_t)255;
}

namespace {

struct DFWCtx {
    HWw w;                  // half-warp areas of the CG grids
    HWw ws;                 // half-warp areas of the 512-point setup transforms
    float2* tw_n;           // step twiddles of the camera grid (filled per image)
    float2* tw_x;           // step twiddles of the image's row grid (filled per image)
    float2* tw_y;           // step twiddles of the image's column grid (filled per image)
    float2 *GU, *GQ, *PF, *bq;
    float2 *dv, *sv, *wv, *xv;
    float2* stage;          // stages of the setup column pass (alias the half-warp areas)
    int n_rs;
    // in the place of tw_n (8 KB) during the CG: its scalars and two lists of the U rows'
    // sums, n_rs entries each (at most the 320 of the longest grid)
    __device__ CgScalars* cg() const { return reinterpret_cast<CgScalars*>(tw_n); }
    __device__ float* rs(int i) const { return reinterpret_cast<float*>(cg() + 1) + i * n_rs; }
};

// plain twiddle table of a 16 G-point grid of the wide solve
__device__ __forceinline__ const float2* wgrid_table(const DevPlan& P, int G) {
    return G == 12 ? P.tw_w12 : G == 16 ? P.tw_w16 : G == 18 ? P.tw_w18 : P.tw_w20;
}

// Solve of one darkfield image (image `img`) on a grid of 16 BX row points x 16 BY
// column points, by the K blocks of the cluster: b = F(I - |p|^2) on Q on the camera
// grid, then CGNR. Returns the CG iterations (negative: did not converge).
template <int BX, int BY, bool CL>
__device__ __forceinline__ int dfw_solve(const DFWCtx& c, const DevPlan& P, const DevDF& D, const float* img,
                                         float2* sp, const float* ph, int iters, float tol) {
    constexpr int n = 16 * kWBN, mx = 16 * BX;
    const HWw& w = c.w;
    const int u_off = D.u_off, p_off = D.p_off, q_off = D.q_off;
    const int uy0 = D.uy0, qy0 = D.qy0, py0 = D.py0;
    const int nU = D.uy1 - uy0 + 1, nQ = D.qy1 - qy0 + 1, nP = D.py1 - py0 + 1;
    const int *urp = P.d_rowptr + D.urp, *qrp = P.d_rowptr + D.qrp, *prp = P.d_rowptr + D.prp;
    const unsigned* qmask = P.d_qmask + D.qmask_off;
    const WValKnown<CL> pval{sp, ph, P.dP_ap + p_off, P.dP_pup + p_off};
    make_step_twiddles(c.tw_n, P.tw_n, kWBN);
    make_step_twiddles(c.tw_x, wgrid_table(P, BX), BX);
    make_step_twiddles(c.tw_y, wgrid_table(P, BY), BY);
    __syncthreads();
    // b = F(I) - P * P on Q (Eq. 13) as the spectrum of I - |p|^2 on the camera grid
    // (exact: P * P's lags reach 2 R < n / 2): the known field's band rows along x,
    // then per column p, the difference and its forward transform, then the rows
    wpass_rows_in<kWBN>(c.ws, c.tw_n, c.GQ, n, nP, prp, P.dP_x + p_off, pval);
    tile_sync<CL>();
    wpass_image_cols_p<CL>(c.ws, c.tw_n, c.stage, img, c.GQ, nP, c.PF, qy0, nQ, D.tr != 0);
    wpass_image_rows<CL>(c.ws, c.tw_n, c.PF, nQ, qrp, P.dQ_x + q_off, c.bq);
    // band rows of the known field P (Eq. 11) along x on the row grid, then p s on
    // the column grid, column-major in PF (s = 1 / (mx my): the two unnormalised
    // transforms around each product)
    const float scale = 1.f / ((float)mx * (float)(16 * BY));
    wpass_rows_in<BX>(w, c.tw_x, c.GQ, mx, nP, prp, P.dP_x + p_off, pval);
    tile_sync<CL>();
    // the field carries the ramp W^((uy0 - qy0) k) of the U <-> Q column passes and
    // W^(-py0 k) for its own band's start (see wpass_cols)
    const int my = 16 * BY, shift = (((uy0 - qy0 - py0) % my) + my) % my;
    wpass_cols<BY, CL>(w, c.tw_y, mx, c.GQ, mx, nP, c.GQ, mx, 0,
                      WMidStoreField<BY>{c.PF, scale, wgrid_table(P, BY), shift});
    // rows of b inverse along x on the row grid; s = d = C^H b
    wpass_rows_in<BX>(w, c.tw_x, c.GQ, mx, nQ, qrp, P.dQ_x + q_off, WValB{c.bq});
    tile_sync<CL>();
    wpass_cols<BY, CL>(w, c.tw_y, mx, c.GQ, mx, nQ, c.GU, mx, nU, WMidTimesField<BY, false>{c.PF});
    wpass_rows_out<BX, CL>(w, c.tw_x, c.GU, mx, nU, urp, P.dU_x + u_off, WOutStart{c.sv, c.dv, c.xv}, c.rs(0));
    tile_sync<CL>();
    // CGNR; each half-warp updates the vector entries of the U rows it gathered
    bool conv = cg_start(c.cg(), c.rs(0), nU, tol);
    int it = 0;
    for (; it < iters && !conv; ++it) {
        wpass_rows_in<BX>(w, c.tw_x, c.GU, mx, nU, urp, P.dU_x + u_off, WValNextDir{c.sv, c.dv, c.cg()->beta});
        tile_sync<CL>();
        wpass_cols<BY, CL>(w, c.tw_y, mx, c.GU, mx, nU, c.GQ, mx, nQ, WMidTimesField<BY, true>{c.PF});
        wpass_rows_mask<BX, CL>(w, c.tw_x, c.GQ, nQ, qmask);
        wpass_cols<BY, CL>(w, c.tw_y, mx, c.GQ, mx, nQ, c.GU, mx, nU, WMidTimesField<BY, false>{c.PF});
        wpass_rows_out<BX, CL>(w, c.tw_x, c.GU, mx, nU, urp, P.dU_x + u_off, WOutDot{c.wv, c.dv}, c.rs(0));
        tile_sync<CL>();
        if (!cg_alpha(c.cg(), c.rs(0), nU)) break;
        const float af = c.cg()->alpha;
        for (int b = w.gh; b < nU; b += w.ghs) {
            float g2 = 0.f;
            for (int e = urp[b] + w.t; e < urp[b + 1]; e += 16) {
                const float2 d = c.dv[e];
                float2 x = c.xv[e];
                x.x += af * d.x;
                x.y += af * d.y;
                c.xv[e] = x;
                const float2 sv = csub(c.sv[e], cscale(c.wv[e], af));
                c.sv[e] = sv;
                g2 += sv.x * sv.x + sv.y * sv.y;
            }
            wrow_sum<CL>(w, g2, b, c.rs(1));
        }
        tile_sync<CL>();
        conv = cg_beta(c.cg(), c.rs(1), nU);
    }
    // corrected unknown spectrum into the tile's spectrum (this block's U rows)
    const int* Upup = P.dU_pup + u_off;
    const int* Uap = P.dU_ap + u_off;
    auto put = [&](int e) {
        float sn, cs;
        sincosf(ph[Upup[e]], &sn, &cs);
        sp[Uap[e]] = cmul(c.xv[e], make_float2(cs, -sn));
    };
    for (int b = w.gh; b < nU; b += w.ghs)
        for (int e = urp[b] + w.t; e < urp[b + 1]; e += 16) put(e);
    tile_sync<CL>();
    return conv ? it : -1 - it;
}

template <bool CL>
__global__ void __launch_bounds__(kWThreads, 1)
k_darkfield_wide(DevPlan P, int n_tiles, const float* __restrict__ I, const float* __restrict__ phi,
                 float2* __restrict__ spec, char* __restrict__ scratch, size_t per_block, int iters, float tol,
                 int32_t* __restrict__ status, unsigned long long* __restrict__ counters, int* __restrict__ work,
                 DfTiles T) {
    constexpr int n = 16 * kWBN;
    n_tiles = T.count(n_tiles);
    if (n_tiles <= 0) return;
    extern __shared__ float4 smem4[];
    char* sbase = reinterpret_cast<char*>(smem4);
    const DFWSmem SL = dfw_smem_layout(P.max_N, max(P.band_q, max(P.band_p, P.band_u)));
    DFWCtx c;
    c.dv = reinterpret_cast<float2*>(sbase + SL.vec);
    c.sv = c.dv + P.max_N;
    c.wv = c.sv + P.max_N;
    c.xv = c.wv + P.max_N;
    c.stage = reinterpret_cast<float2*>(sbase);
    c.tw_n = reinterpret_cast<float2*>(sbase + SL.tw);
    c.tw_x = c.tw_n + 2 * 16 * kWBN;
    c.tw_y = c.tw_x + 2 * 16 * kWMaxB;
    c.n_rs = P.band_u;

    const int rank = CL ? (int)cta_rank() : 0, K = CL ? (int)cta_count() : 1;
    const int slot = blockIdx.x / K, nslots = gridDim.x / K;      // tile slot = the cluster
    c.w.hw = c.ws.hw = threadIdx.x >> 4;
    c.w.gh = c.ws.gh = rank * kWHW + c.w.hw;
    c.w.ghs = c.ws.ghs = K * kWHW;
    c.w.t = c.ws.t = threadIdx.x & 15;
    c.w.mask = c.ws.mask = (threadIdx.x & 16) ? 0xFFFF0000u : 0x0000FFFFu;
    c.w.hs = reinterpret_cast<float2*>(sbase) + c.w.hw * hw_single_size(kWMaxB);
    c.ws.hs = reinterpret_cast<float2*>(sbase) + c.ws.hw * hw_single_size(kWBN);

    char* base = scratch + (size_t)slot * per_block;
    c.GQ = reinterpret_cast<float2*>(base);
    c.PF = c.GQ + (size_t)t4_rows(max(P.band_q, P.band_p)) * n;
    c.GU = c.PF + max((size_t)P.max_mxy, (size_t)P.band_q * n);
    c.bq = c.GU + (size_t)t4_rows(P.band_u) * P.max_mx;
    tile_sync<CL>();

    // one block per tile: tiles taken one at a time from the launch's counter (a block that
    // meets skipped background tiles goes on to the next, so uneven batches balance);
    // clusters (and launches without a counter): by stride
    __shared__ int s_next;
    auto take = [&](int prev) -> int {
        if (CL || !work) return prev < 0 ? slot : prev + nslots;
        __syncthreads();
        if (threadIdx.x == 0) s_next = atomicAdd(work, 1);
        __syncthreads();
        return s_next;
    };
    for (int i = take(-1); i < n_tiles; i = take(i)) {
        const int tile = T.tile(i);
        if (status && (status[tile] & (APIC_TILE_BACKGROUND | APIC_TILE_BADINPUT))) continue;
        const float* ph = phi + (size_t)tile * P.npup;
        float2* sp = spec + (size_t)tile * P.nap;
        bool notconv = false;
        for (int di = 0; di < P.n_used; ++di) {
            const DevDF& D = P.df[di];
            const float* img = I + ((size_t)tile * P.n_img + D.led) * n * n;
            int r;
            switch (16 * D.bx + D.by) {
                case 16 * 18 + 12: r = dfw_solve<18, 12, CL>(c, P, D, img, sp, ph, iters, tol); break;
                case 16 * 18 + 16: r = dfw_solve<18, 16, CL>(c, P, D, img, sp, ph, iters, tol); break;
                case 16 * 18 + 18: r = dfw_solve<18, 18, CL>(c, P, D, img, sp, ph, iters, tol); break;
                case 16 * 20 + 12: r = dfw_solve<20, 12, CL>(c, P, D, img, sp, ph, iters, tol); break;
                case 16 * 20 + 16: r = dfw_solve<20, 16, CL>(c, P, D, img, sp, ph, iters, tol); break;
                case 16 * 20 + 18: r = dfw_solve<20, 18, CL>(c, P, D, img, sp, ph, iters, tol); break;
                default: r = dfw_solve<20, 20, CL>(c, P, D, img, sp, ph, iters, tol); break;
            }
            if (r < 0) notconv = true;
            if (threadIdx.x == 0 && rank == 0 && counters) {
                atomicAdd(counters + 1, (unsigned long long)(r < 0 ? -1 - r : r));
                atomicAdd(counters + 2, 1ull);
                if (di < kCountedImages) atomicAdd(counters + 4 + di, (unsigned long long)(r < 0 ? -1 - r : r));
            }
        }
        if (threadIdx.x == 0 && rank == 0 && notconv && status) atomicOr(status + tile, APIC_TILE_NOTCONV);
    }
}

}  // namespace

using DFWKernel = void (*)(DevPlan, int, const float*, const float*, float2*, char*, size_t, int, float, int32_t*,
                           unsigned long long*, int*, DfTiles);

static DFWKernel dfw_kernel(int K) {
    return K == 1 ? k_darkfield_wide<false> : K >= 2 && K <= kMaxCluster ? k_darkfield_wide<true> : nullptr;
}

// Tile slots (clusters of K blocks) that run at once, 0 on error.
int configure_dfw(size_t smem, int K) { return cluster_slots((const void*)dfw_kernel(K), kWThreads, smem, K); }

// grid: tile slots (clusters); each gets K blocks.
cudaError_t launch_darkfield_wide(const DevPlan& P, int K, int grid, size_t smem, int n_tiles, const float* I,
                                  const float* phi, float2* spec, void* scratch, size_t per_block, int iters,
                                  float tol, int32_t* status, unsigned long long* counters, int* work,
                                  cudaStream_t st, DfTiles tiles) {
    DFWKernel f = dfw_kernel(K);
    if (!f || P.h != 16 * kWBN || P.w != P.h) return cudaErrorInvalidValue;
    const int slots = min(grid, n_tiles);
    if (slots < 1) return cudaErrorInvalidConfiguration;
    if (K == 1 && work) {
        const cudaError_t e = cudaMemsetAsync(work, 0, sizeof(int), st);
        if (e != cudaSuccess) return e;
    }
    return cluster_launch(f, K, slots, kWThreads, smem, st, P, n_tiles, I, phi, spec, (char*)scratch, per_block, iters,
                          tol, status, counters, K == 1 ? work : (int*)nullptr, tiles);
}

}  // namespace apic
