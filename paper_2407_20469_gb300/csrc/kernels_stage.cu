// kernels_stage.cu - per-tile stages before the darkfield extension:
// background statistic (Sec. 3.2), Kramers-Kronig recovery (Eq. 4-7),
// aberration solve (Eq. 8-10), pupil-phase table, correction and stitching,
// pupil output.
#include <math.h>

#include "../../include/apic.h"
#include "cluster.cuh"
#include "passes.cuh"
#include "zernike.h"

namespace apic {

// ---------------------------------------------------------------- background
// Per tile: mean over the NA-matching images of var(I)/mean(I)^2; flags
// tiles below the threshold and stacks with negative or non-finite values.
// Each thread sums its own pixels in FP32 (a few hundred values), the block
// combines the partial sums in FP64; the darkfield images are only checked.
// The tile's images are dealt to the K blocks of a cluster; the first block adds the
// images' values in image order, so the result does not depend on K.
constexpr int kMaxBF = 255;                 // plans take no more NA-matching images

__global__ void __launch_bounds__(kThreads) k_background(DevPlan P, const float* __restrict__ I,
                                                         float* __restrict__ c2, int32_t* __restrict__ status,
                                                         float thresh2, int learned) {
    __shared__ double red[64];
    __shared__ double value[kMaxBF];        // of the first block: var / mean^2 of each NA-matching image
    __shared__ int flags[kMaxCluster];      // of the first block: each block's check
    const int K = (int)cta_count(), rank = (int)cta_rank();
    const int tile = blockIdx.x / K;
    const size_t npix = (size_t)P.h * P.w;
    const float* T = I + (size_t)tile * P.n_img * npix;
    int bad = 0, par = 0;
    auto invalid = [](float4 v) {
        return !(v.x >= 0.f && v.x < INFINITY) || !(v.y >= 0.f && v.y < INFINITY) ||
               !(v.z >= 0.f && v.z < INFINITY) || !(v.w >= 0.f && v.w < INFINITY);
    };
    tile_sync<true>();                      // the first block runs before any other stores into it
    for (int i = rank; i < P.n_img; i += K) {
        const float4* T4 = reinterpret_cast<const float4*>(T + i * npix);
        const int nq = (int)(npix / 4);
        if (i < P.n_bf) {
            float s = 0.f, s2 = 0.f;
#pragma unroll 4
            for (int k = threadIdx.x; k < nq; k += blockDim.x) {
                const float4 v = __ldcs(T4 + k);        // streamed: evict first from L2
                bad |= invalid(v);
                s += (v.x + v.y) + (v.z + v.w);
                s2 += (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
            }
            const double st = block_sum2((double)s, red, par);
            const double st2 = block_sum2((double)s2, red, par);
            if (threadIdx.x == 0) {
                const double mean = st / npix;
                const double var = st2 / npix - mean * mean;
                st_first(value + i, mean > 0 ? var / (mean * mean) : 0.0);
            }
        } else {
#pragma unroll 4
            for (int k = threadIdx.x; k < nq; k += blockDim.x) bad |= invalid(__ldcs(T4 + k));
        }
    }
    const int mine = __syncthreads_or(bad);
    if (threadIdx.x == 0) st_first(flags + rank, mine);
    tile_sync<true>();
    if (rank == 0 && threadIdx.x == 0) {
        double acc = 0;
        for (int i = 0; i < P.n_bf; ++i) acc += value[i];
        int anybad = 0;
        for (int q = 0; q < K; ++q) anybad |= flags[q];
        const float v = (float)(acc / P.n_bf);
        if (c2) c2[tile] = v;
        int st = 0;
        if (v < thresh2) st |= learned ? APIC_TILE_LEARNED : APIC_TILE_BACKGROUND;
        if (anybad) st |= APIC_TILE_BADINPUT;
        status[tile] = st;
    }
}

// Blocks per tile. One block reads 512-pixel images at 0.07 TB/s, so a batch is as slow as its
// first tile until the chip is full: 1.80 ms for 1 tile and 2.14 for 96 with one block each, 0.20
// and 0.66 with eight (256 pixels: 0.22 and 0.43 ms for 1 and 100 tiles, 0.036 and 0.15). Beyond
// some 64 tiles four are as fast: 2.14 ms for 400 tiles of 512 pixels (2.59 with one), 0.34 for
// 1000 of 128 pixels (0.36 with eight).
constexpr int kBgFew = 64;

cudaError_t launch_background(const DevPlan& P, int n_tiles, const float* I, float* c2, int32_t* status,
                              float thresh2, cudaStream_t st, int learned) {
    const int K = n_tiles <= kBgFew ? 8 : 4;
    return cluster_launch(k_background, K, n_tiles, kThreads, 0, st, P, I, c2, status, thresh2, learned);
}

__device__ __forceinline__ bool skip_tile(const int32_t* status, int tile) {
    return status && (status[tile] & (APIC_TILE_BACKGROUND | APIC_TILE_BADINPUT));
}

// The tiles that are not skipped, in order: list[0] their number, list[1 ..] the tiles. One
// block, 1024 tiles at a time.
__global__ void __launch_bounds__(1024) k_list_tiles(int n_tiles, const int32_t* __restrict__ status,
                                                     int* __restrict__ list) {
    __shared__ int warps[32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int found = 0;
    for (int t0 = 0; t0 < n_tiles; t0 += 1024) {
        const int tile = t0 + threadIdx.x;
        const bool on = tile < n_tiles && !skip_tile(status, tile);
        const unsigned mask = __ballot_sync(0xffffffffu, on);
        if (lane == 0) warps[warp] = __popc(mask);
        __syncthreads();
        int before = 0, all = 0;
        for (int w = 0; w < 32; ++w) {
            before += w < warp ? warps[w] : 0;
            all += warps[w];
        }
        if (on) list[1 + found + before + __popc(mask & ((1u << lane) - 1))] = tile;
        found += all;
        __syncthreads();
    }
    if (threadIdx.x == 0) list[0] = found;
}

cudaError_t launch_list_tiles(int n_tiles, const int32_t* status, int* list, cudaStream_t st) {
    k_list_tiles<<<1, 1024, 0, st>>>(n_tiles, status, list);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- Kramers-Kronig
// One block per (tile, NA-matching image) problem, persistent over problems.
// Scratch: an n x n complex grid per block.
//   P1 rows: log(max(I, 1e-6 mean I)), forward transform along x
//   P2 cols: forward along y, half-plane mask of Eq. 5, inverse along y
//   P3 rows: inverse along x, / n^2, exp (Eq. 6), forward along x
//   P4 cols: forward along y, / n^2 (series coefficients, Eq. 7)
// then the values at K = k_p - k_i for every pupil point k_p are gathered.
__global__ void __launch_bounds__(kThreads) k_kk(DevPlan P, int n_tiles, const float* __restrict__ I,
                                                 float2* __restrict__ xdisc, float2* __restrict__ scratch,
                                                 const int32_t* __restrict__ status) {
    extern __shared__ float4 smem4[];
    float2* sm = reinterpret_cast<float2*>(smem4);
    const int n = P.h, ln = ilog2(n);
    float2* tw = sm + 2 * (kChunk / n) * (n + 1);
    double* red = reinterpret_cast<double*>(tw + n);
    load_twiddles(tw, P.tw_n, n);
    const FFTChunk c = make_chunk(sm, n, tw);
    const int S = c.S, ld = c.ld;
    float2* G = scratch + (size_t)blockIdx.x * n * n;
    const float inv_n2 = 1.0f / (float)(n * n);
    const int nprob = n_tiles * P.n_bf;
    for (int prob = blockIdx.x; prob < nprob; prob += gridDim.x) {
        const int tile = prob / P.n_bf, i = prob - tile * P.n_bf;
        if (skip_tile(status, tile)) continue;
        const float* img = I + ((size_t)tile * P.n_img + i) * n * n;
        const int kix = P.led_x[i], kiy = P.led_y[i];
        double s = 0;
        for (int t = threadIdx.x; t < n * n; t += blockDim.x) s += img[t];
        s = block_sum(s, red);
        const float eps = (float)(1e-6 * s / ((double)n * n));
        // P1
        for (int r0 = 0; r0 < n; r0 += S) {
            for (int t = threadIdx.x; t < (S << ln); t += blockDim.x) {
                const int q = t >> ln, x = t & (n - 1);
                c.a[q * ld + x] = make_float2(logf(fmaxf(img[(size_t)(r0 + q) * n + x], eps)), 0.f);
            }
            const float2* R = fft_chunk<false>(c);
            for (int t = threadIdx.x; t < (S << ln); t += blockDim.x) {
                const int q = t >> ln, x = t & (n - 1);
                G[(size_t)(r0 + q) * n + x] = R[q * ld + x];
            }
            __syncthreads();
        }
        // P2
        const long long hh = (long long)P.h * P.h, ww = (long long)P.w * P.w;
        for (int c0 = 0; c0 < n; c0 += S) {
            for (int t = threadIdx.x; t < S * n; t += blockDim.x) {
                const int y = t / S, q = t - y * S;
                c.a[q * ld + y] = G[(size_t)y * n + c0 + q];
            }
            float2* R = fft_chunk<false>(c);
            for (int t = threadIdx.x; t < S * n; t += blockDim.x) {
                const int y = t / S, q = t - y * S;
                const long long dot = (long long)signed_freq(c0 + q, n) * kix * hh + (long long)signed_freq(y, n) * kiy * ww;
                const float f = dot < 0 ? 1.f : (dot == 0 ? 0.5f : 0.f);
                R[q * ld + y] = cscale(R[q * ld + y], f);
            }
            FFTChunk c2 = c;
            c2.a = R;
            c2.b = (R == c.a) ? c.b : c.a;
            const float2* R2 = fft_chunk<true>(c2);
            for (int t = threadIdx.x; t < S * n; t += blockDim.x) {
                const int y = t / S, q = t - y * S;
                G[(size_t)y * n + c0 + q] = R2[q * ld + y];
            }
            __syncthreads();
        }
        // P3
        for (int r0 = 0; r0 < n; r0 += S) {
            for (int t = threadIdx.x; t < (S << ln); t += blockDim.x) {
                const int q = t >> ln, x = t & (n - 1);
                c.a[q * ld + x] = G[(size_t)(r0 + q) * n + x];
            }
            float2* R = fft_chunk<true>(c);
            for (int t = threadIdx.x; t < (S << ln); t += blockDim.x) {
                const int q = t >> ln, x = t & (n - 1);
                const float2 z = cscale(R[q * ld + x], inv_n2);
                float sn, cs;
                sincosf(z.y, &sn, &cs);
                const float e = expf(z.x);
                R[q * ld + x] = make_float2(e * cs, e * sn);
            }
            FFTChunk c2 = c;
            c2.a = R;
            c2.b = (R == c.a) ? c.b : c.a;
            const float2* R2 = fft_chunk<false>(c2);
            for (int t = threadIdx.x; t < (S << ln); t += blockDim.x) {
                const int q = t >> ln, x = t & (n - 1);
                G[(size_t)(r0 + q) * n + x] = R2[q * ld + x];
            }
            __syncthreads();
        }
        // P4
        for (int c0 = 0; c0 < n; c0 += S) {
            for (int t = threadIdx.x; t < S * n; t += blockDim.x) {
                const int y = t / S, q = t - y * S;
                c.a[q * ld + y] = G[(size_t)y * n + c0 + q];
            }
            const float2* R = fft_chunk<false>(c);
            for (int t = threadIdx.x; t < S * n; t += blockDim.x) {
                const int y = t / S, q = t - y * S;
                G[(size_t)y * n + c0 + q] = cscale(R[q * ld + y], inv_n2);
            }
            __syncthreads();
        }
        float2* out = xdisc + ((size_t)tile * P.n_bf + i) * P.npup;
        for (int p = threadIdx.x; p < P.npup; p += blockDim.x) {
            const int Kx = P.pup_x[p] - kix, Ky = P.pup_y[p] - kiy;
            out[p] = G[(size_t)freq_index(Ky, n) * n + freq_index(Kx, n)];
        }
        __syncthreads();
    }
}

cudaError_t launch_kk(const DevPlan& P, const Launch& L, int n_tiles, const float* I, float2* xdisc,
                      float2* scratch, const int32_t* status, cudaStream_t st) {
    const int grid = min(L.grid_kk, n_tiles * P.n_bf);
    k_kk<<<grid, kThreads, L.smem_kk, st>>>(P, n_tiles, I, xdisc, scratch, status);
    return cudaGetLastError();
}

cudaError_t launch_kk_grid(const DevPlan& P, int grid, size_t smem, int n_tiles, const float* I, float2* xdisc,
                           float2* scratch, const int32_t* status, cudaStream_t st) {
    grid = min(grid, n_tiles * P.n_bf);
    if (grid < 1) return cudaErrorInvalidConfiguration;
    k_kk<<<grid, kThreads, smem, st>>>(P, n_tiles, I, xdisc, scratch, status);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- aberration
// One block per tile (persistent). beta(r) = arg(X_i X_l^*) on every overlap
// row (Eq. 9). Stage 1 fits the wrapped differences of neighbouring rows,
// stage 2 runs `passes` refinements on the rows of Eq. 10. Products are
// accumulated per thread in FP32, summed across the block in FP64, and the
// 12 x 12 normal equations are solved in FP64 with the plan's Cholesky factors.
// CL: the tile's 512 threads spread over a cluster of K blocks of 512 / K threads; the warps' sums go
// to every block, and each adds them in warp order and solves, so K does not change the result.
// Bound by the latency of the rows' loads and, per sum, of the FP64 pipe: a call on one tile of
// 128, 256 and 512 pixels takes 0.041, 0.088 and 0.28 ms, against 0.12, 0.20 and 0.51 with one block,
// two rows in flight, each value summed over all lanes and one thread solving.
constexpr int kAbWarps = kThreads / 32;

struct AbShared {
    double s12[2][kAbWarps * 12], s1[2][kAbWarps];      // warps' sums, two sets in turn: a block of a
                                                        // cluster may be one sum ahead of another
    double L[2][144], rd[2][12];                        // factors of the two stages, 1 / their diagonals
    double cc[12], cbest[12];
    float cf[12];
};

// p[0] = v in every block of the tile
template <bool CL>
__device__ __forceinline__ void st_all(double* p, double v) {
    if constexpr (!CL) {
        *p = v;
    } else {
        const uint32_t a = (uint32_t)__cvta_generic_to_shared(p), K = cta_count();
        for (uint32_t q = 0; q < K; ++q) {
            uint32_t ra;
            asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(a), "r"(q));
            asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
        }
    }
}

// Solution of L L^T x = b by the lanes of a warp, lane i < 12 with b_i in and x_i out: as each
// unknown is found, the lanes of those to come take its term off. rd: 1 / L_ii.
__device__ __forceinline__ double chol_solve12(const double* L, const double* rd, double b) {
    const int lane = threadIdx.x & 31;
    double y = b;
    for (int j = 0; j < 12; ++j) {
        const double yj = __shfl_sync(0xffffffffu, y, j) * rd[j];
        if (lane == j) y = yj;
        if (lane > j && lane < 12) y -= L[lane * 12 + j] * yj;
    }
    for (int j = 11; j >= 0; --j) {
        const double xj = __shfl_sync(0xffffffffu, y, j) * rd[j];
        if (lane == j) y = xj;
        if (lane < j) y -= L[j * 12 + lane] * xj;
    }
    return y;
}

// Sum of the tile's g[12] (FP64 from here on), then cc = (add ? cc : 0) + the solution of
// stage `which`, cf = cc in FP32. The warp's sum halves the values with the lanes (13 FP64 adds a
// lane where a sum of each value over all lanes takes 60; the FP64 pipe adds 2 a clock and SM).
template <bool CL>
__device__ void sum_solve12(const float (&g)[12], AbShared& S, int& turn, int vt, int which, bool add) {
    constexpr unsigned kAll = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4, h2 = lane & 2;
    double a[6], b[3], c[2];
#pragma unroll
    for (int i = 0; i < 6; ++i) {
        const float other = __shfl_xor_sync(kAll, h16 ? g[i] : g[6 + i], 16);
        a[i] = (double)(h16 ? g[6 + i] : g[i]) + (double)other;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double other = __shfl_xor_sync(kAll, h8 ? a[i] : a[3 + i], 8);
        b[i] = (h8 ? a[3 + i] : a[i]) + other;
    }
    {
        const double o0 = __shfl_xor_sync(kAll, h4 ? b[0] : b[2], 4), o1 = __shfl_xor_sync(kAll, b[1], 4);
        c[0] = (h4 ? b[2] : b[0]) + o0;                 // value 2 or 0
        c[1] = b[1] + o1;
    }
    double d = (h2 ? c[1] : c[0]) + __shfl_xor_sync(kAll, h2 ? c[0] : c[1], 2);
    d += __shfl_xor_sync(kAll, d, 1);
    // lanes with both bits of (4, 2) set hold value 1 once more
    if (!(lane & 1) && !(h4 && h2))
        st_all<CL>(S.s12[turn] + (vt >> 5) * 12 + 6 * h16 + 3 * h8 + (h2 ? 1 : h4 ? 2 : 0), d);
    tile_sync<CL>();
    if (threadIdx.x < 32) {
        const int i = min(lane, 11);
        double t = 0;
        for (int w = 0; w < kAbWarps; ++w) t += S.s12[turn][w * 12 + i];
        const double x = chol_solve12(S.L[which], S.rd[which], t);
        if (lane < 12) {
            const double v = add ? S.cc[lane] + x : x;
            S.cc[lane] = v;
            S.cf[lane] = (float)v;
        }
    }
    turn ^= 1;
    __syncthreads();
}

// The 12 basis differences of row r: three 16-byte loads (scalar loads of a 48-byte row by
// 32 lanes take 12 instructions of 12 lines each)
struct Row12 {
    float a[12];
    __device__ Row12(const float* __restrict__ rows, int r) {
        const float4* p = reinterpret_cast<const float4*>(rows) + (size_t)3 * r;
#pragma unroll
        for (int q = 0; q < 3; ++q) {
            const float4 v = __ldg(p + q);
            a[4 * q] = v.x;
            a[4 * q + 1] = v.y;
            a[4 * q + 2] = v.z;
            a[4 * q + 3] = v.w;
        }
    }
    __device__ float operator[](int z) const { return a[z]; }
};

// Refinement passes c <- c + LS(wrap(beta - D c)) from the coefficients in
// cc / cf (shared).
template <bool CL>
__device__ void value_passes(const DevPlan& P, const float* beta, int passes, AbShared& S, int& turn, int vt) {
    for (int pass = 0; pass < passes; ++pass) {
        float g[12];
        for (int z = 0; z < 12; ++z) g[z] = 0.f;
#pragma unroll (CL ? 4 : 2)
        for (int r = vt; r < P.nrows; r += kThreads) {
            const Row12 A(P.row_A, r);
            float pred = 0.f;
            for (int z = 0; z < 12; ++z) pred += A[z] * S.cf[z];
            const float e = wrap_pi(beta[r] - pred);
            for (int z = 0; z < 12; ++z) g[z] += A[z] * e;
        }
        sum_solve12<CL>(g, S, turn, vt, 1, true);
    }
}

// Sum of the squared wrapped residuals of cf, in every thread.
template <bool CL>
__device__ double value_residual(const DevPlan& P, const float* beta, AbShared& S, int& turn, int vt) {
    double res = 0;
#pragma unroll (CL ? 4 : 2)
    for (int r = vt; r < P.nrows; r += kThreads) {
        const Row12 A(P.row_A, r);
        float pred = 0.f;
        for (int z = 0; z < 12; ++z) pred += A[z] * S.cf[z];
        const float e = wrap_pi(beta[r] - pred);
        res += (double)(e * e);
    }
    for (int o = 16; o > 0; o >>= 1) res += __shfl_xor_sync(0xffffffffu, res, o);
    if ((threadIdx.x & 31) == 0) st_all<CL>(S.s1[turn] + (vt >> 5), res);
    tile_sync<CL>();
    double t = 0;
    for (int w = 0; w < kAbWarps; ++w) t += S.s1[turn][w];
    turn ^= 1;
    return t;
}

// c0 [tiles][15] (may be NULL): learned coefficients. Tiles marked
// APIC_TILE_LEARNED take c0 as their result. With `warm`, every solved tile
// also runs the refinement passes from c0 and keeps whichever of the two
// solutions leaves the smaller wrapped residual (then sets APIC_TILE_WARM).
template <bool CL>
__global__ void __launch_bounds__(kThreads, CL ? 1 : 2)
k_aberration(DevPlan P, int n_tiles, const float2* __restrict__ xdisc, float* __restrict__ zern,
             float* __restrict__ beta_scratch, int passes, int32_t* __restrict__ status,
             const float* __restrict__ c0, int warm) {
    __shared__ AbShared S;
    const int K = CL ? (int)cta_count() : 1, rank = CL ? (int)cta_rank() : 0;
    const int vt = rank * blockDim.x + threadIdx.x;         // of the tile's 512 threads
    float* beta = beta_scratch + (size_t)(blockIdx.x / K) * P.nrows;
    int turn = 0;
    for (int i = threadIdx.x; i < 288; i += blockDim.x) (&S.L[0][0])[i] = i < 144 ? P.Lgrad[i] : P.Lval[i - 144];
    if (threadIdx.x < 24) {
        const int w = threadIdx.x / 12, i = threadIdx.x - 12 * w;
        S.rd[w][i] = 1.0 / (w ? P.Lval : P.Lgrad)[i * 13];
    }
    tile_sync<CL>();                                        // and every block runs before any stores into it
    for (int tile = blockIdx.x / K; tile < n_tiles; tile += gridDim.x / K) {
        float* Z = zern + (size_t)tile * APIC_N_ZERNIKE;
        if (skip_tile(status, tile)) {
            if (vt < APIC_N_ZERNIKE) Z[vt] = 0.f;
            continue;
        }
        if (c0 && status && (status[tile] & APIC_TILE_LEARNED)) {
            if (vt < APIC_N_ZERNIKE) Z[vt] = vt < 3 ? 0.f : c0[(size_t)tile * APIC_N_ZERNIKE + vt];
            continue;
        }
        const float2* X = xdisc + (size_t)tile * P.n_bf * P.npup;
#pragma unroll 4
        for (int r = vt; r < P.nrows; r += kThreads) {
            const int il = __ldg(P.row_il + r);
            const float2 a = __ldg(X + (size_t)(il & 0xffff) * P.npup + __ldg(P.row_pi + r));
            const float2 b = __ldg(X + (size_t)(il >> 16) * P.npup + __ldg(P.row_pl + r));
            const float2 z = cmulc(a, b);
            beta[r] = atan2f(z.y, z.x);
        }
        tile_sync<CL>();
        float g[12];
        for (int z = 0; z < 12; ++z) g[z] = 0.f;
#pragma unroll (CL ? 2 : 1)
        for (int r = vt; r < P.nrows; r += kThreads) {
            const Row12 A(P.row_A, r);
            const float br = beta[r];
            const int nx = __ldg(P.row_nx + r), ny = __ldg(P.row_ny + r);
            const int jx = nx < 0 ? r : nx, jy = ny < 0 ? r : ny;
            const Row12 Ax(P.row_A, jx), Ay(P.row_A, jy);
            const float ex = wrap_pi(ldx<CL>(beta + jx) - br), ey = wrap_pi(ldx<CL>(beta + jy) - br);
            for (int z = 0; z < 12; ++z) {
                if (nx >= 0) g[z] += (Ax[z] - A[z]) * ex;
                if (ny >= 0) g[z] += (Ay[z] - A[z]) * ey;
            }
        }
        sum_solve12<CL>(g, S, turn, vt, 0, false);
        value_passes<CL>(P, beta, passes, S, turn, vt);
        bool won = false;
        if (c0 && warm) {
            const double res = value_residual<CL>(P, beta, S, turn, vt);
            if (threadIdx.x < 12) {
                S.cbest[threadIdx.x] = S.cc[threadIdx.x];
                S.cc[threadIdx.x] = c0[(size_t)tile * APIC_N_ZERNIKE + 3 + threadIdx.x];
                S.cf[threadIdx.x] = (float)S.cc[threadIdx.x];
            }
            __syncthreads();
            value_passes<CL>(P, beta, passes, S, turn, vt);
            const double res_w = value_residual<CL>(P, beta, S, turn, vt);
            won = res_w < res;
            if (!won && threadIdx.x < 12) S.cc[threadIdx.x] = S.cbest[threadIdx.x];
            __syncthreads();
        }
        if (vt < APIC_N_ZERNIKE) Z[vt] = vt < 3 ? 0.f : (float)S.cc[vt - 3];
        if (won && status && vt == 0) status[tile] |= APIC_TILE_WARM;
        tile_sync<CL>();                                    // cc and beta are overwritten for the next tile
    }
}

// Two blocks per tile while they all run at once (512 pixels, 8 + 24: 0.41 -> 0.28 ms for 1 tile,
// 0.65 -> 0.53 for 152; 304 tiles would take 1.03 instead of 0.79). Four or eight gain nothing
// more (0.26 ms for 1 tile): a thread's rows are then what a tile waits for.
cudaError_t launch_aberration(const DevPlan& P, const Launch& L, int n_tiles, const float2* xdisc, float* zern,
                              float* beta_scratch, int passes, int32_t* status, cudaStream_t st, const float* c0,
                              int warm) {
    const int slots = min(L.grid_ab, n_tiles);
    const int K = 2 * slots <= L.grid_ab ? 2 : 1;
    return cluster_launch(K > 1 ? k_aberration<true> : k_aberration<false>, K, slots, kThreads / K, 0, st, P, n_tiles,
                          xdisc, zern, beta_scratch, passes, status, c0, warm);
}

// ---------------------------------------------------------------- phase table
// phi[tile][p] = sum_j c_j Z_j(k_p / R) at every pupil point.
__global__ void k_phase(DevPlan P, int n_tiles, const float* __restrict__ zern, float* __restrict__ phi) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n_tiles * P.npup) return;
    const int tile = (int)(idx / P.npup), p = (int)(idx - (size_t)tile * P.npup);
    float z[12];
    zernike_4_15<float>((float)P.pup_x[p] / P.Rx, (float)P.pup_y[p] / P.Ry, z);
    const float* c = zern + (size_t)tile * APIC_N_ZERNIKE + 3;
    float v = 0.f;
    for (int j = 0; j < 12; ++j) v += c[j] * z[j];
    phi[idx] = v;
}

cudaError_t launch_phase(const DevPlan& P, int n_tiles, const float* zern, float* phi, cudaStream_t st) {
    const size_t total = (size_t)n_tiles * P.npup;
    k_phase<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(P, n_tiles, zern, phi);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- stitch
// Corrected spectrum X_i(K) exp(-j[phi(K + k_i) - phi(k_i)]) averaged over the
// discs covering each aperture point; zero where only darkfield reaches.
__global__ void k_stitch(DevPlan P, int n_tiles, const float2* __restrict__ xdisc, const float* __restrict__ phi,
                         float2* __restrict__ spec, const int32_t* __restrict__ status) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= (size_t)n_tiles * P.nap) return;
    const int tile = (int)(idx / P.nap), a = (int)(idx - (size_t)tile * P.nap);
    if (skip_tile(status, tile)) {
        spec[idx] = make_float2(0.f, 0.f);
        return;
    }
    const float* ph = phi + (size_t)tile * P.npup;
    const float2* X = xdisc + (size_t)tile * P.n_bf * P.npup;
    float2 acc = make_float2(0.f, 0.f);
    const int e0 = P.st_ptr[a], e1 = P.st_ptr[a + 1];
    for (int e = e0; e < e1; ++e) {
        const int i = P.st_img[e], p = P.st_pup[e];
        float sn, cs;
        sincosf(ph[p] - ph[P.led_pup[i]], &sn, &cs);
        acc = cadd(acc, cmul(X[(size_t)i * P.npup + p], make_float2(cs, -sn)));
    }
    spec[idx] = e1 > e0 ? cscale(acc, 1.f / (float)(e1 - e0)) : make_float2(0.f, 0.f);
}

cudaError_t launch_stitch(const DevPlan& P, int n_tiles, const float2* xdisc, const float* phi, float2* spec,
                          const int32_t* status, cudaStream_t st) {
    const size_t total = (size_t)n_tiles * P.nap;
    k_stitch<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(P, n_tiles, xdisc, phi, spec, status);
    return cudaGetLastError();
}

// ---------------------------------------------------------------- pupil
__global__ void k_pupil(DevPlan P, int n_tiles, const float* __restrict__ phi, float2* __restrict__ pupil,
                        const int32_t* __restrict__ status) {
    const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
    const size_t npix = (size_t)P.h * P.w;
    if (idx >= (size_t)n_tiles * npix) return;
    const int tile = (int)(idx / npix);
    const int r = (int)(idx - (size_t)tile * npix);
    const int ky = signed_freq(r / P.w, P.h), kx = signed_freq(r % P.w, P.w);
    float2 v = make_float2(0.f, 0.f);
    if (!skip_tile(status, tile) && kx >= -P.pup_ax && kx <= P.pup_ax && ky >= -P.pup_ay && ky <= P.pup_ay) {
        const int p = P.pup_lut[(ky + P.pup_ay) * (2 * P.pup_ax + 1) + kx + P.pup_ax];
        if (p >= 0) {
            float sn, cs;
            sincosf(phi[(size_t)tile * P.npup + p], &sn, &cs);
            v = make_float2(cs, sn);
        }
    }
    pupil[idx] = v;
}

cudaError_t launch_pupil(const DevPlan& P, int n_tiles, const float* phi, float2* pupil, const int32_t* status,
                         cudaStream_t st) {
    const size_t total = (size_t)n_tiles * P.h * P.w;
    k_pupil<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(P, n_tiles, phi, pupil, status);
    return cudaGetLastError();
}

}  // namespace apic

namespace apic {
__global__ void k_darkfield(DevPlan, int, const float*, const float*, float2*, char*, size_t, int, float, int32_t*,
                            unsigned long long*);
__global__ void k_synthesize(DevPlan, int, const float2*, float2*, const int32_t*);
__global__ void k_sim_images(DevPlan, int, const float2*, const float*, float, unsigned long long, float*, float2*);
__global__ void k_sim_object(DevPlan, int, const float2*, float2*);

int configure_kernel(int which, size_t smem) {
    const void* f = nullptr;
    switch (which) {
        case 0: f = (const void*)k_kk; break;
        case 1: f = (const void*)k_aberration<false>; break;
        case 2: f = (const void*)k_darkfield; break;
        case 3: f = (const void*)k_synthesize; break;
        case 4: f = (const void*)k_sim_images; break;
        case 5: f = (const void*)k_sim_object; break;
        default: return 0;
    }
    if (smem > 48 * 1024 && raise_smem_limit(f, smem) != cudaSuccess)
        return 0;
    int occ = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, f, kThreads, smem) != cudaSuccess) return 0;
    return occ;
}
}  // namespace apic
