// net.cu - the Zernike-predicting network: input features, BF16 tensor-core
// layers, training (loss, backward, AdamW) and the C interface apic_net_*.
//
// Input per tile: 8 channels f = log(|F(I)| / |F(I)(0)| + 1e-4) on the 64 x 64
// low-frequency crop (kx, ky in [-32, 32)) of each NA-matching image's
// intensity spectrum, plus the tile position (u, v). Layers, NHWC on the device:
//   conv3x3 8->32, ReLU, maxpool2 | conv 32->64, ReLU, pool | conv 64->128,
//   ReLU, pool | conv 128->256, ReLU, global mean | concat (u, v)
//   | dense 258->256, ReLU | dense 256->12 (Noll 4..15).
// Weights and the activations that feed a layer are BF16, products accumulate
// in FP32 on the tensor cores (mma.sync m16n8k16), gradients and the AdamW
// master weights are FP32. The convolutions (forward with ReLU, pool or mean; data and
// weight gradients) are the kernels of netconv.cuh; the dense layers one generic GEMM
// kernel whose operands are gathered through loader functors, with split-K and atomic
// accumulation for the weight gradients.
//
// Parameters: six matrices W_l [out_l][taps_l + 1] stored back to back in FP32,
// the bias in the last column; convolution taps are ordered (dy, dx, c_in),
// dense taps are the input features.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <type_traits>
#include <cstring>
#include <string>
#include <vector>

#include "../../include/apic.h"
#include "internal.cuh"
#include "netconv.cuh"
#include "regfft.cuh"
#include "t4grid.cuh"

namespace apic {
namespace net {

constexpr int kCrop = 64;
constexpr int kIn = 8;
constexpr int kHidden = 256;
constexpr int kOut = 12;
constexpr int kC0 = 8, kC1 = 32, kC2 = 64, kC3 = 128, kC4 = 256;
constexpr int kHin = kC4 + 2;

// FP32 parameters W_l [rows][taps + 1] back to back (off, ld); the BF16 copy the
// GEMMs read has its rows padded to a multiple of 8 values (offp, ldp) so that
// 16-byte vector loads stay aligned.
struct Layout {
    size_t off[6], offp[6];
    int rows[6], taps[6];
    size_t total, total_pad;
    Layout() {
        const int r[6] = {kC1, kC2, kC3, kC4, kHidden, kOut};
        const int t[6] = {9 * kC0, 9 * kC1, 9 * kC2, 9 * kC3, kHin, kHidden};
        size_t o = 0, op = 0;
        for (int l = 0; l < 6; ++l) {
            off[l] = o;
            offp[l] = op;
            rows[l] = r[l];
            taps[l] = t[l];
            o += (size_t)r[l] * (t[l] + 1);
            op += (size_t)r[l] * ((t[l] + 1 + 7) / 8 * 8);
        }
        total = o;
        total_pad = op;
    }
    __host__ __device__ int ld(int l) const { return taps[l] + 1; }
    __host__ __device__ int ldp(int l) const { return (taps[l] + 1 + 7) / 8 * 8; }
    // index in the padded copy of flat parameter i
    __device__ size_t padded(size_t i) const {
        int l = 5;
        while (l > 0 && i < off[l]) --l;
        const size_t q = i - off[l];
        const size_t r = q / (size_t)ld(l), c = q - r * (size_t)ld(l);
        return offp[l] + r * (size_t)ldp(l) + c;
    }
};

// ------------------------------------------------------------------ features
// One block per (tile, image), persistent: forward transform of every row,
// keep the 64 columns kx in [-32, 32), forward transform of those columns,
// keep ky in [-32, 32), log of the magnitude relative to the DC term (the
// image sum). Output NHWC: feat[tile][ky + 32][kx + 32][image].
// Blocks of 256 threads up to 256 pixels, as many per SM as the scratch of n x n values per SM
// holds (three at 256 pixels, two at 128, one at 64), one of 512 at 512: at 256 pixels the kernel
// waits for its shared-memory exchanges and loads, and 24 warps hide more of that than 16 do.
// Bound by the L1 pipeline (the exchanges, twiddles and the kept columns' way through scratch).
// The kept columns are stored in 4 x 4 tiles: a warp's load of two adjacent columns over 16
// rows then touches 4 lines instead of 16. 512 tiles of 256 pixels 628 -> 484 us, of 128 354 -> 276,
// 128 tiles of 512 pixels 507 -> 428 (2 % more since, for the image sum's rows in FP64).
template <int BN>
struct FeatCfg {
    static constexpr int threads = BN <= 16 ? 256 : 512, blocks = BN == 16 ? 3 : BN == 8 ? 2 : 1;
};

// An unevaluated sum hi + lo of floats; Knuth's two-sum makes it exact for two floats.
struct FF {
    float hi, lo;
};
__device__ __forceinline__ FF ff_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z))};
}

template <int BN>
__global__ void __launch_bounds__(FeatCfg<BN>::threads, FeatCfg<BN>::blocks)
k_features(DevPlan P, int n_tiles, const float* __restrict__ I, float* __restrict__ feat, float2* __restrict__ scratch) {
    constexpr int n = 16 * BN, HWS = HWSize<BN>::value, NHW = FeatCfg<BN>::threads / 16, S = Slots<BN>::value;
    extern __shared__ float4 smem4[];
    float2* hw_area = reinterpret_cast<float2*>(smem4);
    float2* tw = hw_area + NHW * HWS;
    __shared__ double red[32];
    make_step_twiddles(tw, P.tw_n, BN);
    __syncthreads();
    const int hw = threadIdx.x >> 4, t = threadIdx.x & 15;
    const HalfWarp h{t, (threadIdx.x & 16) ? 0xFFFF0000u : 0x0000FFFFu, hw_area + hw * HWS};
    float2* G = scratch + (size_t)blockIdx.x * n * kCrop;   // [row][kept column] in 4 x 4 tiles
    const int t_col = t4_col(t), t_row = t4_row(t, kCrop);
    const int nprob = n_tiles * kIn;
    for (int prob = blockIdx.x; prob < nprob; prob += gridDim.x) {
        const int tile = prob / kIn, i = prob - tile * kIn;
        const float* img = I + ((size_t)tile * P.n_img + i) * n * n;
        // the image's sum on the way: a thread's pixels of a row as a float pair (an FP64 add per
        // pixel kept the FP64 pipe busy for a quarter of the kernel's time), rows and threads in
        // FP64. In float64 emulation the sum is then within 2e-15 of exact, as with FP64 adds
        // throughout; one float pair for all of a thread's rows was within 2.5e-13.
        double total = 0.0;
        for (int r = hw; r < n; r += NHW) {
            float2 v[BN], o[S][16];
            FF sum = {0.f, 0.f};
            float2* Gr = G + t4_row(r, kCrop) + t_col;
#pragma unroll
            for (int j = 0; j < BN; ++j) {
                v[j] = make_float2(img[(size_t)r * n + t + 16 * j], 0.f);
                const FF q = ff_two_sum(sum.hi, v[j].x);
                sum = {q.hi, sum.lo + q.lo};
            }
            total += (double)sum.hi + (double)sum.lo;
            fft_a<BN, false>(v, o, h, tw);
#pragma unroll
            for (int sl = 0; sl < S; ++sl)
                if (t + 16 * sl < BN) {
#pragma unroll
                    for (int k1 = 0; k1 < 16; ++k1) {
                        const int kx = t + 16 * sl + BN * k1;
                        const int sx = kx < n / 2 ? kx : kx - n;        // t + a multiple of 4
                        if (sx >= -kCrop / 2 && sx < kCrop / 2) Gr[4 * (sx - t + kCrop / 2)] = o[sl][k1];
                    }
                }
        }
        const double s = block_sum(total, red);     // (a barrier)
        const float inv_dc = s > 0 ? (float)(1.0 / s) : 0.f;
        float* f = feat + (size_t)tile * kCrop * kCrop * kIn + i;
        for (int c = hw; c < kCrop; c += NHW) {
            float2 v[BN], o[S][16];
            const float2* Gc = G + t_row + t4_col(c);
#pragma unroll
            for (int j = 0; j < BN; ++j) v[j] = Gc[16 * j * kCrop];
            fft_a<BN, false>(v, o, h, tw);
#pragma unroll
            for (int sl = 0; sl < S; ++sl)
                if (t + 16 * sl < BN) {
#pragma unroll
                    for (int k1 = 0; k1 < 16; ++k1) {
                        const int ky = t + 16 * sl + BN * k1;
                        const int sy = ky < n / 2 ? ky : ky - n;
                        if (sy >= -kCrop / 2 && sy < kCrop / 2)
                            f[((size_t)(sy + kCrop / 2) * kCrop + c) * kIn] =
                                logf(sqrtf(cabs2(o[sl][k1])) * inv_dc + 1e-4f);
                    }
                }
        }
        __syncthreads();
    }
}

size_t features_smem(int BN) {
    return (size_t)(BN <= 16 ? 16 : 32) * std::max(17 * BN, 16 * (BN + 1)) * sizeof(float2) + (size_t)2 * 16 * BN * sizeof(float2);
}

// ------------------------------------------------------------------ GEMM
// C(m, n) = sum_k A(m, k) B(k, n): bf16 operands, fp32 accumulation.
// Block tile 32 x 32 x 64, four warps of 16 x 16; blockIdx.z splits K (the
// epilogue must then accumulate atomically). The dense layers are small (a few hundred on
// each side) and their operands come from loads that wait on nothing else: what counts is
// the number of blocks and of loads in flight. So the tile is small, a thread's 32 loads of
// a step are all issued at once, a warp's lanes hold neighbouring rows (loads of transposed
// operands are then contiguous), and a step's operands are loaded under the one before.
// A training step of 64 tiles 378 -> 338 us, of 16 tiles 277 -> 248 (64 x 64 x 32 tiles, four loads
// in flight and nothing loaded ahead before); features and forward of 512 tiles 984 -> 966.
constexpr int kBM = 32, kBN = 32, kBK = 64, kLD = kBK + 8;

// Staging of 16 consecutive k of one A row (m fixed) or one B column (n fixed)
// into 16 BF16 values (16-byte aligned). Loaders whose data is
// contiguous along k provide segA / segB with vector loads; the others go
// through their element loaders.
template <class F, class = void>
struct HasSegA : std::false_type {};
template <class F>
struct HasSegA<F, std::void_t<decltype(std::declval<const F&>().segA(0, 0, 0, (__nv_bfloat16*)nullptr))>>
    : std::true_type {};
template <class F, class = void>
struct HasSegB : std::false_type {};
template <class F>
struct HasSegB<F, std::void_t<decltype(std::declval<const F&>().segB(0, 0, 0, (__nv_bfloat16*)nullptr))>>
    : std::true_type {};

__device__ __forceinline__ void zero16(__nv_bfloat16* dst) {
    reinterpret_cast<uint4*>(dst)[0] = make_uint4(0, 0, 0, 0);
    reinterpret_cast<uint4*>(dst)[1] = make_uint4(0, 0, 0, 0);
}

template <class F>
__device__ __forceinline__ void stage_a(const F& f, bool valid, int m, int k0, int kend, __nv_bfloat16* dst) {
    if (!valid) {
        zero16(dst);
    } else if constexpr (HasSegA<F>::value) {
        f.segA(m, k0, kend, dst);
    } else {
#pragma unroll
        for (int c = 0; c < 16; ++c) dst[c] = __float2bfloat16(k0 + c < kend ? f(m, k0 + c) : 0.f);
    }
}

template <class F>
__device__ __forceinline__ void stage_b(const F& f, bool valid, int n, int k0, int kend, __nv_bfloat16* dst) {
    if (!valid) {
        zero16(dst);
    } else if constexpr (HasSegB<F>::value) {
        f.segB(k0, kend, n, dst);
    } else {
#pragma unroll
        for (int c = 0; c < 16; ++c) dst[c] = __float2bfloat16(k0 + c < kend ? f(k0 + c, n) : 0.f);
    }
}

template <class LA, class LB, class EP>
__global__ void __launch_bounds__(128) k_gemm(int M, int N, int K, int k_split, LA la, LB lb, EP ep) {
    __shared__ __align__(16) __nv_bfloat16 As[kBM * kLD];
    __shared__ __align__(16) __nv_bfloat16 Bs[kBN * kLD];
    const int m0 = blockIdx.y * kBM, n0 = blockIdx.x * kBN;
    const int kb = blockIdx.z * k_split, ke = min(K, kb + k_split);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wm = (warp >> 1) * 16, wn = (warp & 1) * 16;
    const int g = lane >> 2, tg = lane & 3;
    float acc[2][4] = {};
    // staging: thread -> (row `lane` of the tile, 16 consecutive k from sc)
    const int sc = warp * 16;
    const int am = m0 + lane, bn = n0 + lane;
    __align__(16) __nv_bfloat16 ra[16], rb[16];
    stage_a(la, am < M, am, kb + sc, ke, ra);
    stage_b(lb, bn < N, bn, kb + sc, ke, rb);
    for (int k0 = kb; k0 < ke; k0 += kBK) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
            reinterpret_cast<uint4*>(As + lane * kLD + sc)[i] = reinterpret_cast<const uint4*>(ra)[i];
            reinterpret_cast<uint4*>(Bs + lane * kLD + sc)[i] = reinterpret_cast<const uint4*>(rb)[i];
        }
        __syncthreads();
        if (k0 + kBK < ke) {
            stage_a(la, am < M, am, k0 + kBK + sc, ke, ra);
            stage_b(lb, bn < N, bn, k0 + kBK + sc, ke, rb);
        }
#pragma unroll
        for (int kk = 0; kk < kBK; kk += 16) {
            const __nv_bfloat16* pa = As + (wm + g) * kLD + kk + tg * 2;
            const unsigned a[4] = {*reinterpret_cast<const unsigned*>(pa),
                                   *reinterpret_cast<const unsigned*>(pa + 8 * kLD),
                                   *reinterpret_cast<const unsigned*>(pa + 8),
                                   *reinterpret_cast<const unsigned*>(pa + 8 * kLD + 8)};
#pragma unroll
            for (int j = 0; j < 2; ++j) {
                const __nv_bfloat16* pb = Bs + (wn + j * 8 + g) * kLD + kk + tg * 2;
                mma_bf16(acc[j], a, *reinterpret_cast<const unsigned*>(pb),
                         *reinterpret_cast<const unsigned*>(pb + 8));
            }
        }
        __syncthreads();
    }
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
            const int m = m0 + wm + g + (e >= 2 ? 8 : 0);
            const int nn = n0 + wn + j * 8 + tg * 2 + (e & 1);
            if (m < M && nn < N) ep(m, nn, acc[j][e]);
        }
}

// splits > 1 only with an accumulating epilogue.
template <class LA, class LB, class EP>
cudaError_t gemm(int M, int N, int K, int splits, LA la, LB lb, EP ep, cudaStream_t st, long long* launches) {
    if (M <= 0 || N <= 0 || K <= 0) return cudaSuccess;
    splits = std::max(1, std::min(splits, (K + kBK - 1) / kBK));
    int k_split = (K + splits - 1) / splits;
    k_split = (k_split + kBK - 1) / kBK * kBK;
    splits = (K + k_split - 1) / k_split;
    const dim3 grid((N + kBN - 1) / kBN, (M + kBM - 1) / kBM, splits);
    k_gemm<<<grid, 128, 0, st>>>(M, N, K, k_split, la, lb, ep);
    if (launches) ++*launches;
    return cudaGetLastError();
}

// ---- operand loaders (A(m, k) or B(k, n), returning float)
struct WT {                 // B(k, n) = W[n][k]; rows padded to multiples of 8
    const __nv_bfloat16* w;
    int ld;
    __device__ float operator()(int k, int n) const { return __bfloat162float(w[(size_t)n * ld + k]); }
    __device__ void segB(int k0, int kend, int n, __nv_bfloat16* dst) const {
        const __nv_bfloat16* p = w + (size_t)n * ld + k0;
        if (k0 + 16 <= kend) {
            reinterpret_cast<uint4*>(dst)[0] = reinterpret_cast<const uint4*>(p)[0];
            reinterpret_cast<uint4*>(dst)[1] = reinterpret_cast<const uint4*>(p)[1];
            return;
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) dst[c] = k0 + c < kend ? p[c] : __float2bfloat16(0.f);
    }
};
struct WN {                 // B(k, n) = W[k][n]
    const __nv_bfloat16* w;
    int ld;
    __device__ float operator()(int k, int n) const { return __bfloat162float(w[(size_t)k * ld + n]); }
};
struct Mat {                // (r, c) -> p[r][c]
    const float* p;
    int ld;
    __device__ float operator()(int r, int c) const { return p[(size_t)r * ld + c]; }
    __device__ void segA(int r, int k0, int kend, __nv_bfloat16* dst) const {
        const float* q = p + (size_t)r * ld + k0;
        if (k0 + 16 <= kend && (ld & 3) == 0) {
            reinterpret_cast<uint4*>(dst)[0] = f8_to_bf16(q);
            reinterpret_cast<uint4*>(dst)[1] = f8_to_bf16(q + 8);
            return;
        }
#pragma unroll
        for (int c = 0; c < 16; ++c) dst[c] = __float2bfloat16(k0 + c < kend ? q[c] : 0.f);
    }
};
struct MatT {               // (r, c) -> p[c][r]
    const float* p;
    int ld;
    __device__ float operator()(int r, int c) const { return p[(size_t)c * ld + r]; }
};
struct MatBias {            // (r, c) -> p[r][c], 1 in column `cols` (bias column)
    const float* p;
    int ld, cols;
    __device__ float operator()(int r, int c) const { return c >= cols ? 1.f : p[(size_t)r * ld + c]; }
};

// ---- epilogues
struct EpDense {            // fp32 acc + bias, optional ReLU
    float* out;
    const float* bias;
    int bias_stride, ld;
    bool relu;
    __device__ void operator()(int m, int n, float v) const {
        const float r = v + bias[(size_t)n * bias_stride];
        out[(size_t)m * ld + n] = relu ? fmaxf(r, 0.f) : r;
    }
};
struct EpOut {              // the network's outputs: fp32 acc + bias to y, and Noll 1..15 (1..3 zero) to out15
    float* y;
    float* out15;
    const float* bias;
    int bias_stride;
    __device__ void operator()(int m, int n, float v) const {
        const float r = v + bias[(size_t)n * bias_stride];
        y[(size_t)m * kOut + n] = r;
        if (out15) {
            float* o = out15 + (size_t)m * APIC_N_ZERNIKE;
            o[n + 3] = r;
            if (n < 3) o[n] = 0.f;
        }
    }
};
struct EpMask {             // gradient of a ReLU's input: v where its output h is positive
    float* out;
    const float* h;
    int ld;
    __device__ void operator()(int m, int n, float v) const {
        const size_t i = (size_t)m * ld + n;
        out[i] = h[i] > 0.f ? v : 0.f;
    }
};
struct EpStore {
    float* out;
    int ld;
    __device__ void operator()(int m, int n, float v) const { out[(size_t)m * ld + n] = v; }
};
struct EpAtomic {
    float* out;
    int ld;
    __device__ void operator()(int m, int n, float v) const { atomicAdd(out + (size_t)m * ld + n, v); }
};

// ------------------------------------------------------------------ other layers
// mean squared error over the batch and the 12 outputs (Noll 4..15 of the
// [b][15] targets) and its gradient
__global__ void k_loss(const float* __restrict__ y, const float* __restrict__ target, float* __restrict__ gy,
                       float* __restrict__ loss, int B) {
    __shared__ double red[32];
    double acc = 0;
    for (int i = threadIdx.x; i < B * kOut; i += blockDim.x) {
        const int b = i / kOut, j = i - b * kOut;
        const float d = y[i] - target[(size_t)b * APIC_N_ZERNIKE + 3 + j];
        gy[i] = 2.f * d / (float)(B * kOut);
        acc += (double)d * d;
    }
    acc = block_sum(acc, red);
    if (threadIdx.x == 0 && loss) *loss = (float)(acc / (B * kOut));
}

__global__ void k_cast_bf16(const float* __restrict__ src, __nv_bfloat16* __restrict__ dst, size_t n, Layout L) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
        dst[L.padded(i)] = __float2bfloat16(src[i]);
}

// AdamW with bias-corrected moments and decoupled weight decay; refreshes the bf16 copy.
__global__ void k_adamw(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                        float* __restrict__ v, __nv_bfloat16* __restrict__ pbf, size_t n, float lr, float b1, float b2,
                        float eps, float wd, float c1, float c2, Layout L) {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
        const float gi = g[i];
        const float mi = b1 * m[i] + (1.f - b1) * gi;
        const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
        m[i] = mi;
        v[i] = vi;
        const float pi = p[i] - lr * ((mi / c1) / (sqrtf(vi / c2) + eps) + wd * p[i]);
        p[i] = pi;
        pbf[L.padded(i)] = __float2bfloat16(pi);
    }
}

int blocks_for(size_t n) { return (int)std::max<size_t>(1, std::min<size_t>((n + 255) / 256, 4096)); }

}  // namespace net

// Features of n_tiles tiles (the first 8 images of each stack) with the plan's register
// transforms on at most `grid` SMs; `scratch` holds h * h complex values for each of them
// (a block uses h * 64).
cudaError_t launch_features(const DevPlan& P, int grid, int n_tiles, const float* I, float* feat, float2* scratch,
                            cudaStream_t st) {
    using namespace net;
    const int BN = P.h / 16;
    const size_t smem = features_smem(BN);
    auto launch = [&](auto kernel, int threads, int per_sm) -> cudaError_t {
        const int blocks = std::min(grid * per_sm, n_tiles * kIn);
        if (blocks < 1) return cudaSuccess;
        const cudaError_t e = raise_smem_limit((const void*)kernel, smem);
        if (e != cudaSuccess) return e;
        kernel<<<blocks, threads, smem, st>>>(P, n_tiles, I, feat, scratch);
        return cudaGetLastError();
    };
    switch (BN) {
        case 4: return launch(k_features<4>, FeatCfg<4>::threads, FeatCfg<4>::blocks);
        case 8: return launch(k_features<8>, FeatCfg<8>::threads, FeatCfg<8>::blocks);
        case 16: return launch(k_features<16>, FeatCfg<16>::threads, FeatCfg<16>::blocks);
        case 32: return launch(k_features<32>, FeatCfg<32>::threads, FeatCfg<32>::blocks);
        default: return cudaErrorInvalidValue;
    }
}

size_t feature_floats() { return (size_t)net::kCrop * net::kCrop * net::kIn; }

}  // namespace apic

using namespace apic;
using namespace apic::net;

struct apic_net {
    int max_batch = 0;
    Layout L;
    float *params = nullptr, *grads = nullptr, *m = nullptr, *v = nullptr;
    __nv_bfloat16* wbf = nullptr;            // bf16 copy of the parameters
    // forward state of the last apic_net_forward
    const float* in = nullptr;               // caller's features
    int last_batch = 0;
    __nv_bfloat16 *r[4] = {}, *pool[3] = {};
    uint8_t* arg[3] = {};
    float *hin = nullptr, *h4 = nullptr, *y = nullptr;
    // gradients of activations
    float *g_pool[3] = {}, *g_hin = nullptr, *g_h4 = nullptr, *g_y = nullptr;
    long long launches = 0;
    std::vector<void*> allocs;
};

namespace {

apic_status net_fail(apic_status s, const std::string& m) {
    record_error((int)s, m.c_str());
    return s;
}

#define NET_TRY(expr)                                                                                         \
    do {                                                                                                      \
        cudaError_t _e = (expr);                                                                              \
        if (_e != cudaSuccess) return net_fail(APIC_ECUDA, std::string(#expr) + ": " + cudaGetErrorString(_e)); \
    } while (0)

template <typename T>
bool nalloc(apic_net* n, T** p, size_t count) {
    if (cudaMalloc((void**)p, std::max<size_t>(count, 1) * sizeof(T)) != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return false;
    }
    n->allocs.push_back((void*)*p);
    return true;
}

// Launch shapes of the layers' kernels: blocks along the pixels of an image (or of the
// images of one tile), and along the output and input channels
template <class Cfg, int TILES, int GY, int GZ = 1>
struct Layer {
    using C = Cfg;
    enum { tiles = TILES, gy = GY, gz = GZ };                    // tiles: blocks along the pixels, per image
};
// forward: 128 or 256 pixels x 32 or 64 channels per block (64 x 64 for the last layer's 8 x 8 maps)
using C1 = Layer<ConvCfg<64, kC0, kC1, 32, 4, 8, 1>, 16, 1>;
using C2 = Layer<ConvCfg<32, kC1, kC2, 64, 4, 4, 2>, 8, 1>;
using C3 = Layer<ConvCfg<16, kC2, kC3, 64, 8, 4, 2>, 2, 2>;
using C4 = Layer<ConvCfg<8, kC3, kC4, 64, 8, 2, 2>, 1, 4>;
using D3 = Layer<DgradCfg<8, kC3, kC4, 32, 8>, 1, 4>;
using D2 = Layer<DgradCfg<16, kC2, kC3, 64, 4>, 4, 1>;
using D1 = Layer<DgradCfg<32, kC1, kC2, 32, 4>, 8, 1>;
// weight gradients: tiles counted per IMG images
using W3 = Layer<WgradCfg<8, kC3, kC4, 64, 64, 8, 2>, 1, 4, 2>;
using W2 = Layer<WgradCfg<16, kC2, kC3, 64, 64, 8, 1>, 2, 2, 1>;
using W1 = Layer<WgradCfg<32, kC1, kC2, 32, 64, 4, 1>, 8, 1, 1>;
using W0 = Layer<WgradCfg<64, kC0, kC1, 8, 32, 4, 1>, 16, 1, 1>;

template <class L, class K, class... A>
cudaError_t launch_layer(K kernel, dim3 grid, int threads, long long* launches, cudaStream_t st, A... args) {
    cudaError_t e = cudaSuccess;
    if (L::C::smem > 48 * 1024) e = raise_smem_limit((const void*)kernel, L::C::smem);
    if (e != cudaSuccess) return e;
    kernel<<<grid, threads, L::C::smem, st>>>(args...);
    ++*launches;
    return cudaGetLastError();
}
template <class L, class K, class... A>
cudaError_t conv(K kernel, int B, long long* launches, cudaStream_t st, A... args) {
    return launch_layer<L>(kernel, dim3(B * L::tiles, L::gy), L::C::NTHR, launches, st, args...);
}
template <class L, class K, class... A>
cudaError_t dgrad(K kernel, int B, long long* launches, cudaStream_t st, A... args) {
    return launch_layer<L>(kernel, dim3(B * L::tiles, L::gy), 256, launches, st, args...);
}
// about one block per SM over all channel tiles (two in the first layer, whose blocks are small):
// each adds its sums to the gradient once
template <class L, class K, class... A>
cudaError_t wgrad(K kernel, int B, long long* launches, cudaStream_t st, A... args) {
    const int img = L::C::IMG, tiles = (B + img - 1) / img * L::tiles;
    const int split = std::max(1, std::min<int>(tiles, L::C::target / (L::gy * L::gz)));
    return launch_layer<L>(kernel, dim3(split, L::gy, L::gz), 256, launches, st, args...);
}

// split-K factor of a dense layer's weight-gradient GEMM
int split_for(long long K) { return (int)std::max(1LL, std::min(512LL, K / 256)); }

}  // namespace

namespace apic {

// Forward pass on `B` tiles; out15 [B][15] (Noll 1..3 zero) may be NULL.
cudaError_t net_predict(apic_net* n, int B, const float* feat, const float* uv, float* out15, cudaStream_t st) {
    const Layout& L = n->L;
    long long* nl = &n->launches;
    n->in = feat;
    n->last_batch = B;
    cudaError_t e;
#define NET_STEP(x)                          \
    if ((e = (x)) != cudaSuccess) return e;
    auto wl = [&](int l) { return n->wbf + L.offp[l]; };
    auto bl = [&](int l) { return n->params + L.off[l] + L.taps[l]; };
    NET_STEP((conv<C1>(k_conv<64, kC0, kC1, 32, 4, 8, 1, true, float>, B, nl, st, feat, wl(0), L.ldp(0), bl(0), L.ld(0),
                       n->r[0], n->pool[0], n->arg[0], nullptr, nullptr)));
    NET_STEP((conv<C2>(k_conv<32, kC1, kC2, 64, 4, 4, 2, true, __nv_bfloat16>, B, nl, st, n->pool[0], wl(1), L.ldp(1),
                       bl(1), L.ld(1), n->r[1], n->pool[1], n->arg[1], nullptr, nullptr)));
    NET_STEP((conv<C3>(k_conv<16, kC2, kC3, 64, 8, 4, 2, true, __nv_bfloat16>, B, nl, st, n->pool[1], wl(2), L.ldp(2),
                       bl(2), L.ld(2), n->r[2], n->pool[2], n->arg[2], nullptr, nullptr)));
    NET_STEP((conv<C4>(k_conv<8, kC3, kC4, 64, 8, 2, 2, false, __nv_bfloat16>, B, nl, st, n->pool[2], wl(3), L.ldp(3),
                       bl(3), L.ld(3), n->r[3], nullptr, nullptr, uv, n->hin)));
    NET_STEP(gemm(B, kHidden, kHin, 1, Mat{n->hin, kHin}, WT{wl(4), L.ldp(4)},
                  EpDense{n->h4, bl(4), L.ld(4), kHidden, true}, st, nl));
    NET_STEP(gemm(B, kOut, kHidden, 1, Mat{n->h4, kHidden}, WT{wl(5), L.ldp(5)}, EpOut{n->y, out15, bl(5), L.ld(5)}, st,
                  nl));
#undef NET_STEP
    return cudaSuccess;
}

int net_max_batch(const apic_net* n) { return n->max_batch; }
long long net_launches(const apic_net* n) { return n->launches; }

}  // namespace apic

extern "C" {

size_t apic_net_param_count(void) { return Layout().total; }

size_t apic_net_feature_count(void) { return feature_floats(); }

apic_status apic_net_create(int max_batch, apic_net** out) {
    if (!out) return net_fail(APIC_EINVAL, "NULL output handle");
    *out = nullptr;
    if (max_batch < 1 || max_batch > 65536) return net_fail(APIC_EINVAL, "max_batch must be in [1, 65536]");
    apic_net* n = new apic_net();
    n->max_batch = max_batch;
    const size_t P = n->L.total, B = (size_t)max_batch;
    bool ok = nalloc(n, &n->params, P) && nalloc(n, &n->grads, P) && nalloc(n, &n->m, P) && nalloc(n, &n->v, P) &&
              nalloc(n, &n->wbf, n->L.total_pad);
    const int C[4] = {kC1, kC2, kC3, kC4};
    int H = kCrop;
    for (int l = 0; l < 4 && ok; ++l) {
        ok = nalloc(n, &n->r[l], B * H * H * C[l]);
        if (ok && l < 3) {
            H /= 2;
            ok = nalloc(n, &n->pool[l], B * H * H * C[l]) && nalloc(n, &n->arg[l], B * H * H * C[l]) &&
                 nalloc(n, &n->g_pool[l], B * H * H * C[l]);
        }
    }
    ok = ok && nalloc(n, &n->hin, B * kHin) && nalloc(n, &n->g_hin, B * kHin) && nalloc(n, &n->h4, B * kHidden) &&
         nalloc(n, &n->g_h4, B * kHidden) && nalloc(n, &n->y, B * kOut) && nalloc(n, &n->g_y, B * kOut);
    if (!ok) {
        apic_net_destroy(n);
        return net_fail(APIC_ENOMEM, "network workspace allocation failed");
    }
    if (cudaMemset(n->params, 0, P * 4) != cudaSuccess || cudaMemset(n->grads, 0, P * 4) != cudaSuccess ||
        cudaMemset(n->m, 0, P * 4) != cudaSuccess || cudaMemset(n->v, 0, P * 4) != cudaSuccess ||
        cudaMemset(n->wbf, 0, n->L.total_pad * 2) != cudaSuccess) {
        cudaGetLastError();
        apic_net_destroy(n);
        return net_fail(APIC_ECUDA, "network initialisation failed");
    }
    *out = n;
    return APIC_OK;
}

apic_status apic_net_destroy(apic_net* n) {
    if (!n) return APIC_OK;
    cudaDeviceSynchronize();
    for (void* p : n->allocs) cudaFree(p);
    delete n;
    return APIC_OK;
}

apic_status apic_net_set_params(apic_net* n, const float* h, size_t count) {
    if (!n || !h || count != n->L.total) return net_fail(APIC_EINVAL, "expected apic_net_param_count() floats");
    NET_TRY(cudaDeviceSynchronize());
    NET_TRY(cudaMemcpy(n->params, h, count * 4, cudaMemcpyHostToDevice));
    k_cast_bf16<<<blocks_for(count), 256>>>(n->params, n->wbf, count, n->L);
    NET_TRY(cudaGetLastError());
    NET_TRY(cudaMemset(n->m, 0, count * 4));
    NET_TRY(cudaMemset(n->v, 0, count * 4));
    NET_TRY(cudaDeviceSynchronize());
    return APIC_OK;
}

// Value of key `key` in a flat JSON object: the string after it ("...") or the
// digits of a number; empty when absent. Enough for the checkpoint header, whose
// writer emits plain keys, strings and integers.
static std::string json_value(const std::string& js, const std::string& key) {
    const std::string k = "\"" + key + "\"";
    size_t p = js.find(k);
    if (p == std::string::npos) return "";
    p += k.size();
    while (p < js.size() && (js[p] == ' ' || js[p] == ':' || js[p] == '\t' || js[p] == '\n')) ++p;
    if (p >= js.size()) return "";
    if (js[p] == '"') {
        const size_t e = js.find('"', p + 1);
        return e == std::string::npos ? "" : js.substr(p + 1, e - p - 1);
    }
    size_t e = p;
    while (e < js.size() && js[e] >= '0' && js[e] <= '9') ++e;
    return js.substr(p, e - p);
}

apic_status apic_net_load(apic_net* n, const void* blob, size_t bytes) {
    static const char kMagic[8] = {'A', 'P', 'I', 'C', 'N', 'B', '1', '6'};
    if (!blob) return net_fail(APIC_EINVAL, "NULL blob");
    const unsigned char* b = static_cast<const unsigned char*>(blob);
    if (bytes < 12 || std::memcmp(b, kMagic, 8) != 0) return net_fail(APIC_EINVAL, "not an APICNB16 checkpoint");
    const size_t L = (size_t)b[8] | ((size_t)b[9] << 8) | ((size_t)b[10] << 16) | ((size_t)b[11] << 24);
    if (L > bytes - 12) return net_fail(APIC_EINVAL, "checkpoint header runs past the blob");
    const std::string head(reinterpret_cast<const char*>(b + 12), L);
    if (json_value(head, "format") != "apic-net-bf16") return net_fail(APIC_EINVAL, "checkpoint format is not apic-net-bf16");
    const std::string cs = json_value(head, "count");
    const Layout lay;
    if (cs.empty() || cs.size() > 12 || std::stoull(cs) != (unsigned long long)lay.total)
        return net_fail(APIC_EINVAL, "checkpoint count differs from apic_net_param_count()");
    if (bytes != 12 + L + 2 * lay.total) return net_fail(APIC_EINVAL, "checkpoint size does not match its count");
    if (!n) return APIC_OK;                          // validation only
    std::vector<float> v(lay.total);
    const unsigned char* q = b + 12 + L;
    for (size_t i = 0; i < lay.total; ++i) {
        const uint32_t bits = ((uint32_t)q[2 * i] | ((uint32_t)q[2 * i + 1] << 8)) << 16;
        std::memcpy(&v[i], &bits, 4);
    }
    return apic_net_set_params(n, v.data(), v.size());
}

apic_status apic_net_get_params(const apic_net* n, float* h, size_t count) {
    if (!n || !h || count != n->L.total) return net_fail(APIC_EINVAL, "expected apic_net_param_count() floats");
    NET_TRY(cudaDeviceSynchronize());
    NET_TRY(cudaMemcpy(h, n->params, count * 4, cudaMemcpyDeviceToHost));
    return APIC_OK;
}

apic_status apic_net_get_grads(const apic_net* n, float* h, size_t count) {
    if (!n || !h || count != n->L.total) return net_fail(APIC_EINVAL, "expected apic_net_param_count() floats");
    NET_TRY(cudaDeviceSynchronize());
    NET_TRY(cudaMemcpy(h, n->grads, count * 4, cudaMemcpyDeviceToHost));
    return APIC_OK;
}

apic_status apic_net_forward(apic_net* n, int batch, const float* feat, const float* uv, float* out15,
                             void* stream) {
    if (!n || !feat) return net_fail(APIC_EINVAL, "NULL network or features");
    if (batch < 1 || batch > n->max_batch) return net_fail(APIC_EINVAL, "batch must be in [1, max_batch]");
    if (reinterpret_cast<uintptr_t>(feat) & 15) return net_fail(APIC_EINVAL, "features must be 16-byte aligned");
    NET_TRY(net_predict(n, batch, feat, uv, out15, (cudaStream_t)stream));
    return APIC_OK;
}

apic_status apic_net_backward(apic_net* n, const float* target15, float* loss, void* stream) {
    if (!n || !target15) return net_fail(APIC_EINVAL, "NULL network or target");
    if (n->last_batch < 1) return net_fail(APIC_EINVAL, "backward needs a preceding forward");
    cudaStream_t st = (cudaStream_t)stream;
    const int B = n->last_batch;
    const Layout& L = n->L;
    long long* nl = &n->launches;
    NET_TRY(cudaMemsetAsync(n->grads, 0, L.total * sizeof(float), st));
    k_loss<<<1, 256, 0, st>>>(n->y, target15, n->g_y, loss, B);
    ++*nl;
    NET_TRY(cudaGetLastError());
    // dense 256 -> 12
    NET_TRY(gemm(kOut, L.ld(5), B, split_for(B), MatT{n->g_y, kOut}, MatBias{n->h4, kHidden, kHidden},
                 EpAtomic{n->grads + L.off[5], L.ld(5)}, st, nl));
    NET_TRY(gemm(B, kHidden, kOut, 1, Mat{n->g_y, kOut}, WN{n->wbf + L.offp[5], L.ldp(5)},
                 EpMask{n->g_h4, n->h4, kHidden}, st, nl));
    // dense 258 -> 256
    NET_TRY(gemm(kHidden, L.ld(4), B, split_for(B), MatT{n->g_h4, kHidden}, MatBias{n->hin, kHin, kHin},
                 EpAtomic{n->grads + L.off[4], L.ld(4)}, st, nl));
    NET_TRY(gemm(B, kHin, kHidden, 1, Mat{n->g_h4, kHidden}, WN{n->wbf + L.offp[4], L.ldp(4)}, EpStore{n->g_hin, kHin},
                 st, nl));
    // convolutions, last first: weights, then the gradient of the layer's input
    const DzMean<8, kC4> dz3{n->g_hin, kHin, n->r[3]};
    const DzPool<16, kC3> dz2{n->g_pool[2], n->arg[2], n->pool[2]};
    const DzPool<32, kC2> dz1{n->g_pool[1], n->arg[1], n->pool[1]};
    const DzPool<64, kC1> dz0{n->g_pool[0], n->arg[0], n->pool[0]};
    NET_TRY((wgrad<W3>(k_wgrad<8, kC3, kC4, 64, 64, 8, 2, 2, 4, 1, __nv_bfloat16, DzMean<8, kC4>>, B, nl, st, n->pool[2],
                       dz3, B, n->grads + L.off[3])));
    NET_TRY((dgrad<D3>(k_dgrad<8, kC3, kC4, 32, 8, 4, 2, DzMean<8, kC4>>, B, nl, st, dz3, n->wbf + L.offp[3], L.ldp(3),
                       n->g_pool[2])));
    NET_TRY((wgrad<W2>(k_wgrad<16, kC2, kC3, 64, 64, 8, 1, 2, 4, 1, __nv_bfloat16, DzPool<16, kC3>>, B, nl, st,
                       n->pool[1], dz2, B, n->grads + L.off[2])));
    NET_TRY((dgrad<D2>(k_dgrad<16, kC2, kC3, 64, 4, 4, 2, DzPool<16, kC3>>, B, nl, st, dz2, n->wbf + L.offp[2], L.ldp(2),
                       n->g_pool[1])));
    NET_TRY((wgrad<W1>(k_wgrad<32, kC1, kC2, 32, 64, 4, 1, 2, 4, 1, __nv_bfloat16, DzPool<32, kC2>>, B, nl, st,
                       n->pool[0], dz1, B, n->grads + L.off[1])));
    NET_TRY((dgrad<D1>(k_dgrad<32, kC1, kC2, 32, 4, 8, 1, DzPool<32, kC2>>, B, nl, st, dz1, n->wbf + L.offp[1], L.ldp(1),
                       n->g_pool[0])));
    NET_TRY((wgrad<W0>(k_wgrad<64, kC0, kC1, 8, 32, 4, 1, 1, 1, 8, float, DzPool<64, kC1>>, B, nl, st, n->in, dz0, B,
                       n->grads + L.off[0])));
    return APIC_OK;
}

apic_status apic_net_adamw(apic_net* n, float lr, float beta1, float beta2, float eps, float weight_decay, int step,
                           void* stream) {
    if (!n) return net_fail(APIC_EINVAL, "NULL network");
    if (step < 1 || !(lr >= 0.f) || !(beta1 >= 0.f && beta1 < 1.f) || !(beta2 >= 0.f && beta2 < 1.f) || !(eps > 0.f))
        return net_fail(APIC_EINVAL, "bad optimizer arguments");
    const size_t P = n->L.total;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    k_adamw<<<blocks_for(P), 256, 0, (cudaStream_t)stream>>>(n->params, n->grads, n->m, n->v, n->wbf, P, lr, beta1,
                                                              beta2, eps, weight_decay, c1, c2, n->L);
    ++n->launches;
    NET_TRY(cudaGetLastError());
    return APIC_OK;
}

apic_status apic_net_activation(const apic_net* n, int which, float* h, size_t count) {
    if (!n || !h) return net_fail(APIC_EINVAL, "NULL network or destination");
    const size_t B = (size_t)n->last_batch;
    if (B == 0) return net_fail(APIC_EINVAL, "no forward pass yet");
    if (which < 0 || which > 6) return net_fail(APIC_EINVAL, "which must be in [0, 6]");
    NET_TRY(cudaDeviceSynchronize());
    if (which < 4) {
        const int C[4] = {kC1, kC2, kC3, kC4}, H[4] = {64, 32, 16, 8};
        const size_t sz = B * H[which] * H[which] * C[which];
        if (count != sz) return net_fail(APIC_EINVAL, "activation size mismatch");
        std::vector<uint16_t> tmp(sz);
        NET_TRY(cudaMemcpy(tmp.data(), n->r[which], sz * 2, cudaMemcpyDeviceToHost));
        for (size_t i = 0; i < sz; ++i) {
            const uint32_t bits = (uint32_t)tmp[i] << 16;
            std::memcpy(h + i, &bits, 4);
        }
        return APIC_OK;
    }
    const float* src = which == 4 ? n->hin : which == 5 ? n->h4 : n->y;
    const size_t sz = B * (which == 4 ? kHin : which == 5 ? kHidden : kOut);
    if (count != sz) return net_fail(APIC_EINVAL, "activation size mismatch");
    NET_TRY(cudaMemcpy(h, src, sz * 4, cudaMemcpyDeviceToHost));
    return APIC_OK;
}

}  // extern "C"
