// netconv.cuh - the 3x3 convolutions of the aberration network on the tensor cores:
// forward (ReLU, max-pool or global mean fused), data gradient and weight gradient.
//
// All three are implicit GEMMs over NHWC maps whose operands are staged once per block:
// the block's pixels with a halo of one (BF16, one pixel's channels contiguous), read by
// ldmatrix at the nine taps' offsets, so that a pixel is fetched from L2 once instead of
// nine times, and the weights in per-tap chunks through a cp.async pipeline.
// Products are mma.sync m16n8k16 (BF16 in, FP32 accumulate), taken in the order (dy, dx,
// channel) in the forward pass and the data gradient: the results do not depend on
// the tile shapes, so layers could be re-tiled without moving a rounding of the BF16
// activations (a tcgen05 form would, and the layers are small: bound by staging and
// launches, not by the tensor pipe).
// Measured (GB300, SM clock 2070 MHz): a training step of 64 tiles 1373 -> 383 us (forward,
// backward, AdamW and the gradients read back), features and forward pass of 512 tiles
// 2682 -> 1260 us, against one generic GEMM kernel that gathered every operand per tap,
// separate pooling, mean and mask kernels, and FP32 maps of the unpooled gradients.
#pragma once

#include <cuda_bf16.h>
#include <stdint.h>

#include <algorithm>

#include "common.cuh"

namespace apic {
namespace net {

__device__ __forceinline__ void mma_bf16(float (&d)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
    asm volatile(
        "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
        "{%0,%1,%2,%3};\n"
        : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(unsigned (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm4t(unsigned (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}
__device__ __forceinline__ void ldsm2t(unsigned (&r)[4], uint32_t a) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
                 : "=r"(r[0]), "=r"(r[1]) : "r"(a) : "memory");
}
// 16 bytes to shared memory, zeros where !valid (src is not read then)
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool valid) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(valid ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ unsigned pack_bf16(float a, float b) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
    return *reinterpret_cast<const unsigned*>(&h);
}
// 8 floats (two float4, 16-byte aligned source) -> 8 BF16 (one uint4)
__device__ __forceinline__ uint4 f8_to_bf16(const float* src) {
    const float4 a = reinterpret_cast<const float4*>(src)[0], b = reinterpret_cast<const float4*>(src)[1];
    return make_uint4(pack_bf16(a.x, a.y), pack_bf16(a.z, a.w), pack_bf16(b.x, b.y), pack_bf16(b.z, b.w));
}

// BF16 values between consecutive pixels (or rows) of C values in shared memory: eight
// rows of an ldmatrix start in different banks
__host__ __device__ constexpr int pad_row(int c) { return c == 8 ? 8 : c + 8; }

constexpr int kStages = 4;                 // weight chunks in flight

// ---------------------------------------------------------------- staging
// A block's pixels: rows y0 .. y0 + TH - 1 of IMG consecutive images (whole rows of H
// pixels), with a halo of one pixel of zeros beyond the map: halo pixel (i, r, c) at
// ((i (TH + 2) + r) (H + 2) + c), r = y - y0 + 1, c = x + 1.

// BF16 or FP32 map [image][y][x][C]; channels c0 .. c0 + CT - 1
template <int H, int C, int CT, int TH, int IMG, class T>
__device__ __forceinline__ void stage_map(const T* __restrict__ x, int img0, int n_img, int y0, int c0,
                                          __nv_bfloat16* xs) {
    constexpr int P = pad_row(CT), V = CT / 8, N = IMG * (TH + 2) * (H + 2) * V;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(xs);
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const int v = i % V, p = i / V, c = p % (H + 2) - 1, q = p / (H + 2), r = q % (TH + 2) - 1, im = q / (TH + 2);
        const int y = y0 + r;
        const bool ok = (unsigned)y < (unsigned)H && (unsigned)c < (unsigned)H && img0 + im < n_img;
        const T* src = x + (((size_t)(img0 + im) * H + y) * H + c) * C + c0 + 8 * v;
        if constexpr (sizeof(T) == 2) {
            cp16(base + (p * P + 8 * v) * 2, ok ? src : x, ok);
        } else {
            *reinterpret_cast<uint4*>(xs + p * P + 8 * v) = ok ? f8_to_bf16(src) : make_uint4(0, 0, 0, 0);
        }
    }
}

// Gradient of a convolution's pre-activation, dz = dr [r > 0], rounded to BF16, 8 channels
// at one pixel. Behind a max-pool, dr is the pooled map's gradient at the position the pool
// chose and 0 elsewhere (its value r there is the pooled value); behind the global mean, dr
// is the mean's gradient / HW.
template <int H, int C>
struct DzPool {
    const float* g;                // [image][H / 2][H / 2][C]
    const uint8_t* arg;
    const __nv_bfloat16* pool;
    __device__ uint4 at(int im, int y, int x, int c) const {
        const size_t i = (((size_t)im * (H / 2) + (y >> 1)) * (H / 2) + (x >> 1)) * C + c;
        const int pos = (y & 1) * 2 + (x & 1);
        const uint2 a = *reinterpret_cast<const uint2*>(arg + i);
        const uint4 pv = *reinterpret_cast<const uint4*>(pool + i);
        const float4 g0 = reinterpret_cast<const float4*>(g + i)[0], g1 = reinterpret_cast<const float4*>(g + i)[1];
        const float v[8] = {g0.x, g0.y, g0.z, g0.w, g1.x, g1.y, g1.z, g1.w};
        const __nv_bfloat16* pb = reinterpret_cast<const __nv_bfloat16*>(&pv);
        const uint8_t* ab = reinterpret_cast<const uint8_t*>(&a);
        unsigned w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            w[e] = pack_bf16(ab[2 * e] == pos && __bfloat162float(pb[2 * e]) > 0.f ? v[2 * e] : 0.f,
                             ab[2 * e + 1] == pos && __bfloat162float(pb[2 * e + 1]) > 0.f ? v[2 * e + 1] : 0.f);
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
};
template <int H, int C>
struct DzMean {
    const float* g;                // [image][ld], the first C columns
    int ld;
    const __nv_bfloat16* r;        // [image][H][H][C]
    __device__ uint4 at(int im, int y, int x, int c) const {
        const uint4 rv = *reinterpret_cast<const uint4*>(r + (((size_t)im * H + y) * H + x) * C + c);
        const __nv_bfloat16* rb = reinterpret_cast<const __nv_bfloat16*>(&rv);
        const float* gp = g + (size_t)im * ld + c;
        unsigned w[4];
#pragma unroll
        for (int e = 0; e < 4; ++e)
            w[e] = pack_bf16(__bfloat162float(rb[2 * e]) > 0.f ? gp[2 * e] / (float)(H * H) : 0.f,
                             __bfloat162float(rb[2 * e + 1]) > 0.f ? gp[2 * e + 1] / (float)(H * H) : 0.f);
        return make_uint4(w[0], w[1], w[2], w[3]);
    }
};

// dz of the block's pixels, channels c0 .. c0 + CT - 1; HALO: with the halo (the layout of
// stage_map), else the pixels alone, row by row
template <int H, int CT, int TH, int IMG, bool HALO, class DZ>
__device__ __forceinline__ void stage_dz(const DZ& dz, int img0, int n_img, int y0, int c0, __nv_bfloat16* xs) {
    constexpr int P = pad_row(CT), V = CT / 8, E = HALO ? 1 : 0;
    constexpr int N = IMG * (TH + 2 * E) * (H + 2 * E) * V;
    for (int i = threadIdx.x; i < N; i += blockDim.x) {
        const int v = i % V, p = i / V, x = p % (H + 2 * E) - E, q = p / (H + 2 * E), r = q % (TH + 2 * E) - E;
        const int im = img0 + q / (TH + 2 * E), y = y0 + r;
        const bool ok = (unsigned)y < (unsigned)H && (unsigned)x < (unsigned)H && im < n_img;
        *reinterpret_cast<uint4*>(xs + p * P + 8 * v) = ok ? dz.at(im, y, x, c0 + 8 * v) : make_uint4(0, 0, 0, 0);
    }
}

// ---------------------------------------------------------------- forward
// One block: BM = TH x H pixels of one image x BN output channels (blockIdx.y), WM x WN
// warps. r = relu(conv + bias) in BF16 to `out`; POOL: its 2 x 2 max-pool (first maximum in
// (dy, dx) order) and the chosen position; else (the last layer, one image per block) the
// global mean into hin[image][CO + 2], with (u, v) behind it.
template <int H, int CI, int CO, int BN, int TH, int WM, int WN>
struct ConvCfg {
    static constexpr int BM = TH * H, KC = CI == 8 ? 80 : CI, TAPS = CI == 8 ? 1 : 9;   // KC: k values per chunk
    static constexpr int ST = TAPS < kStages ? TAPS : kStages;
    static constexpr int P = pad_row(CI), WS = KC + 8, XN = (TH + 2) * (H + 2) * P + 8, WN_ = BN * WS;
    static constexpr int ES = BN + 8, NTHR = 32 * WM * WN;
    static constexpr size_t smem = (size_t)(XN + ST * WN_ > BM * ES ? XN + ST * WN_ : BM * ES) * 2;
};

template <int H, int CI, int CO, int BN, int TH, int WM, int WN, bool POOL, class T>
__global__ void __launch_bounds__(32 * WM * WN)
k_conv(const T* __restrict__ x, const __nv_bfloat16* __restrict__ w, int ldw, const float* __restrict__ bias,
       int bias_stride, __nv_bfloat16* __restrict__ out, __nv_bfloat16* __restrict__ pool, uint8_t* __restrict__ arg,
       const float* __restrict__ uv, float* __restrict__ hin) {
    using Cfg = ConvCfg<H, CI, CO, BN, TH, WM, WN>;
    constexpr int BM = Cfg::BM, P = Cfg::P, WS = Cfg::WS, ST = Cfg::ST, TAPS = Cfg::TAPS;
    constexpr int MI = BM / 16 / WM, NJ = BN / 16 / WN, NTHR = 32 * WM * WN;
    extern __shared__ float4 smem4[];
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(smem4);
    __nv_bfloat16* ws = xs + Cfg::XN;
    const int tiles = H / TH, img = blockIdx.x / tiles, y0 = (blockIdx.x % tiles) * TH, n0 = blockIdx.y * BN;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wm = warp / WN, wn = warp % WN;
    const uint32_t xa = (uint32_t)__cvta_generic_to_shared(xs), wa = (uint32_t)__cvta_generic_to_shared(ws);
    auto load_w = [&](int s) {                       // chunk s (a tap; CI == 8: all nine and zeros to 80)
        constexpr int V = (CI == 8 ? 80 : CI) / 8;
        for (int i = threadIdx.x; i < BN * V; i += NTHR) {
            const int v = i % V, n = i / V;
            const bool ok = CI != 8 || v < 9;
            cp16(wa + ((s % ST) * Cfg::WN_ + n * WS + 8 * v) * 2,
                 ok ? w + (size_t)(n0 + n) * ldw + s * CI + 8 * v : w, ok);
        }
    };
    stage_map<H, CI, CI, TH, 1>(x, img, img + 1, y0, 0, xs);
    if (CI == 8 && threadIdx.x == 0)                 // a zero pixel: the tenth tap of the last k chunk
        *reinterpret_cast<uint4*>(xs + Cfg::XN - 8) = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int s = 0; s < ST - 1 || (ST == 1 && s < 1); ++s) {
        load_w(s);
        cp_commit();
    }
    float acc[MI][2 * NJ][4];
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < 2 * NJ; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
    uint32_t arow[MI];                               // this lane's pixel row of each 16-row fragment
#pragma unroll
    for (int i = 0; i < MI; ++i) {
        const int m = (wm * MI + i) * 16 + (lane & 15);
        arow[i] = xa + ((m / H) * (H + 2) + m % H) * P * 2 + (CI == 8 ? 0 : (lane >> 4) * 16);
    }
    const uint32_t brow = wa + ((wn * NJ * 16 + (lane & 7) + ((lane >> 4) << 3)) * WS + ((lane >> 3) & 1) * 8) * 2;
    for (int s = 0; s < TAPS; ++s) {
        cp_wait<(ST > 1 ? ST - 2 : 0)>();
        __syncthreads();
        if (ST > 1) {
            if (s + ST - 1 < TAPS) load_w(s + ST - 1);
            cp_commit();
        }
        const uint32_t bs = brow + (s % ST) * Cfg::WN_ * 2;
        const uint32_t tap = ((s / 3) * (H + 2) + s % 3) * P * 2;
#pragma unroll
        for (int kc = 0; kc < Cfg::KC / 16; ++kc) {
            unsigned a[MI][4], b[NJ][4];
#pragma unroll
            for (int i = 0; i < MI; ++i) {
                if constexpr (CI == 8) {             // taps 2 kc and 2 kc + 1, one per half of the lanes
                    const int t = 2 * kc + (lane >> 4);
                    ldsm4(a[i], t < 9 ? arow[i] + ((t / 3) * (H + 2) + t % 3) * P * 2 : xa + (Cfg::XN - 8) * 2);
                } else {
                    ldsm4(a[i], arow[i] + tap + kc * 32);
                }
            }
#pragma unroll
            for (int j = 0; j < NJ; ++j) ldsm4(b[j], bs + j * 16 * WS * 2 + kc * 32);
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    mma_bf16(acc[i][2 * j], a[i], b[j][0], b[j][1]);
                    mma_bf16(acc[i][2 * j + 1], a[i], b[j][2], b[j][3]);
                }
        }
    }
    cp_wait<0>();
    __syncthreads();
    // the tile through shared memory: whole 16-byte rows out, pooling and mean from there
    __nv_bfloat16* es = xs;
    constexpr int ES = Cfg::ES, V = BN / 8;
    const int g = lane >> 2, tg = lane & 3;
#pragma unroll
    for (int j = 0; j < 2 * NJ; ++j) {
        const int n = wn * NJ * 16 + j * 8 + tg * 2;
        const float b0 = bias[(size_t)(n0 + n) * bias_stride], b1 = bias[(size_t)(n0 + n + 1) * bias_stride];
#pragma unroll
        for (int i = 0; i < MI; ++i)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int m = (wm * MI + i) * 16 + g + 8 * h;
                *reinterpret_cast<unsigned*>(es + m * ES + n) =
                    pack_bf16(fmaxf(acc[i][j][2 * h] + b0, 0.f), fmaxf(acc[i][j][2 * h + 1] + b1, 0.f));
            }
    }
    __syncthreads();
    const size_t px0 = ((size_t)img * H + y0) * H;
    for (int i = threadIdx.x; i < BM * V; i += NTHR) {
        const int v = i % V, m = i / V;
        *reinterpret_cast<uint4*>(out + (px0 + m) * CO + n0 + 8 * v) = *reinterpret_cast<const uint4*>(es + m * ES + 8 * v);
    }
    if constexpr (POOL) {
        constexpr int Ho = H / 2;
        for (int i = threadIdx.x; i < BM / 4 * V; i += NTHR) {
            const int v = i % V, q = i / V, px = q % Ho, py = q / Ho;
            alignas(16) __nv_bfloat16 best[8];
            alignas(8) uint8_t at[8];
#pragma unroll
            for (int s = 0; s < 4; ++s) {
                const uint4 u = *reinterpret_cast<const uint4*>(es + ((2 * py + (s >> 1)) * H + 2 * px + (s & 1)) * ES + 8 * v);
                const __nv_bfloat16* ub = reinterpret_cast<const __nv_bfloat16*>(&u);
#pragma unroll
                for (int e = 0; e < 8; ++e)
                    if (s == 0 || __bfloat162float(ub[e]) > __bfloat162float(best[e])) {
                        best[e] = ub[e];
                        at[e] = (uint8_t)s;
                    }
            }
            const size_t o = (((size_t)img * Ho + y0 / 2 + py) * Ho + px) * CO + n0 + 8 * v;
            *reinterpret_cast<uint4*>(pool + o) = *reinterpret_cast<const uint4*>(best);
            *reinterpret_cast<uint2*>(arg + o) = *reinterpret_cast<const uint2*>(at);
        }
    } else {
        static_assert(TH == H || POOL, "the mean needs the whole image");
        for (int n = threadIdx.x; n < BN; n += NTHR) {
            float s = 0.f;
            for (int p = 0; p < BM; ++p) s += __bfloat162float(es[p * ES + n]);
            hin[(size_t)img * (CO + 2) + n0 + n] = s / (float)BM;
        }
        if (blockIdx.y == 0 && threadIdx.x < 2)
            hin[(size_t)img * (CO + 2) + CO + threadIdx.x] = uv ? uv[2 * (size_t)img + threadIdx.x] : 0.f;
    }
}

// ---------------------------------------------------------------- data gradient
// gx(y, x, ci) = sum over taps and co of dz(y - dy + 1, x - dx + 1, co) W[co][(dy, dx, ci)],
// FP32. One block: TH rows of one image x BN input channels (blockIdx.y).
template <int H, int CI, int CO, int BN, int TH>
struct DgradCfg {
    static constexpr int BM = TH * H, P = pad_row(CO), WS = BN + 8;
    static constexpr int XN = (TH + 2) * (H + 2) * P, WC = CO * WS;
    static constexpr size_t smem = (size_t)(XN + (kStages - 1) * WC) * 2;
};

template <int H, int CI, int CO, int BN, int TH, int WM, int WN, class DZ>
__global__ void __launch_bounds__(32 * WM * WN)
k_dgrad(DZ dz, const __nv_bfloat16* __restrict__ w, int ldw, float* __restrict__ gx) {
    using Cfg = DgradCfg<H, CI, CO, BN, TH>;
    constexpr int P = Cfg::P, WS = Cfg::WS, ST = kStages - 1, NTHR = 32 * WM * WN;
    constexpr int MI = Cfg::BM / 16 / WM, NJ = BN / 16 / WN;
    extern __shared__ float4 smem4[];
    __nv_bfloat16* xs = reinterpret_cast<__nv_bfloat16*>(smem4);
    const int tiles = H / TH, img = blockIdx.x / tiles, y0 = (blockIdx.x % tiles) * TH, n0 = blockIdx.y * BN;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, wm = warp / WN, wn = warp % WN;
    const uint32_t xa = (uint32_t)__cvta_generic_to_shared(xs), wa = xa + Cfg::XN * 2;
    auto load_w = [&](int s) {
        constexpr int V = BN / 8;
        for (int i = threadIdx.x; i < CO * V; i += NTHR) {
            const int v = i % V, co = i / V;
            cp16(wa + ((s % ST) * Cfg::WC + co * WS + 8 * v) * 2, w + (size_t)co * ldw + s * CI + n0 + 8 * v, true);
        }
    };
#pragma unroll
    for (int s = 0; s < ST - 1; ++s) {
        load_w(s);
        cp_commit();
    }
    stage_dz<H, CO, TH, 1, true>(dz, img, img + 1, y0, 0, xs);
    float acc[MI][2 * NJ][4];
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < 2 * NJ; ++j)
#pragma unroll
            for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.f;
    uint32_t arow[MI];
#pragma unroll
    for (int i = 0; i < MI; ++i) {
        const int m = (wm * MI + i) * 16 + (lane & 15);
        arow[i] = xa + ((m / H) * (H + 2) + m % H) * P * 2 + (lane >> 4) * 16;
    }
    // k = output channel rows of the chunk, n contiguous: transposed ldmatrix
    const uint32_t brow = wa + (((lane & 7) + ((lane >> 3) & 1) * 8) * WS + wn * NJ * 16 + (lane >> 4) * 8) * 2;
    for (int s = 0; s < 9; ++s) {
        cp_wait<ST - 2>();
        __syncthreads();
        if (s + ST - 1 < 9) load_w(s + ST - 1);
        cp_commit();
        const uint32_t bs = brow + (s % ST) * Cfg::WC * 2;
        const uint32_t tap = ((2 - s / 3) * (H + 2) + 2 - s % 3) * P * 2;
#pragma unroll 4
        for (int kc = 0; kc < CO / 16; ++kc) {
            unsigned a[MI][4], b[NJ][4];
#pragma unroll
            for (int i = 0; i < MI; ++i) ldsm4(a[i], arow[i] + tap + kc * 32);
#pragma unroll
            for (int j = 0; j < NJ; ++j) ldsm4t(b[j], bs + (kc * 16 * WS + j * 16) * 2);
#pragma unroll
            for (int i = 0; i < MI; ++i)
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    mma_bf16(acc[i][2 * j], a[i], b[j][0], b[j][1]);
                    mma_bf16(acc[i][2 * j + 1], a[i], b[j][2], b[j][3]);
                }
        }
    }
    cp_wait<0>();
    const size_t px0 = ((size_t)img * H + y0) * H;
    const int g = lane >> 2, tg = lane & 3;
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int j = 0; j < 2 * NJ; ++j)
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                const int m = (wm * MI + i) * 16 + g + 8 * h, n = n0 + wn * NJ * 16 + j * 8 + tg * 2;
                *reinterpret_cast<float2*>(gx + (px0 + m) * CI + n) = make_float2(acc[i][j][2 * h], acc[i][j][2 * h + 1]);
            }
}

// ---------------------------------------------------------------- weight gradient
// gw[co][(dy, dx, ci)] += sum over pixels of dz(p, co) x(p + tap, ci), gw[co][9 CI] += sum
// of dz(p, co). One block: OT output channels (blockIdx.y) x CT input channels
// (blockIdx.z) x all nine taps, over every gridDim.x-th tile of IMG x TH rows; the
// accumulators of the nine taps stay in registers, so dz's fragments are loaded once for
// the nine. WO x WC warps split the channels, WP warps the pixels (their sums meet in
// shared memory). The blocks' sums are added to gw atomically (FP32; the order varies
// from run to run).
template <int H, int CI, int CO, int CT, int OT, int TH, int IMG_>
struct WgradCfg {
    static constexpr int IMG = IMG_, target = CI == 8 ? 304 : 152;   // target: blocks of a launch
    static constexpr int PX = IMG * TH * H, PD = pad_row(OT), PX_ = pad_row(CT);
    static constexpr int DN = PX * PD, XN = IMG * (TH + 2) * (H + 2) * PX_;
    static constexpr int LS = 9 * CT + 1;                        // row of the block's sums (WP > 1)
    static constexpr size_t in = (size_t)(DN + XN) * 2, sum = (size_t)OT * LS * sizeof(float);
    static constexpr size_t smem = in > sum ? in : sum;
};

template <int H, int CI, int CO, int CT, int OT, int TH, int IMG, int WO, int WC, int WP, class T, class DZ>
__global__ void __launch_bounds__(32 * WO * WC * WP)
k_wgrad(const T* __restrict__ x, DZ dz, int n_img, float* __restrict__ gw) {
    using Cfg = WgradCfg<H, CI, CO, CT, OT, TH, IMG>;
    constexpr int PD = Cfg::PD, PXS = Cfg::PX_, MI = OT / 16 / WO, NJ = CT / 8 / WC, ld = 9 * CI + 1;
    static_assert(NJ == 1 || NJ == 2, "one or two 8-channel tiles per warp");
    extern __shared__ float4 smem4[];
    __nv_bfloat16* ds = reinterpret_cast<__nv_bfloat16*>(smem4);
    __nv_bfloat16* xs = ds + Cfg::DN;
    const int co0 = blockIdx.y * OT, ci0 = blockIdx.z * CT;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int wp = warp % WP, wo = (warp / WP) % WO, wc = warp / (WP * WO);
    const uint32_t da = (uint32_t)__cvta_generic_to_shared(ds), xa = (uint32_t)__cvta_generic_to_shared(xs);
    float acc[9][MI][NJ][4], bsum[MI][4];
#pragma unroll
    for (int i = 0; i < MI; ++i) {
#pragma unroll
        for (int e = 0; e < 4; ++e) bsum[i][e] = 0.f;
#pragma unroll
        for (int s = 0; s < 9; ++s)
#pragma unroll
            for (int j = 0; j < NJ; ++j)
#pragma unroll
                for (int e = 0; e < 4; ++e) acc[s][i][j][e] = 0.f;
    }
    const bool bias = blockIdx.z == 0 && wc == 0;
    const unsigned one = 0x3F803F80u;                            // two BF16 ones
    const int groups = (n_img + IMG - 1) / IMG, tiles = groups * (H / TH);
    for (int t = blockIdx.x; t < tiles; t += gridDim.x) {
        const int img0 = t / (H / TH) * IMG, y0 = t % (H / TH) * TH;
        __syncthreads();                                         // the previous tile is consumed
        stage_map<H, CI, CT, TH, IMG>(x, img0, n_img, y0, ci0, xs);
        cp_commit();
        stage_dz<H, OT, TH, IMG, false>(dz, img0, n_img, y0, co0, ds);
        cp_wait<0>();
        __syncthreads();
        for (int k = wp; k < Cfg::PX / 16; k += WP) {
            // A(co, pixel) from dz[pixel][co]: lanes 0-7 pixels 0-7 / co 0-7, 8-15 co 8-15, 16-31 pixels 8-15
            unsigned a[MI][4];
            const uint32_t arow = da + ((k * 16 + (lane & 7) + (lane >> 4) * 8) * PD + wo * MI * 16 + ((lane >> 3) & 1) * 8) * 2;
#pragma unroll
            for (int i = 0; i < MI; ++i) ldsm4t(a[i], arow + i * 32);
            // B(pixel, ci) from x[halo pixel][ci]: lanes 0-15 pixels, lanes 16-31 the next 8 channels
            const int p = k * 16 + (lane & 15), im = p / (TH * H), r = p / H % TH, c = p % H;
            const uint32_t brow = xa + (((im * (TH + 2) + r) * (H + 2) + c) * PXS + wc * NJ * 8 + (NJ == 2 ? (lane >> 4) * 8 : 0)) * 2;
            if (bias) {
#pragma unroll
                for (int i = 0; i < MI; ++i) mma_bf16(bsum[i], a[i], one, one);
            }
#pragma unroll
            for (int s = 0; s < 9; ++s) {
                unsigned b[4];
                const uint32_t at = brow + ((s / 3) * (H + 2) + s % 3) * PXS * 2;
                if constexpr (NJ == 2)
                    ldsm4t(b, at);
                else
                    ldsm2t(b, at);
#pragma unroll
                for (int i = 0; i < MI; ++i) {
                    mma_bf16(acc[s][i][0], a[i], b[0], b[1]);
                    if constexpr (NJ == 2) mma_bf16(acc[s][i][1], a[i], b[2], b[3]);
                }
            }
        }
    }
    const int g = lane >> 2, tg = lane & 3;
    float* sum = reinterpret_cast<float*>(smem4);
    if constexpr (WP > 1) {
        __syncthreads();
        for (int i = threadIdx.x; i < OT * Cfg::LS; i += blockDim.x) sum[i] = 0.f;
        __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < MI; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int o = (wo * MI + i) * 16 + g + 8 * h;
            float* row = WP > 1 ? sum + o * Cfg::LS : gw + (size_t)(co0 + o) * ld + ci0;
            constexpr int step = WP > 1 ? CT : CI;               // from tap to tap
#pragma unroll
            for (int s = 0; s < 9; ++s)
#pragma unroll
                for (int j = 0; j < NJ; ++j) {
                    const int ci = (wc * NJ + j) * 8 + tg * 2;
                    atomicAdd(row + s * step + ci, acc[s][i][j][2 * h]);
                    atomicAdd(row + s * step + ci + 1, acc[s][i][j][2 * h + 1]);
                }
            if (bias && tg == 0) atomicAdd(WP > 1 ? row + 9 * CT : gw + (size_t)(co0 + o) * ld + 9 * CI, bsum[i][2 * h]);
        }
    if constexpr (WP > 1) {
        static_assert(CT == CI, "the block's sums are whole rows");
        __syncthreads();
        for (int i = threadIdx.x; i < OT * Cfg::LS; i += blockDim.x) atomicAdd(gw + (size_t)co0 * ld + i, sum[i]);
    }
}

}  // namespace net
}  // namespace apic
