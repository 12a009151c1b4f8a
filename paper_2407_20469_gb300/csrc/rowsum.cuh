// rowsum.cuh - inner products and scalars of the 512-pixel darkfield CG: one FP32 sum per
// row of unknowns, the rows' sums added whatever the blocks that computed them.
#pragma once

#include "common.cuh"

namespace apic {
inline namespace APIC_ARITH {

constexpr int kTotalNotFinite = 1 << 20;

// A positive total m 2^(exp - 63), the top bit of m set; m = 0 where it is 0 or negative, or
// (exp = kTotalNotFinite) one of its rows is infinite or NaN.
struct RowTotal {
    unsigned long long m;
    int exp;

    __device__ bool finite() const { return exp != kTotalNotFinite; }
    __device__ bool operator<=(const RowTotal& b) const {
        return finite() && (m == 0 || (b.m != 0 && (exp < b.exp || (exp == b.exp && m <= b.m))));
    }
    // this / b rounded to FP32: an approximate quotient of the top 24 bits plus the remainder over b
    __device__ float over(const RowTotal& b) const {
        const float ah = (float)(unsigned)(m >> 40), al = (float)(unsigned)(m >> 8) * 0x1p-32f;
        const float bh = (float)(unsigned)(b.m >> 40), bl = (float)(unsigned)(b.m >> 8) * 0x1p-32f;
        const float q = __fdividef(ah, bh);
        const float r = __fadd_rn(__fmaf_rn(-q, bh, ah), __fmaf_rn(-q, bl, al));
        return ldexpf(__fadd_rn(q, __fdividef(r, bh)), exp - b.exp);
    }
};

// Sum of the rows' FP32 sums rs[0 .. nU), nU < 512, in every lane of the calling warp: as 64-bit
// integers on the scale of the largest. Rows down to 2^-29 of it enter exactly, so the sum has
// no order; what smaller ones lose is below 2^-52 of it. Neither FP64 nor FP32 serves: the FP64
// pipe takes tens of cycles per warp instruction (the totals and quotients of a CG step there,
// by one warp: 2 % of the kernel; as plain divisions 5 %), and the totals grow with the third
// and fourth power of the intensities, beyond FP32 where the rows' sums still are not.
__device__ __forceinline__ RowTotal row_total(const float* rs, int nU) {
    const int lane = threadIdx.x & 31;
    unsigned top = 1;
#pragma unroll 4
    for (int b = lane; b < nU; b += 32) top = max(top, __float_as_uint(rs[b]) >> 23 & 255u);
    top = __reduce_max_sync(0xffffffffu, top);
    if (top == 255) return {0, kTotalNotFinite};
    long long t = 0;
#pragma unroll 4
    for (int b = lane; b < nU; b += 32) {
        const unsigned u = __float_as_uint(rs[b]), e = u >> 23 & 255u, shift = top - max(e, 1u);
        const long long v = (long long)((u & 0x7fffffu) | (e ? 0x800000u : 0u)) << 29;
        const long long q = shift < 64 ? v >> shift : 0;
        t += (int)u < 0 ? -q : q;
    }
    // across the lanes in three parts of 20 bits of t + 2^58 (|t| <= 16 2^53)
    const unsigned long long u = (unsigned long long)t + (1ull << 58);
    const unsigned long long s0 = __reduce_add_sync(0xffffffffu, (unsigned)u & 0xfffffu),
                             s1 = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 20) & 0xfffffu),
                             s2 = __reduce_add_sync(0xffffffffu, (unsigned)(u >> 40));
    t = (long long)(s0 + (s1 << 20) + (s2 << 40) - (32ull << 58));
    if (t <= 0) return {0, 0};
    const int lead = __clzll(t);
    return {(unsigned long long)t << lead, (int)top - 116 - lead};          // t 2^(top - 127 - 23 - 29)
}

// The CG's scalars, in shared memory (in registers across the passes they would push the
// passes' own values out). Every block of a tile forms its own from the same rows' sums, by
// its first warp (the other warps' turns would come before the result: all of them forming
// the scalars takes longer than one and a barrier). A step is called by the whole block,
// once a barrier of the tile's blocks has made the sums visible; its results are written
// again only behind further barriers.
struct CgScalars {
    RowTotal gamma, stop;
    float alpha, beta;
    int go, done;
};

// gamma = |C^H b|^2, beta = 0; true if gamma is 0. One that is not finite (intensities beyond
// what FP32 holds once multiplied) ends the solve at its first step, unconverged.
static __device__ __noinline__ bool cg_start(CgScalars* s, const float* rs, int nU, float tol) {
    if (threadIdx.x < 32) {
        const RowTotal g = row_total(rs, nU);
        if (threadIdx.x == 0) {
            const double stop = (double)tol * (double)tol * ldexp((double)g.m, g.finite() ? g.exp - 63 : 0);
            const long long bits = __double_as_longlong(stop);
            s->gamma = g;
            s->stop = {bits >> 52 ? (unsigned long long)bits << 11 | 1ull << 63 : 0, (int)(bits >> 52) - 1023};
            s->beta = 0.f;
            s->done = g.m == 0 && g.finite();
        }
    }
    __syncthreads();
    return s->done;
}

// alpha = gamma / delta; false if the solve ends here
static __device__ __noinline__ bool cg_alpha(CgScalars* s, const float* rs, int nU) {
    if (threadIdx.x < 32) {
        const RowTotal delta = row_total(rs, nU);
        if (threadIdx.x == 0) {
            const RowTotal gamma = s->gamma;
            s->go = delta.m != 0 && gamma.finite();
            s->alpha = gamma.over(delta);
        }
    }
    __syncthreads();
    return s->go;
}

// beta = gamma' / gamma, with the new gamma' in its place; true once it is within the tolerance
static __device__ __noinline__ bool cg_beta(CgScalars* s, const float* rs, int nU) {
    if (threadIdx.x < 32) {
        const RowTotal next = row_total(rs, nU);
        if (threadIdx.x == 0) {
            s->done = next <= s->stop;
            s->beta = next.over(s->gamma);
            s->gamma = next;
        }
    }
    __syncthreads();
    return s->done;
}

}  // inline namespace
}  // namespace apic
