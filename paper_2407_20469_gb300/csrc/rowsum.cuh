// rowsum.cuh - inner products of the darkfield CG: one FP32 sum per row of unknowns, the
// rows' sums added in one fixed order whatever the blocks that computed them.
#pragma once

#include "common.cuh"

namespace apic {
inline namespace APIC_ARITH {

// A sum or scalar as an unevaluated pair hi + lo of floats (about 48 bits). The FP64 pipe
// issues one warp instruction in 16 cycles and its dependent latency is far higher than
// FP32's: a sum over the rows and a quotient in FP64 took 4.4 k cycles of a 29 k cycle
// iteration twice over (128-pixel tile, 8 blocks), these take a few hundred. The pairs
// are added with Knuth's two-sum; the results are step lengths rounded to FP32.
struct FF {
    float hi, lo;
};
__device__ __forceinline__ FF ff_two_sum(float a, float b) {
    const float s = __fadd_rn(a, b), z = __fsub_rn(s, a);
    return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, z)), __fsub_rn(b, z))};
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
    const FF s = ff_two_sum(a.hi, b.hi), t = ff_two_sum(a.lo, b.lo);
    const FF u = ff_two_sum(s.hi, __fadd_rn(s.lo, t.hi));       // normalised after each part
    return ff_two_sum(u.hi, __fadd_rn(u.lo, t.lo));
}
// a / b rounded to FP32: the FP32 quotient plus its exact remainder over b
__device__ __forceinline__ float ff_div(FF a, FF b) {
    const float q = __fdiv_rn(a.hi, b.hi);
    const float r = __fadd_rn(__fmaf_rn(-q, b.hi, a.hi), __fmaf_rn(-q, b.lo, a.lo));
    return __fadd_rn(q, __fdiv_rn(r, b.hi));
}
// sum of the rows' FP32 sums, in row order per lane, then across the lanes: every warp
// of every block gets the same value
__device__ __forceinline__ FF row_total(const float* rs, int nU) {
    FF t = {0.f, 0.f};
    for (int b = threadIdx.x & 31; b < nU; b += 32) t = ff_add(t, FF{rs[b], 0.f});
    for (int o = 16; o > 0; o >>= 1)
        t = ff_add(t, FF{__shfl_xor_sync(0xffffffffu, t.hi, o), __shfl_xor_sync(0xffffffffu, t.lo, o)});
    return t;
}

// The CG's stopping test gamma <= tol^2 gamma0; both sides scaled up for small gamma0, so
// that the product does not underflow
struct CgStop {
    float scale, value;
    __device__ CgStop(float tol, float gamma0)
        : scale(gamma0 > 1.f ? 1.f : 1.152921504606846976e18f), value(tol * (tol * (scale * gamma0))) {}
    __device__ bool reached(float gamma) const { return gamma * scale <= value; }
};

}  // inline namespace
}  // namespace apic
