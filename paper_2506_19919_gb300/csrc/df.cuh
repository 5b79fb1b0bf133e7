// Double-float arithmetic: a value as the unevaluated sum of two FP32 numbers
// (48 significant bits), for the per-galaxy set-up.  sm_103a does two FP64
// operations per clock and SM against 128 FP32 ones, so a 10-to-20-instruction
// double-float operation is three to six times cheaper than one FP64
// instruction and still far below the FP32 rounding of what the sums feed.
// Error-free transformations after Dekker (1971) and Knuth (TAOCP 2, 4.2.2);
// the rounding intrinsics keep the compiler from contracting them.
#pragma once

#include <cuda_runtime.h>

namespace sps {

struct Df {
    float h, l;
};

__device__ __forceinline__ Df df_from(double x) {
    const float h = (float)x;
    return Df{h, isfinite(h) ? (float)(x - (double)h) : 0.0f};
}
__device__ __forceinline__ double df_to(Df a) { return (double)a.h + (double)a.l; }
__device__ __forceinline__ Df two_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    const float t = __fsub_rn(s, a);
    return Df{s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
// |a| >= |b| or a == 0
__device__ __forceinline__ Df quick_sum(float a, float b) {
    const float s = __fadd_rn(a, b);
    return Df{s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ Df df_add(Df a, Df b) {
    const Df s = two_sum(a.h, b.h);
    return quick_sum(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ Df df_sub(Df a, Df b) { return df_add(a, Df{-b.h, -b.l}); }
__device__ __forceinline__ Df df_mul(Df a, Df b) {
    const float p = __fmul_rn(a.h, b.h);
    float e = __fmaf_rn(a.h, b.h, -p);
    e = __fmaf_rn(a.h, b.l, e);
    e = __fmaf_rn(a.l, b.h, e);
    return quick_sum(p, e);
}

// e^{-x} for 0 <= x <= 40 (u < 6 gives x < 18), relative error below 1e-13 (rms 1e-14): x = n ln2/32 + r with
// |r| <= ln2/64, e^{-x} = 2^{-n/32} e^{-r}.  tab[j] = 2^{-j/32} as Df (32
// entries, shared memory); ln2/32 is split in three parts, the first of 14
// bits so that n times it is exact; e^{-r} - 1 = -r + r^2/2 - r^3/6 + r^4/24
// - r^5/120 with the linear and quadratic terms in double-float (the rest is
// below 3e-7 and enters with 6e-8 relative rounding; r^6/720 < 3e-15).
__device__ __forceinline__ Df df_exp_neg(Df x, const float2* __restrict__ tab) {
    constexpr float c1 = 0x1.62e8p-6f, c2 = -0x1.e8082ep-21f, c3 = -0x1.8432a2p-48f;   // ln2 / 32
    const float nf = rintf(__fmul_rn(x.h, 46.166241308446829f));                        // 32 / ln2
    const float t = __fmaf_rn(-nf, c1, x.h);
    const float p = __fmul_rn(nf, c2);
    const Df r0 = two_sum(t, -p);
    const Df r = quick_sum(r0.h, __fadd_rn(r0.l, __fmaf_rn(-nf, c3, __fsub_rn(x.l, __fmaf_rn(nf, c2, -p)))));
    const float a = r.h;
    const float p2 = __fmul_rn(a, a);                                                   // r^2 = p2 + e2
    const float e2 = __fmaf_rn(a, a, -p2);
    const float q = __fmul_rn(__fmul_rn(p2, a), __fmaf_rn(a, __fmaf_rn(a, -1.0f / 120.0f, 1.0f / 24.0f), -1.0f / 6.0f));
    const Df s0 = two_sum(-a, 0.5f * p2);                                               // e^{-r} - 1
    const Df s = quick_sum(s0.h, __fadd_rn(s0.l, __fadd_rn(q, __fmaf_rn(r.l, a - 1.0f, 0.5f * e2))));
    const int n = (int)nf;
    const float2 tj = tab[n & 31];
    const float y = __fmul_rn(tj.x, s.h);
    float e = __fmaf_rn(tj.x, s.h, -y);
    e = __fmaf_rn(tj.x, s.l, e);
    e = __fmaf_rn(tj.y, s.h, e);
    const Df v = quick_sum(tj.x, y);
    const float sc = __int_as_float((127 - (n >> 5)) << 23);                            // 2^-(n / 32)
    const Df w = quick_sum(v.h, __fadd_rn(v.l, __fadd_rn(e, tj.y)));
    return Df{__fmul_rn(w.h, sc), __fmul_rn(w.l, sc)};
}

}  // namespace sps
