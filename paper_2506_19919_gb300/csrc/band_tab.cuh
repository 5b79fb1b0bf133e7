// Tabulated filter transmission (SPS_BAND_TABLE): the linear interpolant of
// samples T[0..n-1] taken at l = start + m * step (observed frame), zero
// outside the samples.  u = (l_obs - start) / step is the sample coordinate.
#pragma once

#include <cuda_runtime.h>

#include "df.cuh"

namespace sps {

// Double-float (samples as hi + lo), for the once-per-galaxy set-up (zero
// points, lambda_eff, c_SSP): T at sample coordinate u, which the caller has
// found inside the samples, and its slope dT/du (the segment holding u).
__device__ __forceinline__ Df tab_Tdf(const float* __restrict__ Th, const float* __restrict__ Tl, int n, Df u,
                                      Df& slope) {
    // u just below an integer rounds up to it in u.h: the segment is the one before
    const float fl = floorf(u.h);
    const int m = min(max((int)fl - (u.h == fl && u.l < 0.0f ? 1 : 0), 0), n - 2);
    const Df f = two_sum(u.h - (float)m, u.l);
    const Df t0{__ldg(Th + m), __ldg(Tl + m)}, t1{__ldg(Th + m + 1), __ldg(Tl + m + 1)};
    slope = df_sub(t1, t0);
    return df_add(t0, df_mul(f, slope));
}

// FP32, for the exact-path epilogues.
__device__ __forceinline__ float tab_T32(const float* __restrict__ T, int n, float u) {
    if (!(u >= 0.0f && u <= (float)(n - 1))) return 0.0f;
    const int m = min((int)u, n - 2);
    const float t0 = __ldg(T + m);
    return fmaf(u - (float)m, __ldg(T + m + 1) - t0, t0);
}

// dT/du of the interpolant, FP32 (the exact-path epilogues' redshift terms).
__device__ __forceinline__ float tab_dT32(const float* __restrict__ T, int n, float u) {
    if (!(u >= 0.0f && u <= (float)(n - 1))) return 0.0f;
    const int m = min((int)u, n - 2);
    return __ldg(T + m + 1) - __ldg(T + m);
}

}  // namespace sps
