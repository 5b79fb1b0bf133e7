// Pieces of the kernels that give a row a block of four warps, a thread per age
// bin, when there are too few rows to fill the SMs with a warp per row.
#pragma once

#include "sps_device.cuh"

namespace sps {

constexpr int kFewWarps = 4, kFewThreads = 32 * kFewWarps;
static_assert(kFewThreads == kMaxAges, "one thread per age bin");

// The sums of age_met_adjoint over the block's threads (thread t: age bin t, its
// m, pi and wbar in mi, pi, wb; v.wb and v.qb complete): gradient columns 1-8
// into out[] (the others 0).  Only warp 0 gets them (true), the same in each lane.
__device__ __forceinline__ bool few_adjoint(const Consts& c, const AgeView& v, const EdgeTables& et, const float* th,
                                            float lT10, float Mf, float mi, float pi, float wb,
                                            float (*sums)[SPS_NPARAM], float* out) {
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5, A = c.n_age, Zn = c.n_met;
    const float mu = th[5], sig = th[6] * (1.0f / 3.0f), isig = 1.0f / sig, fb = th[4];
    const float xT = (lT10 - mu) * isig, D = tri_cdf(xT);
    float a[SPS_NPARAM];
    const float w0 = t < A ? wb : 0.0f;
    const float d0 = t < A ? v.dm0[t] : 0.0f, d1 = t < A ? v.dm1[t] : 0.0f, d2 = t < A ? v.dm2[t] : 0.0f;
    a[0] = w0 * pi;
    a[1] = w0 * mi;
    a[2] = w0 * d0;
    a[3] = w0 * d1;
    a[4] = w0 * d2;
    a[5] = d0;
    a[6] = d1;
    a[7] = d2;
    a[8] = a[9] = a[10] = a[11] = 0.0f;
    // burst, edge by edge
    for (int e = t; e <= A; e += kFewThreads) {
        const float x = (fminf(et.age[e], lT10) - mu) * isig;
        const float dd = ((e < A) ? v.wb[e] : 0.0f) - ((e > 0) ? v.wb[e - 1] : 0.0f);
        const float tp = tri_pdf(x) * dd;
        a[8] += tp;
        a[9] = fmaf(x, tp, a[9]);
    }
    // metallicity, edge by edge
    if (t <= Zn && t < 32) {
        const float y = (et.lgz[t] - th[7]) * (1.0f / th[8]);
        const float dd = ((t < Zn) ? v.qb[t] : 0.0f) - ((t > 0) ? v.qb[t - 1] : 0.0f);
        a[10] = phi_(y) * dd;
        a[11] = phi_y(y) * dd;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < SPS_NPARAM; ++k) a[k] += __shfl_xor_sync(kFull, a[k], o);
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < SPS_NPARAM; ++k) sums[warp][k] = a[k];
    __syncthreads();
    if (warp != 0) return false;
    float sv = 0.0f;
    if (lane < SPS_NPARAM) sv = (sums[0][lane] + sums[1][lane]) + (sums[2][lane] + sums[3][lane]);
    auto sum = [&](int k) { return __shfl_sync(kFull, sv, k); };
    const float s_wp = sum(0), s_wm = sum(1), s_w0 = sum(2), s_w1 = sum(3), s_w2 = sum(4), s_d0 = sum(5), s_d1 = sum(6),
                s_d2 = sum(7), s_mu = sum(8), s_sg = sum(9), s_gz = sum(10), s_gs = sum(11);
    const float omf = 1.0f - fb, fa = fb * s_wp;
    const float tT = tri_pdf(xT), kb = fb * Mf / (sig * D), isz = 1.0f / th[8];
    out[0] = out[9] = out[10] = out[11] = 0.0f;
    out[1] = omf * s_w0 + fa * s_d0;
    out[2] = omf * s_w1 + fa * s_d1;
    out[3] = omf * s_w2 + fa * s_d2;
    out[4] = Mf * s_wp - s_wm;
    out[5] = kb * (s_mu + s_wp * tT);
    out[6] = kb * (s_sg + s_wp * xT * tT) * (1.0f / 3.0f);
    out[7] = s_gz * isz;
    out[8] = s_gs * isz;
    return true;
}

}  // namespace sps
