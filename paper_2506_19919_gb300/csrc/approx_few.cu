// Approximate photometry and log L + gradient of few independent rows (separable
// model, Eq. photo_integral_approx, App. D.1): one block of four warps per row.
//
// With fewer rows than the SMs hold warps, what a call takes is one row's serial
// chain (k_like_team and k_phot_team: one row per warp).  Here the chain is shared out:
// each warp integrates one group of 32 age bins and takes every fourth band; the
// sums over ages and bands meet in shared memory.
// A call on 64 rows of six bands takes 43 us against 54 (photometry 36 against
// 39), most of the rest in the host's part.
#include "few.cuh"

namespace sps {

namespace {

struct FewWork {
    float m[kMaxAges], dm0[kMaxAges], dm1[kMaxAges], dm2[kMaxAges], pi[kMaxAges], w[kMaxAges], wb[kMaxAges];
    float q[kMaxMets], qb[kMaxMets];
    float th[SPS_NPARAM];
    PanelScratch ps[kFewWarps];
    double Mp[kFewWarps];                          // the warps' parts of M = sum_i m_i
    // observed bands
    const float* ptr[kMaxBands];
    float4 dust[kMaxBands];
    double zp[kMaxBands];
    float mobs[kMaxBands], isig2[kMaxBands];
    float F[kMaxBands], Ah[kMaxBands], Al[kMaxBands], res[kMaxBands], gam[kMaxBands];
    float S[kMaxBands];
    // partial sums of the warps
    float wbp[kFewWarps][kMaxAges];
    float red[kFewThreads][kZnReg + 1];
    float sums[kFewWarps][SPS_NPARAM];
    double ll;
    float gd[4];
};

// kLike: log L and gradient (mag_out unused); otherwise magnitudes.
template <bool kLike>
__global__ void __launch_bounds__(kFewThreads)
k_approx_few(const __grid_constant__ Consts c, const Galaxies g, const float* __restrict__ theta,
             const int32_t* __restrict__ gal_idx, const float* __restrict__ mag_obs, const float* __restrict__ sigma,
             const uint32_t* __restrict__ mask, float* __restrict__ mag_out, float* __restrict__ ll_out,
             float* __restrict__ grad_out, int* __restrict__ nonfinite) {
    __shared__ FewWork s;
    __shared__ EdgeTables et;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int A = c.n_age, Zn = c.n_met, B = c.n_band, K = c.K;
    const int64_t row = blockIdx.x;
    const int64_t gi = gal_idx ? (int64_t)gal_idx[row] : row;
    const float xk = (lane < SPS_NPARAM) ? theta[row * SPS_NPARAM + lane] : 0.0f;
    if (!(__all_sync(kFull, isfinite(xk)) && gi >= 0 && gi < g.n)) {          // the same in every warp
        const float nan = __int_as_float(0x7fc00000);
        if (t == 0) atomicOr(nonfinite, 1);
        if (!kLike && t < B) mag_out[row * B + t] = nan;
        if (kLike && t == 0) ll_out[row] = nan;
        if (kLike && grad_out && t < SPS_NPARAM) grad_out[row * SPS_NPARAM + t] = nan;
        return;
    }
    const uint32_t all = (B >= 32) ? 0xffffffffu : ((1u << B) - 1u);
    const uint32_t bits = kLike ? (mask[gi] & all) : all;
    const int nb = __popc(bits);
    stage_edges(c, et);
    if (warp == 0 && lane < SPS_NPARAM) s.th[lane] = xk;
    if (warp == 1 && lane < B && ((bits >> lane) & 1u)) {
        const int slot = __popc(bits & ((1u << lane) - 1u));
        const size_t gb = (size_t)gi * B + lane;
        const float* p = g.cssp + gb * K;
        if ((K & 3) == 0) prefetch_l2(p, 4u * K);
        s.ptr[slot] = p;
        s.dust[slot] = g.dust_eff[gb];
        s.zp[slot] = g.zp[gb];
        if (kLike) {
            s.mobs[slot] = mag_obs[gb];
            const float sg = sigma[gb];
            s.isig2[slot] = 1.0f / (sg * sg);
        }
    }
    const float lnT = g.lnT[gi], lT10 = g.lT10[gi];
    const AgeView v{s.m, s.dm0, s.dm1, s.dm2, s.pi, s.w, s.wb, s.q, s.qb, &s.ps[warp], et.age, et.lgz};
    __syncthreads();
    // ---- age bins of this warp, burst weights, metallicity weights, dust
    const float mu = s.th[5], sig = s.th[6] * (1.0f / 3.0f), isig = 1.0f / sig;
    const float xT = (lT10 - mu) * isig, D = tri_cdf(xT);
    sfh_bins_raw<true>(c, v, g.bins + (size_t)gi * A, lnT, s.th[1], s.th[2], s.th[3], kLike, 32 * warp, 32 * warp + 32);
    __syncwarp();
    const float mi = t < A ? s.m[t] : 0.0f;
    float pi = 0.0f;
    if (t < A) {
        const float x0 = (fminf(et.age[t], lT10) - mu) * isig, x1 = (fminf(et.age[t + 1], lT10) - mu) * isig;
        pi = (tri_cdf(x1) - tri_cdf(x0)) * (1.0f / D);
        s.pi[t] = pi;
    }
    {
        const double p = warp_sum_d((double)mi);
        if (lane == 0) s.Mp[warp] = p;
    }
    if (warp == kFewWarps - 1) met_weights(c, v, s.th[7], s.th[8]);
    if (t < nb) {
        const float4 dc = s.dust[t];
        s.F[t] = dust_eval(dc.x, dc.y, dc.z, s.th[9], s.th[10], s.th[11]).F;
        if (kLike) {
            // A = zp - m_obs - 2.5 (lgM + 9) as an FP32 hi + lo pair
            const double Aoff = s.zp[t] - (double)s.mobs[t] - 2.5 * ((double)s.th[0] + 9.0);
            const float ah = (float)Aoff;
            s.Ah[t] = ah;
            s.Al[t] = (float)(Aoff - (double)ah);
        }
    }
    __syncthreads();
    const double M = (s.Mp[0] + s.Mp[1]) + (s.Mp[2] + s.Mp[3]);
    const float Mf = (float)M, fb = s.th[4];
    if (t < A) s.w[t] = (1.0f - fb) * mi + fb * pi * Mf;
    __syncthreads();
    // ---- bands: R_i = sum_j q_j C_bij, U_j = sum_i w_i C_bij, S_b = sum_j q_j U_j, and
    //      with g_b = gamma_b / S_b: wbar_i += g_b R_i, qbar_j += g_b U_j (as team_eval)
    constexpr float kL2hi = 0.301025390625f;            // log10(2), 11 bits
    constexpr float kL2lo = 4.6050389811952137e-6f;     // log10(2) - kL2hi
    constexpr int kZ2 = kZnReg / 2;
    float2 qr[kZ2], qbr[kZ2];
    float wl[4], wbl[4];
#pragma unroll
    for (int j = 0; j < kZ2; ++j) {
        qr[j] = make_float2((2 * j < Zn) ? s.q[2 * j] : 0.0f, (2 * j + 1 < Zn) ? s.q[2 * j + 1] : 0.0f);
        qbr[j] = make_float2(0.0f, 0.0f);
    }
#pragma unroll
    for (int tt = 0; tt < 4; ++tt) {
        const int i = lane + 32 * tt;
        wl[tt] = (i < A) ? s.w[i] : 0.0f;
        wbl[tt] = 0.0f;
    }
#pragma unroll 1
    for (int b = warp; b < nb; b += kFewWarps) {
        const float* C = s.ptr[b];
        float2 U[kZ2];
        float R[4];
#pragma unroll
        for (int j = 0; j < kZ2; ++j) U[j] = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int tt = 0; tt < 4; ++tt) {
            const int i = lane + 32 * tt;
            float cs[kZnReg];
#pragma unroll
            for (int j = 0; j < kZnReg; ++j) cs[j] = 0.0f;
            if (i < A) load_row(C + i * Zn, Zn, cs);
            const float2 w2 = make_float2(wl[tt], wl[tt]);
            float2 r2 = make_float2(0.0f, 0.0f);
#pragma unroll
            for (int j = 0; j < kZ2; ++j) {
                const float2 cv = make_float2(cs[2 * j], cs[2 * j + 1]);
                if (kLike) r2 = __ffma2_rn(qr[j], cv, r2);
                U[j] = __ffma2_rn(w2, cv, U[j]);
            }
            R[tt] = r2.x + r2.y;
        }
        float2 a = make_float2(0.0f, 0.0f);
#pragma unroll
        for (int j = 0; j < kZ2; ++j) a = __ffma2_rn(qr[j], U[j], a);
        const float S = warp_sum(a.x + a.y);
        if (!kLike) {
            if (lane == 0) s.S[b] = S;
            continue;
        }
        int e2;
        const float f = frexpf(s.F[b] * S, &e2);
        const float fe = (float)e2;
        const float bh = s.Ah[b] - 2.5f * (fe * kL2hi);
        const float bl = s.Al[b] - 2.5f * (fe * kL2lo);
        const float r = (bh + bl) - 2.5f * log10f(f);
        const float gam = r * s.isig2[b] * 1.0857362047581294f;     // 2.5 / ln 10
        const float gh = __fdividef(gam, S);
        if (lane == 0) {
            s.res[b] = r;
            s.gam[b] = gam;
        }
        const float2 g2 = make_float2(gh, gh);
#pragma unroll
        for (int j = 0; j < kZ2; ++j) qbr[j] = __ffma2_rn(g2, U[j], qbr[j]);
#pragma unroll
        for (int tt = 0; tt < 4; ++tt) wbl[tt] = fmaf(gh, R[tt], wbl[tt]);
    }
    if constexpr (!kLike) {
        __syncthreads();
        if (t < B) {
            const double m = s.zp[t] - 2.5 * (log10_flux(s.F[t] * s.S[t]) + ((double)s.th[0] + 9.0));
            mag_out[row * B + t] = (float)m;
            if (!isfinite(m)) atomicOr(nonfinite, 1);
        }
        return;
    }
#pragma unroll
    for (int tt = 0; tt < 4; ++tt) s.wbp[warp][lane + 32 * tt] = wbl[tt];
#pragma unroll
    for (int j = 0; j < kZ2; ++j) {
        s.red[t][2 * j] = qbr[j].x;
        s.red[t][2 * j + 1] = qbr[j].y;
    }
    __syncthreads();
    // ---- wbar; qbar (threads 0-95: eight per metallicity column); log L and the
    //      dust / lgM gradients (warp 3, one band per lane)
    const float wb = (s.wbp[0][t] + s.wbp[1][t]) + (s.wbp[2][t] + s.wbp[3][t]);
    s.wb[t] = wb;
    if (warp < 3) {
        const int j = t >> 3, l = t & 7;
        float a = 0.0f;
#pragma unroll
        for (int r = 0; r < kFewThreads / 8; ++r) a += s.red[8 * r + l][j];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(kFull, a, o);
        if (l == 0 && j < Zn) s.qb[j] = a;
    } else {
        double ll = 0.0;
        float g0 = 0.f, g1 = 0.f, g2 = 0.f, g3 = 0.f;
        if (lane < nb) {
            const float4 dc = s.dust[lane];
            const DustTerms d = dust_eval(dc.x, dc.y, dc.z, s.th[9], s.th[10], s.th[11]);
            const float r = s.res[lane], gam = s.gam[lane];
            ll = -0.5 * (double)(r * r * s.isig2[lane]);
            const float gF = __fdividef(gam, d.F);
            g0 = gam * kLn10f;
            g1 = gF * d.dF_AV;
            g2 = gF * d.dF_delta;
            g3 = gF * d.dF_floor;
        }
        ll = warp_sum_d(ll);
        g0 = warp_sum(g0);
        g1 = warp_sum(g1);
        g2 = warp_sum(g2);
        g3 = warp_sum(g3);
        if (lane == 0) {
            s.ll = ll;
            s.gd[0] = g0;
            s.gd[1] = g1;
            s.gd[2] = g2;
            s.gd[3] = g3;
        }
    }
    __syncthreads();
    // ---- through the SFH, burst and MDF weights
    float out[SPS_NPARAM];
    if (!few_adjoint(c, v, et, s.th, lT10, Mf, mi, pi, wb, s.sums, out)) return;
    out[0] = s.gd[0];
    out[9] = s.gd[1];
    out[10] = s.gd[2];
    out[11] = s.gd[3];
    float gk = 0.0f;
#pragma unroll
    for (int k = 0; k < SPS_NPARAM; ++k)
        if (lane == k) gk = out[k];
    if (lane == 0) ll_out[row] = (float)s.ll;
    if (grad_out && lane < SPS_NPARAM) grad_out[row * SPS_NPARAM + lane] = gk;
    const bool bad = __any_sync(kFull, !isfinite(gk)) || !isfinite(s.ll);
    if (bad && lane == 0) atomicOr(nonfinite, 1);
}

}  // namespace

// Up to the rows that are resident at once (five blocks per SM): 760 rows take 43
// us a call against 57 in k_like_team (photometry 37 against 41).  Past that it loses
// its lead: 912 rows 64 against 66, 2,432 rows 84 against 72 (timed with 12 us more
// of host work in every call).
int64_t approx_few_rows() { return 5 * kSms; }

cudaError_t launch_like_few(const Consts& c, const Galaxies& g, const float* theta, const int32_t* gal_idx, int64_t n,
                            const float* mag_obs, const float* sigma, const uint32_t* mask, float* ll_out,
                            float* grad_out, int* nonfinite, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_approx_few<true><<<(unsigned)n, kFewThreads, 0, s>>>(c, g, theta, gal_idx, mag_obs, sigma, mask, nullptr, ll_out,
                                                           grad_out, nonfinite);
    return cudaGetLastError();
}
cudaError_t launch_phot_few(const Consts& c, const Galaxies& g, const float* theta, const int32_t* gal_idx, int64_t n,
                            float* mag_out, int* nonfinite, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    k_approx_few<false><<<(unsigned)n, kFewThreads, 0, s>>>(c, g, theta, gal_idx, nullptr, nullptr, nullptr, mag_out,
                                                            nullptr, nullptr, nonfinite);
    return cudaGetLastError();
}

}  // namespace sps
