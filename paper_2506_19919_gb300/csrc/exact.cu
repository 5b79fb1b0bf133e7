// Exact photometry (Eq. photo_integral_exact) and its adjoint, as a chain of
// kernels over a block of rows:
//   weights : W[r][ij] = w_i q_j (FP32, or BF16 scaled by 2^{e_i})
//   fwd     : S = W L over the wavelength grid, reduced in the epilogue with
//             the dust curve and the redshifted band weights into
//             A[r][b][0..3] = sum_n wb S (1, E, E base, E dterm)   (10^-0.4A = E)
//   like    : magnitudes, log L, gamma_b / c_b, dust and lgM gradients
//   vgen    : v[r][n] = F_att(n) sum_b (gamma_b / c_b) wb(n)
//   adj     : Wbar = v L^T (the second contraction: recomputed, not stored)
//   grad    : Wbar -> d logL / d theta through the SFH, burst and MDF weights
// The contractions are in exact_simt.cu (FP32) and exact_tc.cu (tensor cores).
#include <cuda_bf16.h>

#include "band_tab.cuh"
#include "sps_device.cuh"

namespace sps {

namespace {

// ---------------------------------------------------------------- weights
// W rows of the exact path, one row per warp: SFH, burst and MDF weights, then
// W_k = w_i q_j as FP32, its TF32 halves, or BF16 scaled by 2^{e_i}.  Bound by
// the latency of the quadrature's exponentials and of the row's serial chain:
// what a warp keeps is cut to 5.8 KB of shared memory and 80 registers (24
// warps per SM), the bin edges are staged in shared memory (a lane-indexed read
// of kernel parameters is taken lane by lane), and the warps of a block take
// their rows after one barrier, so that they share the instruction cache.
// 100,000 rows, BF16, with the arrays kept for the gradient: 398 us, 507 with four
// rows per block, 9.6 KB a row and the edges in parameter memory.
constexpr int kRowWarps = 8;           // warps per block of the row kernels
struct WeightsWork {
    float m[kMaxAges], dm0[kMaxAges], dm1[kMaxAges], dm2[kMaxAges], pi[kMaxAges], w[kMaxAges];
    float q[kMaxMets];
    float th[SPS_NPARAM];
    PanelScratch ps;
};
template <bool kNonsep>
__global__ void __launch_bounds__(32 * kRowWarps, 3)
k_weights(const __grid_constant__ Consts c, const Grid grid, const Galaxies g, const float* __restrict__ theta,
          const int32_t* __restrict__ gal_idx, int64_t n, int bf16, float* __restrict__ W32,
          uint16_t* __restrict__ Wbf, const int32_t* __restrict__ pos_of, float* __restrict__ W32lo,
          float* __restrict__ keep, uint32_t* __restrict__ hull) {
    __shared__ WeightsWork work[kRowWarps];
    __shared__ EdgeTables et;
    extern __shared__ float qms[];         // kNonsep: per warp, q_ij of the row [K]
    const int warp = threadIdx.x >> 5, lane = lane_id();
    WeightsWork& s = work[warp];
    float* qm = kNonsep ? qms + warp * (kKTileMax * 32) : nullptr;
    const AgeView view{s.m, s.dm0, s.dm1, s.dm2, s.pi, s.w, nullptr, s.q, nullptr, &s.ps, et.age, et.lgz};
    stage_edges(c, et);
    const int A = c.n_age, Zn = c.n_met;
    const int64_t per_round = (int64_t)gridDim.x * kRowWarps;
    const int64_t rounds = (n + per_round - 1) / per_round;
    for (int64_t rd = 0; rd < rounds; ++rd) {
        __syncthreads();
        const int64_t row = (rd * gridDim.x + blockIdx.x) * kRowWarps + warp;
        if (row >= n) continue;
        const int64_t gi = gal_idx ? (int64_t)gal_idx[row] : row;
        const float xk = (lane < SPS_NPARAM) ? theta[row * SPS_NPARAM + lane] : 0.0f;
        const bool in = gi >= 0 && gi < g.n;
        const bool ok = __all_sync(kFull, isfinite(xk)) && in;
        const int64_t wr = pos_of ? (int64_t)pos_of[row] : row;
        if (hull && in) {                              // this row's part of its tile's hull (see row_hull)
            const int2 sp = lane < c.n_band ? g.support[gi * c.n_band + lane] : make_int2(0, 0);
            const bool any = sp.x < sp.y;
            const uint32_t below = __reduce_max_sync(kFull, any ? (uint32_t)(c.n_lam - sp.x) : 0u);
            const uint32_t above = __reduce_max_sync(kFull, any ? (uint32_t)sp.y : 0u);
            if (lane == 0) {
                atomicMax(hull + 2 * (wr / kHullRows), below);
                atomicMax(hull + 2 * (wr / kHullRows) + 1, above);
            }
        }
        if (lane < SPS_NPARAM) s.th[lane] = xk;
        __syncwarp();
        if (ok) {
            // with keep (a gradient follows): the derivative integrals too, and the
            // arrays the adjoint needs are kept for it
            age_met_parts<true>(c, view, g.bins + (size_t)gi * A, g.lnT[gi], g.lT10[gi], s.th, keep != nullptr);
            __syncwarp();
            const double M = warp_sum_d(mass_partial(c, view));
            age_weights(c, view, s.th, M);
            if (keep) {
                float* kr = keep + row * keep_stride(c);
                if (lane == 0) *reinterpret_cast<double*>(kr) = M;
                float* ka = kr + 2;
                for (int i = lane; i < A; i += 32) {
                    ka[i] = s.m[i];
                    ka[A + i] = s.dm0[i];
                    ka[2 * A + i] = s.dm1[i];
                    ka[3 * A + i] = s.dm2[i];
                    ka[4 * A + i] = s.pi[i];
                    ka[5 * A + i] = s.w[i];
                }
                if (lane < Zn) ka[6 * A + lane] = s.q[lane];
            }
            if (kNonsep) mdf_rows_fill(c, et.lgz, s.th[7], s.th[8], qm);
        } else {
            for (int i = lane; i < A; i += 32) s.w[i] = __int_as_float(0x7fc00000);
            if (lane < Zn) s.q[lane] = 1.0f;
            if (kNonsep)
                for (int k = lane; k < c.K; k += 32) qm[k] = 1.0f;
            __syncwarp();
        }
        // W_k = w_i q_j, k = i Zn + j: a lane writes the pair (k, k + 1) for
        // k = 2 lane + 64 t (k_pad is even), with (i, j) of k kept incrementally
        int k = 2 * lane;
        int i = k / Zn, j = k - i * Zn;
        const int di = 64 / Zn, dj = 64 - di * Zn;
        for (; k < c.k_pad; k += 64) {
            int i1 = i, j1 = j + 1;
            if (j1 == Zn) {
                j1 = 0;
                ++i1;
            }
            float v0 = 0.0f, v1 = 0.0f;
            if (k < c.K) v0 = s.w[i] * (kNonsep ? qm[k] : s.q[j]);
            if (k + 1 < c.K) v1 = s.w[i1] * (kNonsep ? qm[k + 1] : s.q[j1]);
            const int64_t o = wr * c.k_pad + k;
            if (bf16) {
                const float2 sc = *reinterpret_cast<const float2*>(grid.col_scale + k);   // 2^{e_i}, 0 past K
                const float b0 = v0 * sc.x, b1 = v1 * sc.y;
                *reinterpret_cast<uint32_t*>(Wbf + o) = (uint32_t)f_to_bf16(b0) | ((uint32_t)f_to_bf16(b1) << 16);
            } else if (W32lo) {                        // 3xTF32 operand halves
                float h0, l0, h1, l1;
                tf32_split(v0, h0, l0);
                tf32_split(v1, h1, l1);
                *reinterpret_cast<float2*>(W32 + o) = make_float2(h0, h1);
                *reinterpret_cast<float2*>(W32lo + o) = make_float2(l0, l1);
            } else {
                *reinterpret_cast<float2*>(W32 + o) = make_float2(v0, v1);
            }
            i += di;
            j += dj;
            if (j >= Zn) {
                j -= Zn;
                ++i;
            }
        }
        __syncwarp();
    }
}

// ---------------------------------------------------------------- likelihood
// The sum of cJ's nsplit slices -> magnitudes, log L, gbar[r][b] = gamma_b / c_b
// and rowinfo[r] = (dlogL/dlgM, dA_V, ddelta, dF_floor).  One thread per (row,
// band), so that the FP64 magnitudes fill their warps and the slices of few
// rows are read side by side; then one thread per row adds up the bands in
// order.  A block takes kLikeThreads / n_band rows.
constexpr int kLikeThreads = 256;
__global__ void __launch_bounds__(kLikeThreads)
k_exact_like(const __grid_constant__ Consts c, const Galaxies g, const float* __restrict__ theta,
             const int32_t* __restrict__ gal_idx, int64_t n, const float* __restrict__ cJ, int nsplit,
             const float* __restrict__ mag_obs, const float* __restrict__ sigma, const uint32_t* __restrict__ mask,
             float* __restrict__ mag_out, float* __restrict__ ll_out, float* __restrict__ gbar,
             float* __restrict__ rowinfo, int* __restrict__ nonfinite, const float* __restrict__ cJz,
             float* __restrict__ rowz, double* __restrict__ ll64_out) {
    __shared__ double sl[kLikeThreads];
    __shared__ float s0[kLikeThreads], sA[kLikeThreads], sd[kLikeThreads], sf[kLikeThreads], sz[kLikeThreads];
    const int B = c.n_band, R = kLikeThreads / B;
    const int t = threadIdx.x;
    const int64_t r0 = (int64_t)blockIdx.x * R;
    bool bad = false;
    if (t < R * B && r0 + t / B < n) {
        const int64_t row = r0 + t / B;
        const int b = t % B;
        const int64_t gi = gal_idx ? (int64_t)gal_idx[row] : row;
        double ll = 0.0;
        float g0 = 0.f, gAV = 0.f, gdl = 0.f, gff = 0.f, gz = 0.f, gb = 0.0f;
        if (gi < 0 || gi >= g.n) {
            bad = true;
            ll = __longlong_as_double(0x7ff8000000000000ll);
            if (mag_out) mag_out[row * B + b] = __int_as_float(0x7fc00000);
        } else {
            const float4* aj = reinterpret_cast<const float4*>(cJ) + row * B + b;
            float4 a = aj[0];
#pragma unroll 8
            for (int p = 1; p < nsplit; ++p) {
                const float4 v = aj[(int64_t)p * n * B];
                a = make_float4(a.x + v.x, a.y + v.y, a.z + v.z, a.w + v.w);
            }
            const float* th = theta + row * SPS_NPARAM;
            const float lgM = th[0], AV = th[9], ff = th[11];
            const float cprime = ff * a.x + (1.0f - ff) * a.y;
            const double m = g.zp[gi * B + b] - 2.5 * (log10_flux(cprime) + (double)lgM + 9.0);
            bad = !isfinite(m);
            if (mag_out) mag_out[row * B + b] = (float)m;
            if (mask && ((mask[gi] >> b) & 1u)) {
                const double is2 = 1.0 / ((double)sigma[gi * B + b] * (double)sigma[gi * B + b]);
                const double r = m - (double)mag_obs[gi * B + b];
                ll = -0.5 * r * r * is2;
                const float gam = (float)(2.5 * r * is2 / 2.302585092994046);
                gb = gam / cprime;
                g0 = gam * kLn10f;
                gAV = gb * (1.0f - ff) * (-0.4f * kLn10f / 4.05f) * a.z;
                gdl = gb * (1.0f - ff) * (-0.4f * kLn10f) * (AV / 4.05f) * a.w;
                gff = gb * (a.x - a.y);
                if (cJz) {        // explicit d log L / dz (zero point, band weights; weights W fixed)
                    const float2* zj = reinterpret_cast<const float2*>(cJz) + row * B + b;
                    float2 az = zj[0];
                    for (int p = 1; p < nsplit; ++p) {
                        const float2 v = zj[(int64_t)p * n * B];
                        az = make_float2(az.x + v.x, az.y + v.y);
                    }
                    gz = (float)(-r * is2) * g.dzp[gi * B + b] + gb * (ff * az.x + (1.0f - ff) * az.y);
                }
            }
        }
        if (gbar) gbar[row * B + b] = gb;
        sl[t] = ll;
        s0[t] = g0;
        sA[t] = gAV;
        sd[t] = gdl;
        sf[t] = gff;
        sz[t] = gz;
    }
    __syncthreads();
    if (t < R && r0 + t < n) {
        const int64_t row = r0 + t;
        double ll = 0.0;
        float g0 = 0.f, gAV = 0.f, gdl = 0.f, gff = 0.f, gz = 0.f;
        for (int e = t * B; e < (t + 1) * B; ++e) {
            ll += sl[e];
            g0 += s0[e];
            gAV += sA[e];
            gdl += sd[e];
            gff += sf[e];
            gz += sz[e];
        }
        if (rowz) rowz[row] = gz;
        if (ll_out) ll_out[row] = (float)ll;
        if (ll64_out) ll64_out[row] = ll;
        if (rowinfo) *reinterpret_cast<float4*>(rowinfo + row * 4) = make_float4(g0, gAV, gdl, gff);
        bad = bad || (mask && !isfinite(ll));
    }
    if (bad) atomicOr(nonfinite, 1);
}

// ---------------------------------------------------------------- adjoint source
// One block per position of the redshift order (perm): v[n] = F_att(n) q_n /
// lambda_n sum_b gbar_b T_b(n) inside the hull of the position's row tile, which
// is all that the adjoint contraction reads.  Bound by issue slots: a warp takes
// 64 wavelengths, a pair per lane in packed FP32x2, and visits only the bands
// whose support reaches them (one ballot), so that the sum stays in registers,
// without a row buffer, barriers or tail passes per band; the dust factor
// (dust_eval's terms) follows at once and the pair is stored as one word.
// 100,000 rows, six bands, BF16: a log L + gradient call 3.48 ms, 3.86 ms with a
// shared row buffer filled band by band; the constants of a pair side by side
// (lamp) save 52 us more.
__global__ void __launch_bounds__(256)
k_exact_vgen(const __grid_constant__ Consts c, const Grid grid, const Galaxies g,
             const float* __restrict__ theta, const int32_t* __restrict__ gal_idx, int64_t n,
             const float* __restrict__ gbar, float* __restrict__ V, uint16_t* __restrict__ Vbf,
             float* __restrict__ Vlo, const int32_t* __restrict__ perm, const uint32_t* __restrict__ hull) {
    __shared__ float4 par[kMaxBands];       // gbar / kPairScale, -rest centre, inverse width (0 top-hat, < 0 table)
    __shared__ int2 sp[kMaxBands];
    const int64_t pos = blockIdx.x;
    if (pos >= n) return;
    const int64_t row = perm[pos];
    const int2 h = row_hull(c, hull, pos);
    const int B = c.n_band;
    int64_t gi = gal_idx ? (int64_t)gal_idx[row] : row;
    if (gi < 0 || gi >= g.n) gi = 0;          // row already flagged; gbar is zero
    if (threadIdx.x < B) {
        const int b = threadIdx.x;
        const float gb = gbar[row * B + b];
        const float2 ga = g.gauss[gi * B + b];
        const int kind = c.band_kind[b];
        // e^{-u^2 / 2} = 2^{-(u sqrt(log2(e) / 2))^2}
        par[b] = make_float4(gb * (1.0f / kPairScale), -ga.x, kind == 1 ? ga.y * 0.84932180028801904f : kind == 2 ? ga.y : 0.0f, 0.0f);
        const int2 s = g.support[gi * B + b];
        sp[b] = gb == 0.0f ? make_int2(0, 0) : make_int2(s.x, min(s.y, c.n_lam));
    }
    const float* t = theta + row * SPS_NPARAM;
    const float AV = t[9], dl = t[10], ff = t[11];
    // F = F_floor + (1 - F_floor) 2^{cA (k0 e^{delta lnr} + E_b D)}
    const float eb = fmaxf(0.85f - 1.9f * dl, 0.0f);
    const float cA = -0.4f * kLog2_10f * AV * (1.0f / 4.05f);
    const float dlg = dl * 1.4426950408889634f;     // delta log2(e)
    const float2 dl2 = make_float2(dlg, dlg), eb2 = make_float2(eb, eb), cA2 = make_float2(cA, cA);
    const float2 ff2 = make_float2(ff, ff), omf2 = make_float2(1.0f - ff, 1.0f - ff);
    __syncthreads();
    const int lane = lane_id();
    for (int n0 = h.x + 64 * (int)(threadIdx.x >> 5); n0 < h.y; n0 += 64 * 8) {   // h is in multiples of 32
        const int nn = n0 + 2 * lane;
        const int2 s = lane < B ? sp[lane] : make_int2(0, 0);
        uint32_t act = __ballot_sync(kFull, s.x < n0 + 64 && s.y > n0 && s.x < s.y);
        const float4* cp = grid.lamp + 3 * (min(nn, c.lam_pad - 2) >> 1);       // this pair's constants
        const float4 lq = __ldg(cp);                             // lambda, kPairScale q / lambda
        float2 sum = make_float2(0.f, 0.f);
        for (; act; act &= act - 1) {
            const int b = __ffs(act) - 1;
            const float4 p = par[b];
            const int2 sb = sp[b];
            float2 w = make_float2(1.0f, 1.0f);
            if (p.z > 0.0f) {
                const float2 u = __fmul2_rn(__fadd2_rn(make_float2(lq.x, lq.y), make_float2(p.y, p.y)),
                                            make_float2(p.z, p.z));
                const float2 v = __fmul2_rn(u, u);
                w = make_float2(ex2_(-v.x), ex2_(-v.y));
            } else if (p.z < 0.0f) {
                const float* T = grid.band_T + c.tab_off[b];
                w = make_float2(tab_T32(T, c.tab_n[b], (lq.x + p.y) * -p.z), tab_T32(T, c.tab_n[b], (lq.y + p.y) * -p.z));
            }
            if (sb.x > n0 || sb.y < n0 + 64) {                   // an edge of the support in this chunk
                w.x = (nn >= sb.x && nn < sb.y) ? w.x : 0.0f;
                w.y = (nn + 1 >= sb.x && nn + 1 < sb.y) ? w.y : 0.0f;
            }
            sum = __ffma2_rn(make_float2(p.x, p.x), w, sum);
        }
        float2 v = make_float2(0.f, 0.f);
        if (__any_sync(kFull, sum.x != 0.0f || sum.y != 0.0f)) {
            const float4 kl = __ldg(cp + 1);                     // k0, ln(lambda / lambda_V)
            const float2 dr = __ldg(reinterpret_cast<const float2*>(cp + 2));
            const float2 pa = __fmul2_rn(dl2, make_float2(kl.z, kl.w));
            const float2 pw = make_float2(ex2_(pa.x), ex2_(pa.y));
            const float2 base = __ffma2_rn(make_float2(kl.x, kl.y), pw, __fmul2_rn(eb2, dr));
            const float2 ea = __fmul2_rn(cA2, base);
            float2 E;                                            // as dust_eval's
            if (__any_sync(kFull, fminf(ea.x, ea.y) < -126.0f)) E = make_float2(exp2f(ea.x), exp2f(ea.y));
            else E = make_float2(ex2_(ea.x), ex2_(ea.y));
            const float2 F = __ffma2_rn(omf2, E, ff2);
            v = __fmul2_rn(F, __fmul2_rn(make_float2(lq.z, lq.w), sum));
        }
        if (nn >= h.y) continue;                                 // the hull's end is a multiple of 32
        const int64_t o = pos * c.lam_pad + nn;
        if (Vbf) {
            *reinterpret_cast<uint32_t*>(Vbf + o) = (uint32_t)f_to_bf16(v.x) | ((uint32_t)f_to_bf16(v.y) << 16);
        } else if (Vlo) {                                        // 3xTF32 operand halves
            float h0, l0, h1, l1;
            tf32_split(v.x, h0, l0);
            tf32_split(v.y, h1, l1);
            *reinterpret_cast<float2*>(V + o) = make_float2(h0, h1);
            *reinterpret_cast<float2*>(Vlo + o) = make_float2(l0, l1);
        } else {
            *reinterpret_cast<float2*>(V + o) = v;
        }
    }
}

// ---------------------------------------------------------------- gradient assembly
__global__ void __launch_bounds__(32 * kWarpsApprox)
k_exact_grad(const __grid_constant__ Consts c, const Galaxies g, const float* __restrict__ theta,
             const int32_t* __restrict__ gal_idx, int64_t n, const float* __restrict__ rowinfo,
             const float* __restrict__ Wbar, float* __restrict__ grad_out, const float* __restrict__ rowz,
             const float* __restrict__ keep, const int32_t* __restrict__ pos_of, int nsplit) {
    __shared__ RowScratch scratch[kWarpsApprox];
    const int warp = threadIdx.x >> 5, lane = lane_id();
    RowScratch& s = scratch[warp];
    const int A = c.n_age, Zn = c.n_met, K = c.K;
    const int NG = rowz ? SPS_NPARAM + 1 : SPS_NPARAM;       // with rowz: d/dz last
    for (int64_t row = (int64_t)blockIdx.x * kWarpsApprox + warp; row < n;
         row += (int64_t)gridDim.x * kWarpsApprox) {
        const int64_t gi = gal_idx ? (int64_t)gal_idx[row] : row;
        RowParams p;
        load_params(c, theta + row * SPS_NPARAM, false, p);
        if (gi < 0 || gi >= g.n) p.finite = false;
        if (!p.finite) {
            if (lane < NG) grad_out[row * NG + lane] = __int_as_float(0x7fc00000);
            continue;
        }
        double M;
        if (keep) {                                // the weights kernel's arrays of this row
            const float* kr = keep + row * keep_stride(c);
            M = *reinterpret_cast<const double*>(kr);
            const float* ka = kr + 2;
            for (int i = lane; i < A; i += 32) {
                s.m[i] = ka[i];
                s.dm[0][i] = ka[A + i];
                s.dm[1][i] = ka[2 * A + i];
                s.dm[2][i] = ka[3 * A + i];
                s.pi[i] = ka[4 * A + i];
                s.w[i] = ka[5 * A + i];
            }
            if (lane < Zn) s.q[lane] = ka[6 * A + lane];
        } else {
            M = age_met_weights(c, s, g.bins + (size_t)gi * A, g.lnT[gi], g.lT10[gi], p, true);
        }
        const float* wr = Wbar + (pos_of ? (int64_t)pos_of[row] : row) * c.k_pad;
        for (int k = lane; k < K; k += 32) s.u.kbuf[k] = wr[k];
        for (int p = 1; p < nsplit; ++p) {
            const float* wp = wr + (int64_t)p * n * c.k_pad;
#pragma unroll 8
            for (int k = lane; k < K; k += 32) s.u.kbuf[k] += wp[k];
        }
        __syncwarp();
        float gr[SPS_NPARAM];
#pragma unroll
        for (int k = 0; k < SPS_NPARAM; ++k) gr[k] = 0.0f;
        if (c.mdf_age) {
            mdf_rows_adjoint(c, s.view(c), s.u.kbuf, p.th[7], p.th[8], gr);
        } else {
            for (int i = lane; i < A; i += 32) {
                float a = 0.0f;
                for (int j = 0; j < Zn; ++j) a = fmaf(s.u.kbuf[i * Zn + j], s.q[j], a);
                s.wb[i] = a;
            }
            if (lane < Zn) {
                float a = 0.0f;
                for (int i = 0; i < A; ++i) a = fmaf(s.u.kbuf[i * Zn + lane], s.w[i], a);
                s.qb[lane] = a;
            }
            __syncwarp();
        }
        gr[0] = rowinfo[row * 4 + 0];
        gr[9] = rowinfo[row * 4 + 1];
        gr[10] = rowinfo[row * 4 + 2];
        gr[11] = rowinfo[row * 4 + 3];
        age_met_adjoint(c, s, g.lT10[gi], M, p, gr);
        float gzt = 0.0f;          // d log L / dz through t_obs (age bins, M, burst clipping)
        if (rowz)
            gzt = rowz[row] + g.dtdz[gi] * tobs_adjoint(c, s.view(c), g.bins + (size_t)gi * A, g.lnT[gi],
                                                         g.lT10[gi], M, p.th);
        if (lane == 0) {
#pragma unroll
            for (int k = 0; k < SPS_NPARAM; ++k) grad_out[row * NG + k] = gr[k];
            if (rowz) grad_out[row * NG + SPS_NPARAM] = gzt;
        }
        __syncwarp();
    }
}

// k_exact_grad for the separable model with Zn <= kZnReg: lane i takes age rows
// i, i + 32, ... of Wbar in 16-byte loads straight from memory, wbar_i = sum_j
// Wbar_ij q_j and its share of qbar_j = sum_i w_i Wbar_ij in registers, and the
// lanes' shares are added up through shared memory; k_exact_grad stages the row
// in shared memory and sums each qbar_j in one lane over all ages.  Blocks in
// step and edges in shared memory as in k_weights.
// 100,000 rows: 206 us against 317.
struct GradWork {
    float m[kMaxAges], dm0[kMaxAges], dm1[kMaxAges], dm2[kMaxAges], pi[kMaxAges], wb[kMaxAges];
    float qb[kMaxMets];
    float th[SPS_NPARAM];
    float red[32][kZnReg + 1];
};
__global__ void __launch_bounds__(32 * kRowWarps, 4)
k_exact_grad_sep(const __grid_constant__ Consts c, const Galaxies g, const float* __restrict__ theta,
                 const int32_t* __restrict__ gal_idx, int64_t n, const float* __restrict__ rowinfo,
                 const float* __restrict__ Wbar, float* __restrict__ grad_out, const float* __restrict__ rowz,
                 const float* __restrict__ keep, const int32_t* __restrict__ pos_of, int nsplit) {
    __shared__ GradWork work[kRowWarps];
    __shared__ EdgeTables et;
    const int warp = threadIdx.x >> 5, lane = lane_id();
    GradWork& s = work[warp];
    const AgeView view{s.m, s.dm0, s.dm1, s.dm2, s.pi, nullptr, s.wb, nullptr, s.qb, nullptr, et.age, et.lgz};
    stage_edges(c, et);
    const int A = c.n_age, Zn = c.n_met;
    const int NG = rowz ? SPS_NPARAM + 1 : SPS_NPARAM;       // with rowz: d/dz last
    const int64_t per_round = (int64_t)gridDim.x * kRowWarps;
    const int64_t rounds = (n + per_round - 1) / per_round;
    for (int64_t rd = 0; rd < rounds; ++rd) {
        __syncthreads();
        const int64_t row = (rd * gridDim.x + blockIdx.x) * kRowWarps + warp;
        if (row >= n) continue;
        const int64_t gi = gal_idx ? (int64_t)gal_idx[row] : row;
        const float xk = (lane < SPS_NPARAM) ? theta[row * SPS_NPARAM + lane] : 0.0f;
        if (!(__all_sync(kFull, isfinite(xk)) && gi >= 0 && gi < g.n)) {
            if (lane < NG) grad_out[row * NG + lane] = __int_as_float(0x7fc00000);
            continue;
        }
        if (lane < SPS_NPARAM) s.th[lane] = xk;
        const float* kr = keep + row * keep_stride(c);           // the weights kernel's arrays of this row
        const double M = *reinterpret_cast<const double*>(kr);
        const float* ka = kr + 2;
        const float* wr = Wbar + (pos_of ? (int64_t)pos_of[row] : row) * c.k_pad;
        float q[kZnReg], U[kZnReg];
#pragma unroll
        for (int j = 0; j < kZnReg; ++j) {
            q[j] = j < Zn ? __ldg(ka + 6 * A + j) : 0.0f;
            U[j] = 0.0f;
        }
#pragma unroll 2
        for (int i = lane; i < A; i += 32) {
            float v[kZnReg];
            load_row(wr + i * Zn, Zn, v);
            for (int p = 1; p < nsplit; ++p) {
                float x[kZnReg];
                load_row(wr + (int64_t)p * n * c.k_pad + i * Zn, Zn, x);
#pragma unroll
                for (int j = 0; j < kZnReg; ++j) v[j] += x[j];
            }
            const float wi = ka[5 * A + i];
            s.m[i] = ka[i];
            s.dm0[i] = ka[A + i];
            s.dm1[i] = ka[2 * A + i];
            s.dm2[i] = ka[3 * A + i];
            s.pi[i] = ka[4 * A + i];
            float a = 0.0f;
#pragma unroll
            for (int j = 0; j < kZnReg; ++j) {
                a = fmaf(v[j], q[j], a);
                U[j] = fmaf(v[j], wi, U[j]);
            }
            s.wb[i] = a;
        }
#pragma unroll
        for (int j = 0; j < kZnReg; ++j) s.red[lane][j] = U[j];
        __syncwarp();
        {
            const int j = lane & 15, h = lane >> 4;
            float a = 0.0f;
            if (j < kZnReg) {
#pragma unroll 8
                for (int r = 0; r < 16; ++r) a += s.red[16 * h + r][j];
            }
            a += __shfl_down_sync(kFull, a, 16);
            if (lane < Zn) s.qb[lane] = a;
        }
        __syncwarp();
        float gr[SPS_NPARAM];
#pragma unroll
        for (int k = 0; k < SPS_NPARAM; ++k) gr[k] = 0.0f;
        const float4 ri = *reinterpret_cast<const float4*>(rowinfo + row * 4);
        gr[0] = ri.x;
        gr[9] = ri.y;
        gr[10] = ri.z;
        gr[11] = ri.w;
        age_met_adjoint(c, view, g.lT10[gi], M, s.th, gr);
        float gzt = 0.0f;          // d log L / dz through t_obs (age bins, M, burst clipping)
        if (rowz)
            gzt = rowz[row] + g.dtdz[gi] * tobs_adjoint(c, view, g.bins + (size_t)gi * A, g.lnT[gi], g.lT10[gi], M,
                                                         s.th);
        float out = gr[0];
#pragma unroll
        for (int k = 1; k < SPS_NPARAM; ++k)
            if (lane == k) out = gr[k];
        if (lane == SPS_NPARAM) out = gzt;
        if (lane < NG) grad_out[row * NG + lane] = out;
        __syncwarp();
    }
}

// Blocks of a row kernel: persistent, as many as are resident.
template <class K>
cudaError_t row_blocks(K kern, size_t smem, int64_t n, int& blocks) {
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
    if ((e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess) return e;
    if ((e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, 32 * kRowWarps, smem)) != cudaSuccess) return e;
    const int64_t need = (n + kRowWarps - 1) / kRowWarps;
    const int64_t most = (int64_t)(per_sm > 0 ? per_sm : 1) * sms;
    blocks = (int)(need < most ? need : most);
    return cudaSuccess;
}

int blocks_rows(int64_t rows, int per_block) {
    int64_t b = (rows + per_block - 1) / per_block;
    if (b > 152LL * 64) b = 152LL * 64;
    return (int)(b < 1 ? 1 : b);
}

}  // namespace

cudaError_t launch_exact_weights(const Consts& c, const Grid& grid, const Galaxies& g,
                                 const float* theta, const int32_t* gal_idx, int64_t n, int bf16,
                                 float* W32, uint16_t* Wbf, cudaStream_t s, const int32_t* pos_of,
                                 float* W32lo, float* keep, uint32_t* hull) {
    if (n <= 0) return cudaSuccess;
    if (!c.mdf_age && n <= exact_few_rows())
        return launch_weights_few(c, grid, g, theta, gal_idx, n, bf16, W32, Wbf, s, pos_of, W32lo, keep, hull);
    int blocks = 0;
    cudaError_t e;
    if (c.mdf_age) {
        const size_t smem = sizeof(float) * kKTileMax * 32 * kRowWarps;
        e = cudaFuncSetAttribute(k_weights<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess || (e = row_blocks(k_weights<true>, smem, n, blocks)) != cudaSuccess) return e;
        k_weights<true><<<blocks, 32 * kRowWarps, smem, s>>>(c, grid, g, theta, gal_idx, n, bf16, W32, Wbf, pos_of,
                                                             W32lo, keep, hull);
    } else {
        if ((e = row_blocks(k_weights<false>, 0, n, blocks)) != cudaSuccess) return e;
        k_weights<false><<<blocks, 32 * kRowWarps, 0, s>>>(c, grid, g, theta, gal_idx, n, bf16, W32, Wbf, pos_of,
                                                           W32lo, keep, hull);
    }
    return cudaGetLastError();
}

// ---------------------------------------------------------------- redshift order
// Rows bucketed by log(1 + z) of their galaxy (2048 buckets over [0, 2.5]),
// so that the rows of a tile see nearly the same band supports; by row index
// within a bucket, because the tile a row falls into decides where its sums start
// and the same call has to give the same bits.  A stable counting sort: the rows
// in kZSegs segments at most, a bucket histogram of each, the histograms' running
// sums over the segments, and in each segment the warps take their places in turn.
constexpr int kZBuckets = 2048;
constexpr int kZSegs = 128;
constexpr int kZThreads = 1024;
constexpr int kZFew = 1024;            // up to here the order takes one launch and no scratch

// Rows per segment, a multiple of kZThreads.
static int64_t zsort_seg(int64_t n) {
    return (n + (int64_t)kZThreads * kZSegs - 1) / ((int64_t)kZThreads * kZSegs) * kZThreads;
}
// Grows with the rows up to a chunk's 131,072 (24 KB for 1,025, 1 MB), so that a
// chunk's buffer serves the last, shorter one; a megabyte for every call added 100 us
// to the first call of a context.
size_t zsort_scratch(int64_t n) {
    if (n <= kZFew) return 0;
    return (size_t)kZBuckets * (size_t)((n + zsort_seg(n) - 1) / zsort_seg(n) + 1);
}

namespace {
__device__ __forceinline__ int zbucket(const Galaxies& g, const int32_t* gal_idx, int64_t row) {
    const int64_t gi = gal_idx ? (int64_t)gal_idx[row] : row;
    const float z = (gi >= 0 && gi < g.n) ? g.z[gi] : 0.0f;
    const float u = log1pf(fmaxf(z, 0.0f)) * ((float)kZBuckets / 2.5f);
    return (u < (float)(kZBuckets - 1)) ? (int)u : kZBuckets - 1;   // NaN goes last
}
// Histogram of segment blockIdx.x into hist[segment][bucket]; also zeroes the
// `extra` ints at `zero`.
__global__ void __launch_bounds__(kZThreads) k_zcount(const Galaxies g, const int32_t* __restrict__ gal_idx, int64_t n,
                                                      int64_t seg, int32_t* __restrict__ hist,
                                                      int32_t* __restrict__ zero, int64_t extra) {
    __shared__ int32_t h[kZBuckets];
    for (int i = threadIdx.x; i < kZBuckets; i += kZThreads) h[i] = 0;
    __syncthreads();
    const int64_t r0 = (int64_t)blockIdx.x * seg, r1 = min(n, r0 + seg);
    for (int64_t row = r0 + threadIdx.x; row < r1; row += kZThreads) atomicAdd(&h[zbucket(g, gal_idx, row)], 1);
    for (int64_t i = (int64_t)blockIdx.x * kZThreads + threadIdx.x; i < extra; i += (int64_t)gridDim.x * kZThreads)
        zero[i] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < kZBuckets; i += kZThreads) hist[(int64_t)blockIdx.x * kZBuckets + i] = h[i];
}
// One thread per bucket: hist becomes the rows of the bucket in the segments
// before; total[bucket] all of them.
__global__ void __launch_bounds__(64) k_zprefix(int segs, int32_t* __restrict__ hist, int32_t* __restrict__ total) {
    const int b = blockIdx.x * 64 + threadIdx.x;
    int32_t sum = 0;
#pragma unroll 16
    for (int s = 0; s < segs; ++s) {
        const int32_t v = hist[(int64_t)s * kZBuckets + b];
        hist[(int64_t)s * kZBuckets + b] = sum;
        sum += v;
    }
    total[b] = sum;
}
// Rows of segment blockIdx.x to their places.
__global__ void __launch_bounds__(kZThreads) k_zscatter(const Galaxies g, const int32_t* __restrict__ gal_idx, int64_t n,
                                                        int64_t seg, const int32_t* __restrict__ hist,
                                                        const int32_t* __restrict__ total, int32_t* __restrict__ perm,
                                                        int32_t* __restrict__ pos_of) {
    __shared__ int32_t cursor[kZBuckets], part[kZThreads];
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    // exclusive scan of the totals, plus this segment's offset in each bucket
    const int a = total[2 * t], b = total[2 * t + 1];
    part[t] = a + b;
    __syncthreads();
    for (int o = 1; o < kZThreads; o <<= 1) {
        const int v = (t >= o) ? part[t - o] : 0;
        __syncthreads();
        part[t] += v;
        __syncthreads();
    }
    const int base = part[t] - (a + b);
    const int32_t* hs = hist + (int64_t)blockIdx.x * kZBuckets;
    cursor[2 * t] = base + hs[2 * t];
    cursor[2 * t + 1] = base + a + hs[2 * t + 1];
    __syncthreads();
    const int64_t r0 = (int64_t)blockIdx.x * seg, r1 = min(n, r0 + seg);
    for (int64_t c0 = r0; c0 < r1; c0 += kZThreads) {
        const int64_t row = c0 + t;
        const int key = row < r1 ? zbucket(g, gal_idx, row) : -1;
        const uint32_t same = __match_any_sync(kFull, key);
        const int rank = __popc(same & ((1u << lane) - 1u));
        int pos = 0;
        for (int w = 0; w < kZThreads / 32; ++w) {         // the warps in order
            if (w == warp) {
                const int at = key >= 0 ? cursor[key] : 0;
                __syncwarp();
                if (key >= 0 && rank == 0) cursor[key] = at + __popc(same);
                pos = at + rank;
            }
            __syncthreads();
        }
        if (key >= 0) {
            perm[pos] = (int32_t)row;
            pos_of[row] = pos;
        }
    }
}
// The order of few rows in one launch: every row's position is the number of
// rows before it in (z, row), counted against the keys in shared memory.  Also
// zeroes the `extra` ints at `zero`.
__global__ void __launch_bounds__(kZFew) k_zorder_few(const Galaxies g, const int32_t* __restrict__ gal_idx, int n,
                                                      int32_t* __restrict__ perm, int32_t* __restrict__ pos_of,
                                                      int32_t* __restrict__ zero, int extra) {
    __shared__ __align__(16) float key[kZFew];
    const int t = threadIdx.x;
    float z = INFINITY;
    if (t < n) {
        const int64_t gi = gal_idx ? (int64_t)gal_idx[t] : t;
        z = (gi >= 0 && gi < g.n) ? g.z[gi] : 0.0f;
    }
    key[t] = z;
    for (int i = t; i < extra; i += blockDim.x) zero[i] = 0;
    __syncthreads();
    if (t >= n) return;
    int r = 0;
    for (int j = 0; j < n; j += 4) {
        const float4 k = *reinterpret_cast<const float4*>(key + j);
        r += (k.x < z || (k.x == z && j < t)) + (k.y < z || (k.y == z && j + 1 < t)) +
             (k.z < z || (k.z == z && j + 2 < t)) + (k.w < z || (k.w == z && j + 3 < t));
    }
    perm[r] = t;
    pos_of[t] = r;
}
}  // namespace

cudaError_t launch_zsort(const Galaxies& g, const int32_t* gal_idx, int64_t n, int32_t* perm,
                         int32_t* pos_of, int32_t* scratch, cudaStream_t s, int32_t* zero, int64_t extra) {
    if (n <= 0) return cudaSuccess;
    static_assert(kZBuckets == 2 * kZThreads, "scan layout");
    if (n <= kZFew) {          // one launch instead of three
        k_zorder_few<<<1, (unsigned)((n + 31) / 32 * 32), 0, s>>>(g, gal_idx, (int)n, perm, pos_of, zero, (int)extra);
        return cudaGetLastError();
    }
    const int64_t seg = zsort_seg(n);
    const int segs = (int)((n + seg - 1) / seg);
    int32_t* total = scratch + (size_t)kZBuckets * segs;
    k_zcount<<<segs, kZThreads, 0, s>>>(g, gal_idx, n, seg, scratch, zero, extra);
    k_zprefix<<<kZBuckets / 64, 64, 0, s>>>(segs, scratch, total);
    k_zscatter<<<segs, kZThreads, 0, s>>>(g, gal_idx, n, seg, scratch, total, perm, pos_of);
    return cudaGetLastError();
}

cudaError_t launch_exact_like(const Consts& c, const Galaxies& g, const float* theta,
                              const int32_t* gal_idx, int64_t n, const float* cJ, float* rowinfo,
                              const float* mag_obs, const float* sigma, const uint32_t* mask,
                              float* mag_out, float* loglike_out, float* gbar, int* nonfinite,
                              cudaStream_t s, const float* cJz, float* rowz, double* ll64_out, int nsplit) {
    if (n <= 0) return cudaSuccess;
    const int rows = kLikeThreads / c.n_band;
    k_exact_like<<<(unsigned)((n + rows - 1) / rows), kLikeThreads, 0, s>>>(c, g, theta, gal_idx, n, cJ, nsplit, mag_obs,
                                                             sigma, mask, mag_out, loglike_out, gbar,
                                                             rowinfo, nonfinite, cJz, rowz, ll64_out);
    return cudaGetLastError();
}

cudaError_t launch_exact_vgen(const Consts& c, const Grid& grid, const Galaxies& g,
                              const float* theta, const int32_t* gal_idx, int64_t n,
                              const float* gbar, float* V32, uint16_t* Vbf, cudaStream_t s, float* V32lo,
                              const int32_t* perm, const uint32_t* hull) {
    if (n <= 0) return cudaSuccess;
    k_exact_vgen<<<(unsigned)n, 256, 0, s>>>(c, grid, g, theta, gal_idx, n, gbar, V32, Vbf, V32lo, perm, hull);
    return cudaGetLastError();
}

cudaError_t launch_exact_grad(const Consts& c, const Galaxies& g, const float* theta,
                              const int32_t* gal_idx, int64_t n, const float* rowinfo,
                              const float* Wbar, float* grad_out, cudaStream_t s, const float* rowz,
                              const float* keep, const int32_t* pos_of, int nsplit) {
    if (n <= 0) return cudaSuccess;
    if (!c.mdf_age && c.n_met <= kZnReg && keep) {
        if (n <= exact_few_rows())
            return launch_grad_few(c, g, theta, gal_idx, n, rowinfo, Wbar, grad_out, s, rowz, keep, pos_of, nsplit);
        int blocks = 0;
        const cudaError_t e = row_blocks(k_exact_grad_sep, 0, n, blocks);
        if (e != cudaSuccess) return e;
        k_exact_grad_sep<<<blocks, 32 * kRowWarps, 0, s>>>(c, g, theta, gal_idx, n, rowinfo, Wbar, grad_out, rowz, keep,
                                                           pos_of, nsplit);
        return cudaGetLastError();
    }
    k_exact_grad<<<blocks_rows(n, kWarpsApprox), 32 * kWarpsApprox, 0, s>>>(c, g, theta, gal_idx, n,
                                                                            rowinfo, Wbar, grad_out, rowz, keep,
                                                                            pos_of, nsplit);
    return cudaGetLastError();
}

}  // namespace sps
