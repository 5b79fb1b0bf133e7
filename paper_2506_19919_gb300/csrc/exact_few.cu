// The exact path's weights and their adjoint for few rows (separable model): one
// block of four warps per row, a thread per age bin.  With a warp per row
// (k_weights, k_exact_grad_sep) a row's chain is most of the time when the rows do
// not fill the SMs, and each of its steps is latency: here a warp integrates 32 age
// bins, and the gradient loads an age row's slices of Wbar together.
#include "few.cuh"

namespace sps {

namespace {

struct FewWeights {
    float m[kMaxAges], dm0[kMaxAges], dm1[kMaxAges], dm2[kMaxAges], pi[kMaxAges], w[kMaxAges];
    float q[kMaxMets];
    float th[SPS_NPARAM];
    PanelScratch ps[kFewWarps];
    double Mp[kFewWarps];
};

// Block = row; outputs as k_weights<false>.
__global__ void __launch_bounds__(kFewThreads)
k_weights_few(const __grid_constant__ Consts c, const Grid grid, const Galaxies g, const float* __restrict__ theta,
              const int32_t* __restrict__ gal_idx, int bf16, float* __restrict__ W32, uint16_t* __restrict__ Wbf,
              const int32_t* __restrict__ pos_of, float* __restrict__ W32lo, float* __restrict__ keep,
              uint32_t* __restrict__ hull) {
    __shared__ FewWeights s;
    __shared__ EdgeTables et;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int A = c.n_age, Zn = c.n_met;
    const int64_t row = blockIdx.x;
    const int64_t gi = gal_idx ? (int64_t)gal_idx[row] : row;
    const float xk = (lane < SPS_NPARAM) ? theta[row * SPS_NPARAM + lane] : 0.0f;
    const bool in = gi >= 0 && gi < g.n;
    const bool ok = __all_sync(kFull, isfinite(xk)) && in;             // the same in every warp
    const int64_t wr = pos_of ? (int64_t)pos_of[row] : row;
    stage_edges(c, et);
    if (warp == 0 && lane < SPS_NPARAM) s.th[lane] = xk;
    if (warp == 1 && hull && in) {                 // this row's part of its tile's hull (see row_hull)
        const int2 sp = lane < c.n_band ? g.support[gi * c.n_band + lane] : make_int2(0, 0);
        const bool any = sp.x < sp.y;
        const uint32_t below = __reduce_max_sync(kFull, any ? (uint32_t)(c.n_lam - sp.x) : 0u);
        const uint32_t above = __reduce_max_sync(kFull, any ? (uint32_t)sp.y : 0u);
        if (lane == 0) {
            atomicMax(hull + 2 * (wr / kHullRows), below);
            atomicMax(hull + 2 * (wr / kHullRows) + 1, above);
        }
    }
    __syncthreads();
    if (ok) {
        const AgeView v{s.m, s.dm0, s.dm1, s.dm2, s.pi, s.w, nullptr, s.q, nullptr, &s.ps[warp], et.age, et.lgz};
        const float lnT = g.lnT[gi], lT10 = g.lT10[gi], fb = s.th[4];
        const float mu = s.th[5], isig = 1.0f / (s.th[6] * (1.0f / 3.0f));
        const float D = tri_cdf((lT10 - mu) * isig);
        sfh_bins_raw<true>(c, v, g.bins + (size_t)gi * A, lnT, s.th[1], s.th[2], s.th[3], keep != nullptr, 32 * warp,
                           32 * warp + 32);
        __syncwarp();
        const float mi = t < A ? s.m[t] : 0.0f;
        float pi = 0.0f;
        if (t < A) {
            const float x0 = (fminf(et.age[t], lT10) - mu) * isig, x1 = (fminf(et.age[t + 1], lT10) - mu) * isig;
            pi = (tri_cdf(x1) - tri_cdf(x0)) * (1.0f / D);
        }
        const double p = warp_sum_d((double)mi);
        if (lane == 0) s.Mp[warp] = p;
        if (warp == kFewWarps - 1) met_weights(c, v, s.th[7], s.th[8]);
        __syncthreads();
        const double M = (s.Mp[0] + s.Mp[1]) + (s.Mp[2] + s.Mp[3]);
        const float wi = (1.0f - fb) * mi + fb * pi * (float)M;
        if (t < A) s.w[t] = wi;
        if (keep) {                                // a gradient follows: its arrays (see keep_stride)
            float* kr = keep + row * keep_stride(c);
            if (t == 0) *reinterpret_cast<double*>(kr) = M;
            float* ka = kr + 2;
            if (t < A) {
                ka[t] = mi;
                ka[A + t] = s.dm0[t];
                ka[2 * A + t] = s.dm1[t];
                ka[3 * A + t] = s.dm2[t];
                ka[4 * A + t] = pi;
                ka[5 * A + t] = wi;
            }
            if (t < Zn) ka[6 * A + t] = s.q[t];
        }
    } else {
        if (t < A) s.w[t] = __int_as_float(0x7fc00000);
        if (t < Zn) s.q[t] = 1.0f;
    }
    __syncthreads();
    // W_k = w_i q_j, k = i Zn + j, in pairs (k, k + 1) (k_pad is even)
    int k = 2 * t;
    int i = k / Zn, j = k - i * Zn;
    const int di = 2 * kFewThreads / Zn, dj = 2 * kFewThreads - di * Zn;
    for (; k < c.k_pad; k += 2 * kFewThreads) {
        int i1 = i, j1 = j + 1;
        if (j1 == Zn) {
            j1 = 0;
            ++i1;
        }
        float v0 = 0.0f, v1 = 0.0f;
        if (k < c.K) v0 = s.w[i] * s.q[j];
        if (k + 1 < c.K) v1 = s.w[i1] * s.q[j1];
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
}

struct FewGrad {
    float m[kMaxAges], dm0[kMaxAges], dm1[kMaxAges], dm2[kMaxAges], pi[kMaxAges], wb[kMaxAges];
    float qb[kMaxMets];
    float th[SPS_NPARAM];
    float red[kFewThreads][kZnReg + 1];
    float sums[kFewWarps][SPS_NPARAM];
};

// Block = row; inputs and outputs as k_exact_grad_sep.
__global__ void __launch_bounds__(kFewThreads)
k_grad_few(const __grid_constant__ Consts c, const Galaxies g, const float* __restrict__ theta,
           const int32_t* __restrict__ gal_idx, int64_t n, const float* __restrict__ rowinfo,
           const float* __restrict__ Wbar, float* __restrict__ grad_out, const float* __restrict__ rowz,
           const float* __restrict__ keep, const int32_t* __restrict__ pos_of, int nsplit) {
    __shared__ FewGrad s;
    __shared__ EdgeTables et;
    const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
    const int A = c.n_age, Zn = c.n_met;
    const int NG = rowz ? SPS_NPARAM + 1 : SPS_NPARAM;       // with rowz: d/dz last
    const int64_t row = blockIdx.x;
    const int64_t gi = gal_idx ? (int64_t)gal_idx[row] : row;
    const float xk = (lane < SPS_NPARAM) ? theta[row * SPS_NPARAM + lane] : 0.0f;
    if (!(__all_sync(kFull, isfinite(xk)) && gi >= 0 && gi < g.n)) {          // the same in every warp
        if (t < NG) grad_out[row * NG + t] = __int_as_float(0x7fc00000);
        return;
    }
    stage_edges(c, et);
    if (warp == 0 && lane < SPS_NPARAM) s.th[lane] = xk;
    const AgeView v{s.m, s.dm0, s.dm1, s.dm2, s.pi, nullptr, s.wb, nullptr, s.qb, nullptr, et.age, et.lgz};
    const float* kr = keep + row * keep_stride(c);           // the weights kernel's arrays of this row
    const double M = *reinterpret_cast<const double*>(kr);
    const float* ka = kr + 2;
    const float* wr = Wbar + (pos_of ? (int64_t)pos_of[row] : row) * c.k_pad + t * Zn;
    float mi = 0.0f, pi = 0.0f, wb = 0.0f;
    float U[kZnReg];
#pragma unroll
    for (int j = 0; j < kZnReg; ++j) U[j] = 0.0f;
    if (t < A) {
        float x[kZnReg];
        load_row(wr, Zn, x);
#pragma unroll 4
        for (int p = 1; p < nsplit; ++p) {
            float y[kZnReg];
            load_row(wr + (int64_t)p * n * c.k_pad, Zn, y);
#pragma unroll
            for (int j = 0; j < kZnReg; ++j) x[j] += y[j];
        }
        const float wi = ka[5 * A + t];
        mi = ka[t];
        pi = ka[4 * A + t];
        s.m[t] = mi;
        s.pi[t] = pi;
        s.dm0[t] = ka[A + t];
        s.dm1[t] = ka[2 * A + t];
        s.dm2[t] = ka[3 * A + t];
#pragma unroll
        for (int j = 0; j < kZnReg; ++j) {
            const float qj = j < Zn ? __ldg(ka + 6 * A + j) : 0.0f;
            wb = fmaf(x[j], qj, wb);
            U[j] = x[j] * wi;
        }
        s.wb[t] = wb;
    }
#pragma unroll
    for (int j = 0; j < kZnReg; ++j) s.red[t][j] = U[j];
    __syncthreads();
    if (warp < 3) {                                // qbar: eight threads per column
        const int j = t >> 3, l = t & 7;
        float a = 0.0f;
#pragma unroll
        for (int r = 0; r < kFewThreads / 8; ++r) a += s.red[8 * r + l][j];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(kFull, a, o);
        if (l == 0 && j < Zn) s.qb[j] = a;
    }
    __syncthreads();
    float gr[SPS_NPARAM];
    const float lT10 = g.lT10[gi];
    if (!few_adjoint(c, v, et, s.th, lT10, (float)M, mi, pi, wb, s.sums, gr)) return;
    const float4 ri = *reinterpret_cast<const float4*>(rowinfo + row * 4);
    gr[0] = ri.x;
    gr[9] = ri.y;
    gr[10] = ri.z;
    gr[11] = ri.w;
    float gzt = 0.0f;                              // d log L / dz through t_obs (age bins, M, burst clipping)
    if (rowz)
        gzt = rowz[row] + g.dtdz[gi] * tobs_adjoint(c, v, g.bins + (size_t)gi * A, g.lnT[gi], lT10, M, s.th);
    float out = gr[0];
#pragma unroll
    for (int k = 1; k < SPS_NPARAM; ++k)
        if (lane == k) out = gr[k];
    if (lane == SPS_NPARAM) out = gzt;
    if (lane < NG) grad_out[row * NG + lane] = out;
}

}  // namespace

// Up to eight rows per SM: BF16 log L + gradient of six bands, a block / a warp per
// row: 1 row 104 / 125 us a call, 100 rows 115 / 132, 608 rows 127 / 140, 1,216 rows
// 141 / 146; 2,432 rows 189 / 185 (timed before the forward's parts met in shared
// memory; the rows then fill the SMs either way).
int64_t exact_few_rows() { return 8 * kSms; }

cudaError_t launch_weights_few(const Consts& c, const Grid& grid, const Galaxies& g, const float* theta,
                               const int32_t* gal_idx, int64_t n, int bf16, float* W32, uint16_t* Wbf, cudaStream_t s,
                               const int32_t* pos_of, float* W32lo, float* keep, uint32_t* hull) {
    k_weights_few<<<(unsigned)n, kFewThreads, 0, s>>>(c, grid, g, theta, gal_idx, bf16, W32, Wbf, pos_of, W32lo, keep,
                                                      hull);
    return cudaGetLastError();
}
cudaError_t launch_grad_few(const Consts& c, const Galaxies& g, const float* theta, const int32_t* gal_idx, int64_t n,
                            const float* rowinfo, const float* Wbar, float* grad_out, cudaStream_t s,
                            const float* rowz, const float* keep, const int32_t* pos_of, int nsplit) {
    k_grad_few<<<(unsigned)n, kFewThreads, 0, s>>>(c, g, theta, gal_idx, n, rowinfo, Wbar, grad_out, rowz, keep, pos_of,
                                                   nsplit);
    return cudaGetLastError();
}

}  // namespace sps
