// Per-galaxy preparation (once per galaxy set, FP64 or double-float) and the per-galaxy
// c_SSP table of the approximate path (the c_SSP definition of Sec. 3).
#include <cuda_runtime.h>
#include <math.h>

#include "band_tab.cuh"
#include "df.cuh"
#include "sps_internal.h"

namespace sps {

namespace {

constexpr double kMpcCm = 3.0856775814913673e24;
constexpr double kMpcKm = 3.0856775814913673e19;
constexpr double kGyrS = 3.15576e16;
constexpr double kCkms = 299792.458;
constexpr double kLsun = 3.828e33;
constexpr double kAbZp = 3631e-23;
constexpr double kFwhmToSigma = 0.42466090014400953;  // 1 / (2 sqrt(2 ln 2))
constexpr int64_t kPrepChunk = 32768;                 // galaxies per pass of the set-up (bounds its scratch)
constexpr int64_t kCsspDense = 320;

// Calzetti et al. (2000) k'(lambda), R_V = 4.05, clamped at zero; Drude bump
// of unit amplitude at 0.2175 um with width 0.035 um (App. A.3).
__device__ double calzetti_k0(double lum) {
    double k = (lum < 0.63)
                   ? 2.659 * (-2.156 + 1.509 / lum - 0.198 / (lum * lum) + 0.011 / (lum * lum * lum)) + 4.05
                   : 2.659 * (-1.857 + 1.040 / lum) + 4.05;
    return k > 0.0 ? k : 0.0;
}
__device__ double drude_shape(double lum) {
    double x = (lum * 0.035) * (lum * 0.035);
    double d = lum * lum - 0.2175 * 0.2175;
    return x / (d * d + x);
}

// d k0 / d lambda and d D / d lambda [per um] of the two curves above.
__device__ double calzetti_dk0(double lum) {
    if (calzetti_k0(lum) <= 0.0) return 0.0;
    const double i1 = 1.0 / lum, i2 = i1 * i1;
    return (lum < 0.63) ? 2.659 * (-1.509 * i2 + 2.0 * 0.198 * i2 * i1 - 3.0 * 0.011 * i2 * i2)
                        : 2.659 * (-1.040 * i2);
}
__device__ double drude_dshape(double lum) {
    const double x = (lum * 0.035) * (lum * 0.035);
    const double dx = 2.0 * 0.035 * 0.035 * lum;
    const double d = lum * lum - 0.2175 * 0.2175;
    const double dd = 2.0 * lum;
    const double den = d * d + x;
    return (dx * d * d - 2.0 * x * d * dd) / (den * den);
}

// Per-wavelength constants: (q_n / lambda_n, k0, ln(lambda/lambda_V), Drude),
// lambda, q / lambda, q as double-float pairs for the set-up kernels, and the
// constants of neighbouring wavelengths side by side for packed arithmetic
// (lamp, its q / lambda times kPairScale; zero past the grid).
__global__ void k_lambda_consts(const double* __restrict__ lam, int L, int lam_pad, float4* __restrict__ out,
                                float* __restrict__ lam32, float4* __restrict__ lamd, float2* __restrict__ lamdq,
                                float* __restrict__ lamp) {
    int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= lam_pad) return;
    float* pr = lamp + 12 * (n >> 1) + (n & 1);
    if (n >= L) {
        for (int k = 0; k < 12; k += 2) pr[k] = 0.0f;
        return;
    }
    double l = lam[n];
    double q = (n == 0) ? 0.5 * (lam[1] - lam[0])
             : (n == L - 1) ? 0.5 * (lam[L - 1] - lam[L - 2])
                            : 0.5 * (lam[n + 1] - lam[n - 1]);
    double lum = l * 1e-4;
    out[n] = make_float4((float)(q / l), (float)calzetti_k0(lum), (float)log(l / 5500.0),
                         (float)drude_shape(lum));
    lam32[n] = (float)l;
    pr[0] = (float)l;
    pr[2] = kPairScale * (float)(q / l);
    pr[4] = out[n].y;
    pr[6] = out[n].z;
    pr[8] = out[n].w;
    pr[10] = 0.0f;
    const Df ld = df_from(l), rd = df_from(q / l), qd = df_from(q);
    lamd[n] = make_float4(ld.h, ld.l, rd.h, rd.l);
    lamdq[n] = make_float2(qd.h, qd.l);
}

// ---------------------------------------------------------------- per-galaxy set-up
// What it computes is FP64, but sm_103a does two FP64 operations per clock and
// SM, so the work is laid out for that pipe: scalars with one thread per galaxy
// (or galaxy and band), so that every lane of an FP64 instruction counts, and
// the sums over wavelength (the bulk: B bands x the band's support) in
// double-float, one warp per galaxy and band, over the support only.  One
// block per galaxy in FP64 over the whole grid took 15.5 ms for 4,001 galaxies
// x 12 bands x 5,994 wavelengths; the five kernels here take 0.50 ms.
struct GalScalars {
    double T_yr, K0, dlnDL, opz;     // age [yr], (1+z) L_sun / (4 pi d_L^2 3631 Jy), d ln d_L / dz, 1 + z
};

// One thread per galaxy: age of the universe and luminosity distance.  The
// distance integral of 1/E over [0, z] is taken in y = ln(1+x), where the
// nearest singularities are pi/3 off the real axis at any Omega_m: the 32-node
// Gauss-Legendre rule is exact to ~1e-16 for every accepted redshift (< 20).
__global__ void __launch_bounds__(128)
k_gal_scalars(const float* __restrict__ zin, int64_t G, double h0, double om, const double* __restrict__ gl32,
              float* __restrict__ lnT_out, float* __restrict__ lT10_out, float* __restrict__ dtdz,
              GalScalars* __restrict__ scal) {
    const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= G) return;
    const double z = (double)zin[g];
    const double opz = 1.0 + z;
    const double ol = 1.0 - om;
    const double th = kMpcKm / h0 / kGyrS;                    // Hubble time [Gyr]
    // age of a flat matter + Lambda universe (closed form)
    const double t_obs = (2.0 / (3.0 * sqrt(ol))) * th * asinh(sqrt(ol / om) * pow(opz, -1.5));
    const double Y = log1p(z);
    double part = 0.0;
#pragma unroll 1
    for (int k = 0; k < 32; ++k) {
        const double e = exp(0.5 * Y * (1.0 + gl32[k]));
        part += gl32[32 + k] * e / sqrt(om * e * e * e + ol);
    }
    const double dc = 0.5 * Y * part * (kCkms / h0);          // comoving distance [Mpc]
    const double dl_cm = opz * dc * kMpcCm;
    const double T_yr = t_obs * 1e9;
    // redshift derivatives: dt/dz = -1 / ((1+z) H(z)); d ln d_L / dz = 1/(1+z) + (c/H0) / (E d_C)
    const double Ez = sqrt(om * opz * opz * opz + ol);
    lnT_out[g] = (float)log(t_obs);
    lT10_out[g] = (float)log10(T_yr);
    dtdz[g] = (float)(-th / (opz * Ez));
    scal[g] = GalScalars{T_yr, opz * kLsun / (4.0 * M_PI * dl_cm * dl_cm * kAbZp),
                         1.0 / opz + (kCkms / h0) / (Ez * dc), opz};
}

// One thread per (galaxy, age bin): the bin in cosmic time (Eq. smoothPsfh),
// ages [min(E_i,T), min(E_{i+1},T)].
__global__ void __launch_bounds__(256)
k_age_bins(int A, const double* __restrict__ age_edges_yr, int64_t G, const GalScalars* __restrict__ scal,
           float2* __restrict__ bins) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= G * A) return;
    const int64_t g = t / A;
    const int i = (int)(t - g * A);
    const double T_yr = scal[g].T_yr;
    const double e0 = age_edges_yr[i], e1 = age_edges_yr[i + 1];
    float2 b = make_float2(0.f, 0.f);
    if (e0 < T_yr) {
        const double t_hi = (T_yr - e0) * 1e-9;
        if (e1 >= T_yr) {
            b = make_float2((float)log(t_hi), -1.0f);               // reaches t = 0
        } else {
            const double t_lo = (T_yr - e1) * 1e-9;
            const double c0 = 0.5 * (log(t_lo) + log(t_hi));
            const double hw = 0.5 * log1p((e1 - e0) / (T_yr - e1));
            b = make_float2((float)c0, (float)hw);
        }
    }
    bins[t] = b;
}

// Position of a wavelength against a band: -1 below its support, 0 inside, 1 above.
// lo_ is the observed wavelength (1+z) lambda, which grows with the index, so
// the support is one index range.  A Gaussian's is |u| < 6: the rest is 2e-9 of
// the band's weight, below FP32 rounding; zero point and fluxes use the same.
__device__ __forceinline__ int band_side(int kind, double p0, double p1, int tab_n, double lo_) {
    if (kind == 0) return lo_ < p0 ? -1 : (lo_ < p1 ? 0 : 1);
    if (kind == 1) {
        const double u = (lo_ - p0) / (p1 * kFwhmToSigma);
        return u <= -6.0 ? -1 : (u < 6.0 ? 0 : 1);
    }
    const double u = (lo_ - p0) / p1;
    return u < 0.0 ? -1 : (u <= (double)(tab_n - 1) ? 0 : 1);
}

// One thread per (galaxy, band, end): first index not below the support (end
// 0) or above it (end 1).  An FP32 search gives the neighbourhood, the FP64
// test of band_side decides.
__global__ void __launch_bounds__(256)
k_support(const __grid_constant__ Consts c, const Grid grid, const double* __restrict__ band_p0,
          const double* __restrict__ band_p1, int64_t G, const GalScalars* __restrict__ scal,
          int* __restrict__ ends) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t GB = G * c.n_band;
    if (t >= 2 * GB) return;
    const int end = t >= GB ? 1 : 0;
    const int64_t gb = t - end * GB;
    const int b = (int)(gb % c.n_band);
    const double opz = scal[gb / c.n_band].opz;
    const int kind = c.band_kind[b];
    const double p0 = band_p0[b], p1 = band_p1[b];
    double edge = end ? p1 : p0;                                // observed wavelength of the edge
    if (kind == 1) edge = p0 + (end ? 6.0 : -6.0) * (p1 * kFwhmToSigma);
    if (kind == 2) edge = p0 + (end ? p1 * (c.tab_n[b] - 1) : 0.0);
    const float x = (float)(edge / opz);
    int a = 0, e = c.n_lam;                                     // first index with lambda >= x, in FP32
    while (a < e) {
        const int m = (a + e) >> 1;
        if (grid.lam[m] < x) a = m + 1;
        else e = m;
    }
    const int want = end ? 1 : 0;                               // first index whose side is >= want
    while (a > 0 && band_side(kind, p0, p1, c.tab_n[b], opz * grid.lam64[a - 1]) >= want) --a;
    while (a < c.n_lam && band_side(kind, p0, p1, c.tab_n[b], opz * grid.lam64[a]) < want) ++a;
    ends[2 * gb + end] = a;
}

// One warp per (galaxy, band): sums over the support in double-float, with T
// the transmission, q_n the trapezoid weights, d = lambda - p0 / (1+z) and D
// the transmission's derivative up to a factor (T d for a Gaussian, the
// table's slope): sum q T / lambda, q T, q T d, q D, q D d, q D d^2.
constexpr int kBandSums = 6;
__global__ void __launch_bounds__(256)
k_band_sums(const __grid_constant__ Consts c, const Grid grid, const double* __restrict__ band_p0,
            const double* __restrict__ band_p1, int64_t G, const GalScalars* __restrict__ scal,
            const int2* __restrict__ ends, double* __restrict__ sums) {
    __shared__ float2 tab[32];
    if (threadIdx.x < 32) {
        const Df v = df_from(exp2(-(double)threadIdx.x / 32.0));
        tab[threadIdx.x] = make_float2(v.h, v.l);
    }
    __syncthreads();
    const int lane = threadIdx.x & 31;
    const int64_t gb = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
    if (gb >= G * c.n_band) return;
    const int b = (int)(gb % c.n_band);
    const int kind = c.band_kind[b];
    const double opz = scal[gb / c.n_band].opz;
    const Df crest = df_from(band_p0[b] / opz);
    const Df inv = df_from(opz / (kind == 1 ? band_p1[b] * kFwhmToSigma : band_p1[b]));
    const int2 sp = ends[gb];
    Df s[kBandSums];
#pragma unroll
    for (int k = 0; k < kBandSums; ++k) s[k] = Df{0.f, 0.f};
    for (int n = sp.x + lane; n < sp.y; n += 32) {
        const float4 A = __ldg(grid.lamd + n);
        const float2 Q = __ldg(grid.lamdq + n);
        const Df q{Q.x, Q.y}, r{A.z, A.w};
        const Df d = df_sub(Df{A.x, A.y}, crest);
        Df T{1.0f, 0.0f};
        if (kind == 1) {
            const Df u = df_mul(d, inv);
            const Df x = df_mul(u, u);
            T = df_exp_neg(Df{0.5f * x.h, 0.5f * x.l}, tab);
        } else if (kind == 2) {
            Df sl;
            T = tab_Tdf(grid.band_T + c.tab_off[b], grid.band_Tl + c.tab_off[b], c.tab_n[b], df_mul(d, inv), sl);
            const Df qs = df_mul(q, sl), qsd = df_mul(qs, d);
            s[3] = df_add(s[3], qs);
            s[4] = df_add(s[4], qsd);
            s[5] = df_add(s[5], df_mul(qsd, d));
        }
        const Df qT = df_mul(q, T), qTd = df_mul(qT, d);
        s[0] = df_add(s[0], df_mul(r, T));
        s[1] = df_add(s[1], qT);
        s[2] = df_add(s[2], qTd);
        if (kind == 1) {
            const Df m2 = df_mul(qTd, d);
            s[4] = df_add(s[4], m2);
            s[5] = df_add(s[5], df_mul(m2, d));
        }
    }
    if (kind == 1) s[3] = s[2];
#pragma unroll
    for (int k = 0; k < kBandSums; ++k)
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            s[k] = df_add(s[k], Df{__shfl_xor_sync(0xffffffffu, s[k].h, o), __shfl_xor_sync(0xffffffffu, s[k].l, o)});
    if (lane == 0)
#pragma unroll
        for (int k = 0; k < kBandSums; ++k) sums[gb * kBandSums + k] = df_to(s[k]);
}

// One thread per (galaxy, band): zero point, support, rest-frame filter
// parameters, dust constants at lambda_eff and the redshift derivatives.
__global__ void __launch_bounds__(256)
k_band_finish(const __grid_constant__ Consts c, const double* __restrict__ band_p0,
              const double* __restrict__ band_p1, int64_t G, const GalScalars* __restrict__ scal,
              const int2* __restrict__ ends, const double* __restrict__ sums, double* __restrict__ zp,
              int2* __restrict__ support, float2* __restrict__ gauss, float4* __restrict__ dust_eff,
              float* __restrict__ dzp, float4* __restrict__ ddust) {
    const int64_t gb = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (gb >= G * c.n_band) return;
    const int b = (int)(gb % c.n_band);
    const int kind = c.band_kind[b];
    const GalScalars gs = scal[gb / c.n_band];
    const double p0 = band_p0[b], p1 = band_p1[b], opz = gs.opz;
    const double sg = p1 * kFwhmToSigma, crest = p0 / opz;
    const double* s = sums + gb * kBandSums;
    const int2 e = ends[gb];
    const double sN = s[0], sQT = s[1];
    const double sQTL = crest * s[1] + s[2];
    // z derivatives of the three sums over lambda, d T((1+z) l) / dz = l T':
    // T' = -(opz d / s^2) T (Gaussian), slope / step (table), 0 (top-hat)
    const double f = kind == 1 ? -opz / (sg * sg) : kind == 2 ? 1.0 / p1 : 0.0;
    const double sNd = f * s[3];
    const double sQTd = f * (crest * s[3] + s[4]);
    const double sQTLd = f * (crest * (crest * s[3] + 2.0 * s[4]) + s[5]);
    zp[gb] = -2.5 * log10(gs.K0 / sN);
    support[gb] = (e.y > e.x) ? e : make_int2(0, 0);
    // (rest centre, (1+z)/s) of a Gaussian; (rest start, -(1+z)/step) of a table
    gauss[gb] = (kind == 2) ? make_float2((float)crest, (float)(-opz / p1))
                            : make_float2((float)crest, (float)(opz / sg));
    const double le = sQTL / sQT;                           // rest-frame lambda_eff
    const double lum = le * 1e-4;
    dust_eff[gb] = make_float4((float)calzetti_k0(lum), (float)log(le / 5500.0), (float)drude_shape(lum), (float)le);
    // zp = -2.5 log10((1+z) L_sun / (4 pi d_L^2 3631 Jy N_b))
    dzp[gb] = (float)(-2.5 / M_LN10 * (1.0 / opz - 2.0 * gs.dlnDL - sNd / sN));
    const double dle = (sQTLd * sQT - sQTL * sQTd) / (sQT * sQT);   // d lambda_eff / dz
    ddust[gb] = make_float4((float)(calzetti_dk0(lum) * 1e-4 * dle), (float)(dle / le),
                            (float)(drude_dshape(lum) * 1e-4 * dle), 0.0f);
}

// ---------------------------------------------------------------- c_SSP
// c_SSP[g][b][k] = sum_n (q_n/lambda_n) T_b((1+z_g) lambda_n) L[k][n], or its
// redshift derivative: per band a contraction of the galaxies' weights with the
// SSP table.  Bound by the FP32 FMA pipe: a block takes GT galaxies that are
// neighbours in redshift (perm: their supports nearly coincide), one band and
// a tile of columns k, two columns per thread, so that a table value loaded
// once serves GT galaxies, as packed FP32x2 over galaxy pairs.  The weights of
// 64 wavelengths are staged in shared memory (two buffers), the next chunk's
// formed before the current one is consumed.  This runs once per galaxy set
// and keeps its accuracy: the Gaussian argument is formed in double-float, the
// weight uses the accurate expf, and FP32 partial sums of 32 terms are added
// up in double-float (an FP64 addition per 32 FMAs would cost twice the FMAs).
// 4,001 galaxies x 12 bands on the 107 x 12 x 5,994 grid: 3.1 ms (33 TFLOP/s of
// the 97 GFLOP inside the supports), 11.8 ms with one galaxy per block.
constexpr int kCsspChunk = 64;
constexpr int kCsspThreads = 256;       // at most, per block
template <int GT>
__global__ void __launch_bounds__(kCsspThreads, 2)
k_cssp(const __grid_constant__ Consts c, const Grid grid, const Galaxies gal, const int32_t* __restrict__ perm,
       const double* __restrict__ band_p0, const double* __restrict__ band_p1, float* __restrict__ out,
       int deriv) {
    __shared__ __align__(16) float wsh[2][kCsspChunk][GT];
    __shared__ float2 tab[32];
    __shared__ int64_t gidx[GT];
    __shared__ int2 sup[GT];
    __shared__ Df crs[GT], inv[GT];
    __shared__ Df istep;                   // 1 / s of a Gaussian, 1 / step of a table
    const int tid = threadIdx.x, nt = blockDim.x;
    const int b = blockIdx.y;
    const int kind = c.band_kind[b];
    if (tid < 32) {
        const Df v = df_from(exp2(-(double)tid / 32.0));
        tab[tid] = make_float2(v.h, v.l);
    }
    if (tid < GT) {
        const int64_t pos = (int64_t)blockIdx.x * GT + tid;
        const int64_t g = pos < gal.n ? (int64_t)perm[pos] : -1;
        gidx[tid] = g;
        sup[tid] = make_int2(0, 0);
        crs[tid] = inv[tid] = Df{0.f, 0.f};
        if (g >= 0) {
            const double opz = 1.0 + (double)gal.z[g];
            sup[tid] = gal.support[(size_t)g * c.n_band + b];
            crs[tid] = df_from(band_p0[b] / opz);
            inv[tid] = df_from(opz / (kind == 1 ? band_p1[b] * kFwhmToSigma : band_p1[b]));
        }
    }
    if (tid == 31) istep = df_from(1.0 / (kind == 1 ? band_p1[b] * kFwhmToSigma : band_p1[b]));
    __syncthreads();
    int lo = c.n_lam, hi = 0;                                   // hull of the tile's supports
#pragma unroll
    for (int j = 0; j < GT; ++j)
        if (sup[j].x < sup[j].y) {
            lo = min(lo, sup[j].x);
            hi = max(hi, sup[j].y);
        }
    // from a multiple of the 32-term partial sums, so that a galaxy's row of the table
    // has the same bits whichever galaxies share its tile (an empty term adds 0; 2%
    // more wavelengths than from the hull's own start, whose loop bounds would vary)
    lo &= ~31;
    auto fill = [&](int n0, float (*w)[GT]) {
        for (int e = tid; e < kCsspChunk * GT; e += nt) {
            const int t = e / GT, j = e % GT, n = n0 + t;
            const int2 sp = sup[j];
            float v = 0.0f;
            if (n >= sp.x && n < sp.y) {
                const float4 A = __ldg(grid.lamd + n);
                const Df d = df_sub(Df{A.x, A.y}, crs[j]);
                const Df u = df_mul(d, inv[j]);
                if (!deriv) {
                    v = A.z;
                    if (kind == 1) {
                        v *= expf(-0.5f * u.h * u.h);
                    } else if (kind == 2) {
                        Df sl;
                        v = df_mul(Df{A.z, A.w}, tab_Tdf(grid.band_T + c.tab_off[b], grid.band_Tl + c.tab_off[b],
                                                         c.tab_n[b], u, sl)).h;
                    }
                } else if (kind != 0) {
                    // d/dz of (q_n / l_n) T((1+z) l_n) = q_n T'((1+z) l_n): zero for a top-hat
                    const float2 Q = __ldg(grid.lamdq + n);
                    Df dT;
                    if (kind == 1) {
                        const Df x = df_mul(u, u);
                        dT = df_mul(Df{-u.h, -u.l}, df_exp_neg(Df{0.5f * x.h, 0.5f * x.l}, tab));
                    } else {
                        tab_Tdf(grid.band_T + c.tab_off[b], grid.band_Tl + c.tab_off[b], c.tab_n[b], u, dT);
                    }
                    v = df_mul(df_mul(Df{Q.x, Q.y}, dT), istep).h;
                }
            }
            w[t][j] = v;
        }
    };
    const int k = 2 * (int)(blockIdx.z * nt + tid);
    const bool live = k < c.k_pad;
    float2 acc0[GT / 2], acc1[GT / 2], low0[GT / 2], low1[GT / 2];   // columns k, k + 1; galaxy pairs
#pragma unroll
    for (int j = 0; j < GT / 2; ++j) acc0[j] = acc1[j] = low0[j] = low1[j] = make_float2(0.f, 0.f);
    // acc + low += p by two-sum, elementwise
    auto add = [](float2& a, float2& l, float2 p) {
        const float2 s = __fadd2_rn(a, p);
        const float2 na = make_float2(-a.x, -a.y);
        const float2 t = __fadd2_rn(s, na);
        const float2 r = __fadd2_rn(s, make_float2(-t.x, -t.y));
        const float2 e = __fadd2_rn(__fadd2_rn(a, make_float2(-r.x, -r.y)), __fadd2_rn(p, make_float2(-t.x, -t.y)));
        a = s;
        l = __fadd2_rn(l, e);
    };
    if (lo < hi) fill(lo, wsh[0]);
    int buf = 0;
    for (int n0 = lo; n0 < hi; n0 += kCsspChunk, buf ^= 1) {
        __syncthreads();
        if (n0 + kCsspChunk < hi) fill(n0 + kCsspChunk, wsh[buf ^ 1]);
        if (live) {
            const float* col = grid.ssp_t + (size_t)n0 * c.k_pad + k;
            const int nn = min(kCsspChunk, hi - n0);
            for (int t0 = 0; t0 < nn; t0 += 32) {
                float2 p0[GT / 2], p1[GT / 2];
#pragma unroll
                for (int j = 0; j < GT / 2; ++j) p0[j] = p1[j] = make_float2(0.f, 0.f);
                const int te = min(t0 + 32, nn);
#pragma unroll 8
                for (int t = t0; t < te; ++t) {
                    const float2 L = __ldg(reinterpret_cast<const float2*>(col + (size_t)t * c.k_pad));
                    const float2 L0 = make_float2(L.x, L.x), L1 = make_float2(L.y, L.y);
                    const float4* wr = reinterpret_cast<const float4*>(wsh[buf][t]);
#pragma unroll
                    for (int j = 0; j < GT / 4; ++j) {
                        const float4 w4 = wr[j];
                        const float2 wa = make_float2(w4.x, w4.y), wb = make_float2(w4.z, w4.w);
                        p0[2 * j] = __ffma2_rn(wa, L0, p0[2 * j]);
                        p1[2 * j] = __ffma2_rn(wa, L1, p1[2 * j]);
                        p0[2 * j + 1] = __ffma2_rn(wb, L0, p0[2 * j + 1]);
                        p1[2 * j + 1] = __ffma2_rn(wb, L1, p1[2 * j + 1]);
                    }
                }
#pragma unroll
                for (int j = 0; j < GT / 2; ++j) {
                    add(acc0[j], low0[j], p0[j]);
                    add(acc1[j], low1[j], p1[j]);
                }
            }
        }
    }
    if (k >= c.K) return;
    auto store = [&](int j, float v0, float v1) {
        if (gidx[j] < 0) return;
        float* o = out + ((size_t)gidx[j] * c.n_band + b) * c.K + k;
        if ((c.K & 1) == 0) {
            *reinterpret_cast<float2*>(o) = make_float2(v0, v1);
        } else {
            o[0] = v0;
            if (k + 1 < c.K) o[1] = v1;
        }
    };
#pragma unroll
    for (int j = 0; j < GT / 2; ++j) {
        store(2 * j, acc0[j].x + low0[j].x, acc1[j].x + low1[j].x);
        store(2 * j + 1, acc0[j].y + low0[j].y, acc1[j].y + low1[j].y);
    }
}

}  // namespace

cudaError_t launch_lambda_consts(const double* lam, int L, int lam_pad, float4* out, float* lam32, float4* lamd,
                                 float2* lamdq, float* lamp, cudaStream_t s) {
    k_lambda_consts<<<(lam_pad + 255) / 256, 256, 0, s>>>(lam, L, lam_pad, out, lam32, lamd, lamdq, lamp);
    return cudaGetLastError();
}

size_t prepare_scratch_bytes(const Consts& c, int64_t n_gal) {
    const size_t m = (size_t)(n_gal < kPrepChunk ? n_gal : kPrepChunk);
    return m * (sizeof(GalScalars) + (size_t)c.n_band * (kBandSums * sizeof(double) + sizeof(int2)));
}

cudaError_t launch_prepare_galaxies(const Consts& c, const Grid& grid, const double* band_p0,
                                    const double* band_p1, const double* age_edges_yr, const double* gl32,
                                    const float* z, int64_t n_gal, double h0, double om, float* lnT, float* lT10,
                                    float2* bins, double* zp, int2* support, float2* gauss, float4* dust_eff,
                                    float* dtdz, float* dzp, float4* ddust, void* scratch, cudaStream_t s) {
    const int B = c.n_band;
    auto blocks = [](int64_t n, int per) { return (unsigned)((n + per - 1) / per); };
    for (int64_t g0 = 0; g0 < n_gal; g0 += kPrepChunk) {
        const int64_t m = n_gal - g0 < kPrepChunk ? n_gal - g0 : kPrepChunk;
        const int64_t mb = m * B, b0 = g0 * B;
        GalScalars* scal = static_cast<GalScalars*>(scratch);
        double* sums = reinterpret_cast<double*>(scal + m);
        int2* ends = reinterpret_cast<int2*>(sums + mb * kBandSums);
        k_gal_scalars<<<blocks(m, 128), 128, 0, s>>>(z + g0, m, h0, om, gl32, lnT + g0, lT10 + g0, dtdz + g0, scal);
        k_age_bins<<<blocks(m * c.n_age, 256), 256, 0, s>>>(c.n_age, age_edges_yr, m, scal, bins + g0 * c.n_age);
        k_support<<<blocks(2 * mb, 256), 256, 0, s>>>(c, grid, band_p0, band_p1, m, scal,
                                                      reinterpret_cast<int*>(ends));
        k_band_sums<<<blocks(mb, 8), 256, 0, s>>>(c, grid, band_p0, band_p1, m, scal, ends, sums);
        k_band_finish<<<blocks(mb, 256), 256, 0, s>>>(c, band_p0, band_p1, m, scal, ends, sums, zp + b0,
                                                      support + b0, gauss + b0, dust_eff + b0, dzp + b0, ddust + b0);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t launch_cssp(const Consts& c, const Grid& grid, const Galaxies& g, const int32_t* perm,
                        const double* band_p0, const double* band_p1, float* cssp, cudaStream_t s, int deriv) {
    if (g.n <= 0) return cudaSuccess;
    // columns per block: the split of K into equal tiles of at most 256 threads
    // x 2 columns that leaves the fewest columns over (1,284: 3 tiles of 224)
    int nt = 0, tiles = 0;
    for (int kt = 1; kt <= 16; ++kt) {
        const int th = ((c.K + 2 * kt - 1) / (2 * kt) + 31) / 32 * 32;
        if (th > kCsspThreads) continue;
        if (nt == 0 || kt * th < tiles * nt) {
            nt = th;
            tiles = kt;
        }
    }
    // 16 galaxies a block where the catalogue is dense enough in redshift that
    // their supports nearly coincide and the grid still fills the SMs; 4 below.
    // Set-up and magnitudes of G galaxies (z to 3, 12 bands), 16 / 4 a block: G = 128
    // 523 / 435 us, 256 577 / 562, 384 681 / 732, 512 805 / 908, 2,048 2,037 / 2,892
    if (g.n >= kCsspDense) {
        const dim3 grd((unsigned)((g.n + 15) / 16), c.n_band, tiles);
        k_cssp<16><<<grd, nt, 0, s>>>(c, grid, g, perm, band_p0, band_p1, cssp, deriv);
    } else {
        const dim3 grd((unsigned)((g.n + 3) / 4), c.n_band, tiles);
        k_cssp<4><<<grd, nt, 0, s>>>(c, grid, g, perm, band_p0, band_p1, cssp, deriv);
    }
    return cudaGetLastError();
}

}  // namespace sps
