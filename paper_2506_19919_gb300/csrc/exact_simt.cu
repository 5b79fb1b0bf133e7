// SIMT contractions of the exact path: FP32 operands (the reference precision),
// or the BF16 table without the tensor cores.
//   forward: S[r][n] = sum_k W[r][k] L[k][n], folded in the epilogue with the
//            dust curve and the redshifted band weights into
//            A[r][b][0..3] = sum_n wb S (1, E, E base, E dterm)   (10^-0.4A = E)
//   adjoint: Wbar[r][k] = sum_n v[r][n] L[k][n]
// Both are bound by the FP32 FMA pipe (128 lanes per SM), so what they do is
// cut to what is needed and packed: a tile of rows that are neighbours in
// redshift contracts only the wavelengths inside the hull of its rows' band
// supports (for six bands over 360-970 nm 44% of the production grid), and a
// thread holds an 8 x 8 block of the tile in packed FP32x2 accumulators
// (FFMA2: half the issue slots), fed from a double-buffered shared tile with
// the next k-slice already in registers.  On the 107 x 12 x 5994 grid with six
// bands: forward of 20,011 rows 3.1 ms (44 TFLOP/s on the products inside the
// supports; 26.6 ms for a 64 x 128 scalar tile over the whole grid), of 8,192
// rows 1.23 ms, their adjoint 1.18 ms (12.1 and 6.8 ms).
#include <cuda_bf16.h>

#include <algorithm>

#include "band_tab.cuh"
#include "sps_device.cuh"

namespace sps {

namespace {

constexpr int kBK = 16;            // reduction slice held in shared memory
constexpr int kNT = 256;           // threads per block: 16 x 16

__device__ __forceinline__ float4 ld4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 ld4(const uint16_t* p) {                    // four BF16
    const uint2 v = __ldg(reinterpret_cast<const uint2*>(p));
    return make_float4(__uint_as_float(v.x << 16), __uint_as_float(v.x & 0xffff0000u), __uint_as_float(v.y << 16),
                       __uint_as_float(v.y & 0xffff0000u));
}

template <int BM, int BN>
struct Slice {
    float a[2][kBK][BM + 4];       // A transposed; the pad keeps the transposing stores conflict-free
    float b[2][kBK][BN];
};

// Row (column) of the tile that accumulator i of thread coordinate t holds:
// groups of four, TM / 4 groups BM / 2 apart.
template <int BM, int TM>
__device__ __forceinline__ int tile_at(int t, int i) { return (i >> 2) * (BM / 2) + 4 * t + (i & 3); }

// acc = sum over r in [r0, r1) of A[m0 + .][r] B[r][n0 + .]; r0 and r1 are
// multiples of kBK inside both operands' padding, n0 a multiple of 4.  Rows
// past M repeat the last one, columns past ldb are zero.  Each element is one
// chain of FP32 FMAs in ascending r.
template <int BM, int BN, typename TA, typename TB>
__device__ __forceinline__ void contract(const TA* __restrict__ A, int64_t lda, int64_t m0, int64_t M,
                                         const TB* __restrict__ B, int64_t ldb, int n0, int r0, int r1,
                                         Slice<BM, BN>& sh, float2 (&acc)[BM / 16][BN / 32]) {
    constexpr int TM = BM / 16, TN = BN / 16, QA = BM * 4 / kNT, QB = BN * 4 / kNT, NB4 = BN / 4;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ty = tid >> 4, tx = tid & 15;
#pragma unroll
    for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
    // A: a warp takes 16 rows x 8 of the slice's 16 columns (32-byte pieces), a
    // second pass the other 8; B: passes of kNT / NB4 rows
    static_assert(QA == 1 ? BM == 64 : (QA == 2 && BM == 128), "loader layout");
    constexpr int RB = kNT / NB4;
    const int am = (warp % (BM / 16)) * 16 + (lane & 15);
    const int ak = (warp / (BM / 16)) * 8 + (lane >> 4) * 4;
    const TA* pa = A + (m0 + am < M ? m0 + am : M - 1) * lda + ak + r0;
    const int bk = tid / NB4, bn = 4 * (tid % NB4);
    const bool bin = n0 + bn < ldb;
    const TB* pb = B + (int64_t)(r0 + bk) * ldb + n0 + bn;
    float4 va[QA], vb[QB];
    auto load = [&]() {
#pragma unroll
        for (int q = 0; q < QA; ++q) va[q] = ld4(pa + 8 * q);
#pragma unroll
        for (int q = 0; q < QB; ++q) vb[q] = bin ? ld4(pb + (int64_t)(q * RB) * ldb) : make_float4(0.f, 0.f, 0.f, 0.f);
        pa += kBK;
        pb += kBK * ldb;
    };
    auto store = [&](int s) {
#pragma unroll
        for (int q = 0; q < QA; ++q) {
            sh.a[s][ak + 8 * q + 0][am] = va[q].x;
            sh.a[s][ak + 8 * q + 1][am] = va[q].y;
            sh.a[s][ak + 8 * q + 2][am] = va[q].z;
            sh.a[s][ak + 8 * q + 3][am] = va[q].w;
        }
#pragma unroll
        for (int q = 0; q < QB; ++q) *reinterpret_cast<float4*>(&sh.b[s][bk + q * RB][bn]) = vb[q];
    };
    load();
    store(0);
    __syncthreads();
    int s = 0;
    for (int r = r0; r < r1; r += kBK, s ^= 1) {
        const bool more = r + kBK < r1;
        if (more) load();
#pragma unroll
        for (int k = 0; k < kBK; ++k) {
            float a[TM];
            float2 b[TN / 2];
#pragma unroll
            for (int i = 0; i < TM; i += 4) {
                const float4 v = *reinterpret_cast<const float4*>(&sh.a[s][k][tile_at<BM, TM>(ty, i)]);
                a[i] = v.x; a[i + 1] = v.y; a[i + 2] = v.z; a[i + 3] = v.w;
            }
#pragma unroll
            for (int j = 0; j < TN; j += 4) {
                const float4 v = *reinterpret_cast<const float4*>(&sh.b[s][k][tile_at<BN, TN>(tx, j)]);
                b[j / 2] = make_float2(v.x, v.y);
                b[j / 2 + 1] = make_float2(v.z, v.w);
            }
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                const float2 ai = make_float2(a[i], a[i]);
#pragma unroll
                for (int j = 0; j < TN / 2; ++j) acc[i][j] = __ffma2_rn(ai, b[j], acc[i][j]);
            }
        }
        if (more) store(s ^ 1);
        __syncthreads();
    }
}

// ---------------------------------------------------------------- forward + epilogue
// Block (x, y): BM rows, and part y of gridDim.y of the BN-wide wavelength
// tiles of the rows' hull.  The epilogue folds each tile into A[r][b][4] in
// shared memory (fixed order); part y writes its own slice cJ + y n B 4, which
// the likelihood kernel adds up in order.  KZ also folds the redshift
// derivative of the band weights, wb' = d wb / dz = q_n T'((1+z) l_n), into
// Az[r][b][2] = sum_n wb' S (1, E).  perm: the row at each position of W.
template <int BM, int BN, typename T, bool KZ>
__global__ void __launch_bounds__(kNT, 2)
k_fwd_simt(const __grid_constant__ Consts c, const Grid grid, const Galaxies g, const float* __restrict__ theta,
           const int32_t* __restrict__ gal_idx, const int32_t* __restrict__ perm, int64_t n,
           const T* __restrict__ W, const T* __restrict__ Ltab, float* __restrict__ cJ, float* __restrict__ cJz) {
    constexpr int TM = BM / 16, TN = BN / 16;
    __shared__ __align__(16) Slice<BM, BN> sh;
    __shared__ float4 lc[BN];
    __shared__ float lamt[BN];
    __shared__ float4 rdust[BM];   // A_V/4.05, delta, F_floor, E_b
    __shared__ int blo[kMaxBands], bhi[kMaxBands];     // hull of each band's support over the rows
    extern __shared__ float dyn[];
    const int B = c.n_band;
    float* accsm = dyn;                                              // [BM][B][4]
    int2* sup = reinterpret_cast<int2*>(dyn + BM * B * 4);           // [BM][B]
    float2* ga = reinterpret_cast<float2*>(sup + BM * B);            // [BM][B]
    float* accz = reinterpret_cast<float*>(ga + BM * B);             // KZ: [BM][B][2]
    float* gzf = accz + BM * B * 2;                                  // KZ: [BM][B] 1/sigma or 1/step
    const int64_t m0 = (int64_t)blockIdx.x * BM;
    const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
    if (tid < B) {
        blo[tid] = c.n_lam;
        bhi[tid] = 0;
    }
    for (int e = tid; e < BM * B * 4; e += kNT) accsm[e] = 0.0f;
    if (KZ)
        for (int e = tid; e < BM * B * 2; e += kNT) accz[e] = 0.0f;
    __syncthreads();
    for (int e = tid; e < BM * B; e += kNT) {
        const int r = e / B, b = e - r * B;
        const int64_t pos = m0 + r;
        const int64_t row = pos < n ? (perm ? (int64_t)perm[pos] : pos) : -1;
        const int64_t gi = row >= 0 ? (gal_idx ? (int64_t)gal_idx[row] : row) : -1;
        int2 sp = make_int2(0, 0);
        float2 gg = make_float2(0.f, 0.f);
        if (gi >= 0 && gi < g.n) {
            sp = g.support[gi * B + b];
            gg = g.gauss[gi * B + b];
            if (KZ) gzf[e] = fabsf(gg.y) / (1.0f + g.z[gi]);         // (1+z)/s / (1+z)
            if (sp.x < sp.y) {
                atomicMin(&blo[b], sp.x);
                atomicMax(&bhi[b], sp.y);
            }
        } else if (KZ) {
            gzf[e] = 0.0f;
        }
        sup[e] = sp;
        ga[e] = gg;
    }
    for (int r = tid; r < BM; r += kNT) {
        const int64_t pos = m0 + r;
        float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
        if (pos < n) {
            const float* t = theta + (perm ? (int64_t)perm[pos] : pos) * SPS_NPARAM;
            d = make_float4(t[9] * (1.0f / 4.05f), t[10], t[11], fmaxf(0.85f - 1.9f * t[10], 0.0f));
        }
        rdust[r] = d;
    }
    __syncthreads();
    int lo = c.n_lam, hi = 0;
    for (int b = 0; b < B; ++b) {
        lo = min(lo, blo[b]);
        hi = max(hi, bhi[b]);
    }
    lo &= ~3;                                                        // 16-byte loads of the table
    const int tiles = hi > lo ? (hi - lo + BN - 1) / BN : 0;
    const int t_end = (int)((int64_t)tiles * (blockIdx.y + 1) / gridDim.y);
    const int kr = (c.K + kBK - 1) / kBK * kBK;                      // <= k_pad (zero padded)
    float2 acc[TM][TN / 2];
    for (int t = (int)((int64_t)tiles * blockIdx.y / gridDim.y); t < t_end; ++t) {
        const int n0 = lo + t * BN;
        contract<BM, BN>(W, c.k_pad, m0, n, Ltab, c.lam_pad, n0, 0, kr, sh, acc);
        for (int j = tid; j < BN; j += kNT) {
            const int nn = n0 + j;
            lc[j] = (nn < c.n_lam) ? grid.lamc[nn] : make_float4(0.f, 0.f, 0.f, 0.f);
            lamt[j] = (nn < c.n_lam) ? grid.lam[nn] : 0.0f;
        }
        __syncthreads();
#pragma unroll 1
        for (int b = 0; b < B; ++b) {
            if (blo[b] >= n0 + BN || bhi[b] <= n0) continue;         // block-uniform
            const int kind = c.band_kind[b];
            const float* tabT = grid.band_T + c.tab_off[b];
            const int tabn = c.tab_n[b];
#pragma unroll
            for (int i = 0; i < TM; ++i) {
                float v[4] = {0.f, 0.f, 0.f, 0.f};
                float vz[2] = {0.f, 0.f};
                const int r = tile_at<BM, TM>(ty, i);
                const int2 sp = sup[r * B + b];
                const float2 gg = ga[r * B + b];
                const float4 rd = rdust[r];
                const float fz = KZ ? gzf[r * B + b] : 0.0f;
#pragma unroll
                for (int j = 0; j < TN; ++j) {
                    const int nl = tile_at<BN, TN>(tx, j), nn = n0 + nl;
                    if (nn >= sp.x && nn < sp.y) {
                        const float4 L4 = lc[nl];
                        float wb = L4.x;
                        float wz = 0.0f;
                        if (kind == 1) {
                            const float u = (lamt[nl] - gg.x) * gg.y;
                            wb *= expf_(-0.5f * u * u);
                            if (KZ) wz = -wb * lamt[nl] * u * fz;       // q T' with T' = -u T / s
                        } else if (kind == 2) {
                            const float ut = (lamt[nl] - gg.x) * -gg.y;
                            wb *= tab_T32(tabT, tabn, ut);
                            if (KZ) wz = L4.x * lamt[nl] * tab_dT32(tabT, tabn, ut) * fz;
                        }
                        const float pw = expf_(rd.y * L4.z);
                        const float base = L4.y * pw + rd.w * L4.w;
                        const float E = exp2f(-0.4f * kLog2_10f * rd.x * base);   // as dust_eval's
                        const float dterm = L4.y * pw * L4.z - (rd.w > 0.0f ? 1.9f * L4.w : 0.0f);
                        const float Sn = (j & 1) ? acc[i][j / 2].y : acc[i][j / 2].x;
                        const float S = Sn * wb;
                        const float es = S * E;
                        v[0] += S;
                        v[1] += es;
                        v[2] += es * base;
                        v[3] += es * dterm;
                        if (KZ) {
                            const float Sz = Sn * wz;
                            vz[0] += Sz;
                            vz[1] += Sz * E;
                        }
                    }
                }
#pragma unroll
                for (int o = 8; o > 0; o >>= 1) {
#pragma unroll
                    for (int q = 0; q < 4; ++q) v[q] += __shfl_xor_sync(kFull, v[q], o);
                    if (KZ) {
                        vz[0] += __shfl_xor_sync(kFull, vz[0], o);
                        vz[1] += __shfl_xor_sync(kFull, vz[1], o);
                    }
                }
                if (tx == 0) {
                    float4* o = reinterpret_cast<float4*>(accsm) + r * B + b;
                    const float4 p = *o;
                    *o = make_float4(p.x + v[0], p.y + v[1], p.z + v[2], p.w + v[3]);
                    if (KZ) {
                        accz[(r * B + b) * 2 + 0] += vz[0];
                        accz[(r * B + b) * 2 + 1] += vz[1];
                    }
                }
            }
        }
        __syncthreads();
    }
    __syncthreads();
    float* oJ = cJ + (int64_t)blockIdx.y * n * B * 4;
    for (int e = tid; e < BM * B; e += kNT) {
        const int r = e / B, b = e - r * B;
        const int64_t pos = m0 + r;
        if (pos >= n) continue;
        const int64_t row = perm ? (int64_t)perm[pos] : pos;
        reinterpret_cast<float4*>(oJ)[row * B + b] = reinterpret_cast<const float4*>(accsm)[e];
        if (KZ) {
            float* oz = cJz + ((int64_t)blockIdx.y * n + row) * B * 2 + b * 2;
            oz[0] = accz[e * 2];
            oz[1] = accz[e * 2 + 1];
        }
    }
}

// ---------------------------------------------------------------- adjoint contraction
// Wbar[m][k] = sum_n V[m][n] Lt[n][k] (x 2^{e_i} for the scaled BF16 table), over
// the hull of the rows' supports (v is zero elsewhere).  Block (x, y, z): BM
// rows, BN columns, part z of gridDim.z of the reduction, written to its own
// slice Wbar + z n k_pad.  hull: see row_hull.
template <int BM, int BN, typename TB>
__global__ void __launch_bounds__(kNT, 2)
k_adj_simt(const __grid_constant__ Consts c, const Grid grid, int64_t n, const float* __restrict__ V,
           const TB* __restrict__ Lt, int scaled, const uint32_t* __restrict__ hull, float* __restrict__ Wbar) {
    constexpr int TM = BM / 16, TN = BN / 16;
    __shared__ __align__(16) Slice<BM, BN> sh;
    const int64_t m0 = (int64_t)blockIdx.x * BM;
    const int k0 = blockIdx.y * BN;
    const int2 h = row_hull(c, hull, m0);
    const int r0 = h.x / kBK, nr = (h.y + kBK - 1) / kBK - r0;       // slices of the reduction
    const int s0 = r0 + (int)((int64_t)nr * blockIdx.z / gridDim.z);
    const int s1 = r0 + (int)((int64_t)nr * (blockIdx.z + 1) / gridDim.z);
    float2 acc[TM][TN / 2];
    if (s0 < s1) {
        contract<BM, BN>(V, c.lam_pad, m0, n, Lt, c.k_pad, k0, s0 * kBK, s1 * kBK, sh, acc);
    } else {
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
            for (int j = 0; j < TN / 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
    }
    const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
    float* out = Wbar + (int64_t)blockIdx.z * n * c.k_pad;
#pragma unroll
    for (int i = 0; i < TM; ++i) {
        const int64_t row = m0 + tile_at<BM, TM>(ty, i);
        if (row >= n) continue;
#pragma unroll
        for (int j = 0; j < TN; j += 4) {
            const int k = k0 + tile_at<BN, TN>(tx, j);
            if (k >= c.K) continue;                                  // k_pad is a multiple of 4
            float4 v = make_float4(acc[i][j / 2].x, acc[i][j / 2].y, acc[i][j / 2 + 1].x, acc[i][j / 2 + 1].y);
            if (scaled) {
                const float4 cs = __ldg(reinterpret_cast<const float4*>(grid.col_scale + k));
                v = make_float4(v.x * cs.x, v.y * cs.y, v.z * cs.z, v.w * cs.w);
            }
            *reinterpret_cast<float4*>(out + row * c.k_pad + k) = v;
        }
    }
}

// A 128 x 128 tile per block reads each operand half as often as a 64 x 64 one
// (shared memory feeds 64 FMAs per 16-byte load instead of 32) but leaves SMs
// idle when the rows are few: the small tile where 128-row tiles would give
// under a block per SM even with every split.
bool small_tile(int64_t n, int64_t units_per_row_tile) {
    return (n + 127) / 128 * units_per_row_tile < 2 * kSms;
}

}  // namespace

// Wavelength parts of the forward: enough blocks for about ten waves of two
// blocks per SM, so that the last wave costs little, at most one part per tile
// of half the grid; limited by what the caller's cJ holds (max_split).
int simt_fwd_split(const Consts& c, int64_t n, int max_split) {
    const int tiles = (c.n_lam + 127) / 128;
    const bool small = small_tile(n, tiles / 2 + 1);
    const int64_t mt = small ? (n + 63) / 64 : (n + 127) / 128;
    const int most = small ? 2 * tiles : tiles;
    int64_t s = (20 * kSms + mt - 1) / mt;
    s = std::min<int64_t>(s, std::min(most, 64));
    return (int)std::max<int64_t>(1, std::min<int64_t>(s, max_split));
}
// Reduction parts of the adjoint.
int simt_adj_split(const Consts& c, int64_t n) {
    const int ct = (c.K + 127) / 128;
    const bool small = small_tile(n, ct);
    const int64_t blocks = small ? (n + 63) / 64 * ((c.K + 63) / 64) : (n + 127) / 128 * ct;
    const int64_t s = (12 * kSms + blocks - 1) / blocks;
    return (int)std::max<int64_t>(1, std::min<int64_t>(s, 8));
}

cudaError_t launch_exact_fwd(const Consts& c, const Grid& grid, const Galaxies& g, const float* theta,
                             const int32_t* gal_idx, const int32_t* perm, int64_t n, int bf16, const float* W32,
                             const uint16_t* Wbf, float* cJ, int nsplit, cudaStream_t s, float* cJz) {
    if (n <= 0) return cudaSuccess;
    const bool kz = cJz != nullptr;
    const bool small = small_tile(n, (c.n_lam + 127) / 128 / 2 + 1);
    const int BM = small ? 64 : 128;
    const size_t dyn = (size_t)BM * c.n_band *
                       (4 * sizeof(float) + sizeof(int2) + sizeof(float2) + (kz ? 3 * sizeof(float) : 0));
    const dim3 grd((unsigned)((n + BM - 1) / BM), nsplit);
    auto go = [&](auto kern, const auto* Wp, const auto* Lp) -> cudaError_t {
        const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dyn);
        if (e != cudaSuccess) return e;
        kern<<<grd, kNT, dyn, s>>>(c, grid, g, theta, gal_idx, perm, n, Wp, Lp, cJ, cJz);
        return cudaGetLastError();
    };
    auto shape = [&](const auto* Wp, const auto* Lp) -> cudaError_t {
        using T = std::remove_const_t<std::remove_pointer_t<decltype(Wp)>>;
        if (small) return kz ? go(k_fwd_simt<64, 64, T, true>, Wp, Lp) : go(k_fwd_simt<64, 64, T, false>, Wp, Lp);
        return kz ? go(k_fwd_simt<128, 128, T, true>, Wp, Lp) : go(k_fwd_simt<128, 128, T, false>, Wp, Lp);
    };
    return bf16 ? shape(Wbf, grid.ssp_bf) : shape(W32, grid.ssp);
}

cudaError_t launch_exact_adj(const Consts& c, const Grid& grid, int64_t n, int bf16, const float* V32,
                             const uint32_t* hull, float* Wbar, int nsplit, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const bool small = small_tile(n, (c.K + 127) / 128);
    const int BM = small ? 64 : 128;
    const dim3 grd((unsigned)((n + BM - 1) / BM), (unsigned)((c.K + BM - 1) / BM), nsplit);
    if (bf16) {
        if (small) k_adj_simt<64, 64><<<grd, kNT, 0, s>>>(c, grid, n, V32, grid.ssp_t_bf, 1, hull, Wbar);
        else k_adj_simt<128, 128><<<grd, kNT, 0, s>>>(c, grid, n, V32, grid.ssp_t_bf, 1, hull, Wbar);
    } else {
        if (small) k_adj_simt<64, 64><<<grd, kNT, 0, s>>>(c, grid, n, V32, grid.ssp_t, 0, hull, Wbar);
        else k_adj_simt<128, 128><<<grd, kNT, 0, s>>>(c, grid, n, V32, grid.ssp_t, 0, hull, Wbar);
    }
    return cudaGetLastError();
}

}  // namespace sps
