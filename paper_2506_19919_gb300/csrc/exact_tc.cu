// Tensor-core (tcgen05) contractions of the exact path (Eq. photo_integral_exact)
// for sm_103a, FP32 accumulation in TMEM, with either
//   BF16 operands (kind::f16) with per-age-row power-of-two scaling, or
//   FP32 operands as 3xTF32 (kind::tf32): x = x_hi + x_lo with x_hi the TF32
//   rounding of x, and A B ~ A_hi B_hi + A_hi B_lo + A_lo B_hi (the dropped
//   A_lo B_lo term is ~2^-22 relative), which keeps FP32-level accuracy.
//
// Forward: S[r][n] = sum_k W[r][k] L[k][n] for a 128-row tile and wavelength
// tiles of 96 to 256 columns (fwd_shape), with the dust x filter reduction over n
// fused into the epilogue (the SED never reaches HBM).  Adjoint: Wbar[r][k] =
// sum_n v[r][n] L[k][n] for 128 x 224 tiles.
//
// One block per SM: warp 0 issues TMA loads of A and B k-blocks (128-byte rows,
// 128-byte swizzle) into a ring of stages; one lane of warp 1 issues tcgen05.mma
// into one of two TMEM accumulators and commits to mbarriers; the other warps (8 to
// 16 in the forward, 4 in the adjoint) drain the other accumulator with
// tcgen05.ld.  Every
// wait is bounded: a timeout sets the block's abort flag and the global error
// word, the roles unwind, in-flight copies are waited for (bounded) and TMEM
// is released.
#include <algorithm>
#include <cstdlib>

#include "exact_tc.cuh"

namespace sps {

namespace {

// ---------------------------------------------------------------- wait probe
// Exercises the pipeline's bounded wait: warp 0 waits on an mbarrier that
// warp 1 arrives on when `ready`; otherwise nothing completes it, the wait
// gives up after `limit` polls, sets the abort flag and raises error bit 2,
// and the kernel returns normally.
__global__ void __launch_bounds__(64) k_wait_probe(int ready, uint32_t limit, int* err) {
    __shared__ Ctl ctl;
    if (threadIdx.x == 0) {
        tc::mbar_init(&ctl.drain, 1);
        ctl.abort = 0;
        tc::fence_mbar_init();
    }
    __syncthreads();
    if (threadIdx.x == 32 && ready) tc::mbar_arrive(&ctl.drain);
    if (threadIdx.x == 0) wait_or_abort(&ctl.drain, 0u, &ctl, err, limit);
    __syncthreads();
}

// ---------------------------------------------------------------- adjoint
constexpr int kTrPitch = 36;     // floats per row of an epilogue warp's 32 x 32 block: 16-byte rows, no conflicts
template <bool TF>
__global__ void __launch_bounds__(kThreadsTC, 1)
k_adj_tc(const __grid_constant__ TcMaps tm, const __grid_constant__ Consts c, const Grid grid, int64_t n,
         const uint32_t* __restrict__ hull, float* __restrict__ Wbar, int* err, int tpc) {
    extern __shared__ unsigned char smem_raw[];
    constexpr int ST = TF ? 2 : kAdjStages;
    using R = Ring<kAdjBN, ST, TF>;
    Ctl* ctl;
    uint8_t* ring = carve<kAdjBN, ST, TF>(smem_raw, ctl);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // a block takes tpc of the row block's n tiles; the groups of a row block
    // are adjacent in launch order, so they run together and read its V rows
    // from L2 after the first has brought them in
    const int n_tiles_all = (c.K + kAdjBN - 1) / kAdjBN;
    const int groups = (n_tiles_all + tpc - 1) / tpc;
    const int m0 = (int)(blockIdx.x / groups) * kTM;
    const int nt0 = (int)(blockIdx.x % groups) * tpc;
    const int n_tiles = min(tpc, n_tiles_all - nt0);

    // v is zero outside the hull of the rows' supports: the reduction covers its
    // k-blocks only (the grid's last one reads zero fill); 100,000 rows, six bands:
    // 0.64 ms against 1.11 ms over the whole grid (both before the stores below)
    const int2 hr = row_hull(c, hull, m0);
    // and of these the block takes part blockIdx.y of gridDim.y, into its own
    // slice of Wbar
    const int kb_lo = hr.x / R::kBK, n_all = (hr.y + R::kBK - 1) / R::kBK - kb_lo;
    const int kb0 = kb_lo + n_all * (int)blockIdx.y / (int)gridDim.y;
    const int kb1 = kb_lo + n_all * ((int)blockIdx.y + 1) / (int)gridDim.y;
    const bool none = kb0 >= kb1;                          // fewer k-blocks than parts: a slice of zeros
    tc_setup<ST>(ctl, warp);
    if (warp == 0) {
        if (lane == 0 && !none)
            tc_produce<kAdjBN, ST, TF>(ctl, ring, tm.a, tm.b, m0, n_tiles, nt0 * kAdjBN, kb0, kb1, err);
    } else if (warp == 1) {
        if (lane == 0) tc_mma<kAdjBN, ST, TF>(ctl, ring, none ? 0 : n_tiles, kb1 - kb0, err);
    } else {
        const int q = warp & 3;
        for (int nt = 0; nt < n_tiles; ++nt) {
            const int buf = nt & 1;
            const uint32_t use = (uint32_t)(nt >> 1);
            if (!none) {
                if (!warp_wait(&ctl->tfull[buf], use & 1u, ctl, err)) break;
                tc::tc_fence_after();
            }
            // a lane owns one row of the accumulator: 32 columns at a time are turned
            // through shared memory, so that eight lanes store 128 bytes of one row
            // (a lane storing its own row's 16 bytes uses half of each of 32 sectors:
            // the stores, not the products, set the pace; 100,000 rows, BF16, log L +
            // gradient 3.04 ms a call against 3.15)
            float* tr = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(ctl) + 256) + q * (32 * kTrPitch);
            for (int cc = 0; cc < kAdjBN / 32; ++cc) {
                float S[32];
                if (none) {
#pragma unroll
                    for (int j = 0; j < 32; ++j) S[j] = 0.0f;
                } else
                    tc::tmem_ld32(ctl->tmem_base + ((uint32_t)(32 * q) << 16) + (uint32_t)(buf * kAdjBN + cc * 32), S);
#pragma unroll
                for (int j = 0; j < 32; j += 4)
                    *reinterpret_cast<float4*>(tr + lane * kTrPitch + j) = make_float4(S[j], S[j + 1], S[j + 2], S[j + 3]);
                __syncwarp();
                const int k = (nt0 + nt) * kAdjBN + cc * 32 + 4 * (lane & 7);
                if (k < c.K) {                               // k_pad is a multiple of 4
                    float4 cs = make_float4(1.0f, 1.0f, 1.0f, 1.0f);
                    if (!TF) cs = __ldg(reinterpret_cast<const float4*>(grid.col_scale + k));
#pragma unroll
                    for (int r = 0; r < 8; ++r) {
                        const int rl = 4 * r + (lane >> 3);
                        const int64_t row = (int64_t)m0 + 32 * q + rl;
                        const float4 v = *reinterpret_cast<const float4*>(tr + rl * kTrPitch + 4 * (lane & 7));
                        if (row < n)
                            *reinterpret_cast<float4*>(Wbar + ((int64_t)blockIdx.y * n + row) * c.k_pad + k) =
                                make_float4(v.x * cs.x, v.y * cs.y, v.z * cs.z, v.w * cs.w);
                    }
                }
                __syncwarp();
            }
            if (!none) {
                tc::tc_fence_before();
                tc::mbar_arrive(&ctl->tempty[buf]);
            }
        }
    }
    tc_teardown<ST>(ctl, warp);
}

// n tiles per block: 3 keeps the TMEM double buffer busy while the row block's
// 2 blocks share V in L2 (measured 2-7% faster than one block streaming V for
// all 6 tiles); 1 while that leaves SMs without a block.
int adj_tpc(const Consts& c, int64_t n) {
    const int n_tiles_all = (c.K + kAdjBN - 1) / kAdjBN;
    if (const char* v = std::getenv("SPS_ADJ_TPC")) return std::max(1, std::min(std::atoi(v), n_tiles_all));
    const int64_t mt = (n + kTM - 1) / kTM;
    return mt * ((n_tiles_all + 2) / 3) < kSms ? 1 : std::min(3, n_tiles_all);
}

}  // namespace

// Parts of the forward's wavelength tiles: one block per SM runs a row tile, so
// fewer row tiles than SMs leave the rest idle; they get as many parts as fit
// (100 rows, 107 x 12 x 5994 grid, BF16: log L + gradient 197 us against 573 in
// one part).  From one row tile per SM on the parts only add set-ups and slices
// (100,000 rows in 3 parts: 2.04 ms against 1.96).
int tc_fwd_split(const Consts& c, int64_t n, bool tf) {
    const int64_t mt = (n + kTM - 1) / kTM;
    const int bn = tc_fwd_columns(c, tf);
    const int most = std::min(24, (c.n_lam + bn - 1) / bn);
    return (int)std::max<int64_t>(1, std::min<int64_t>(kSms / mt, most));
}
// Parts of the adjoint's reduction: few row tiles only (each part writes a
// slice of Wbar that the gradient kernel reads back).
int tc_adj_split(const Consts& c, int64_t n) {
    const int n_tiles_all = (c.K + kAdjBN - 1) / kAdjBN, tpc = adj_tpc(c, n);
    const int64_t blocks = (n + kTM - 1) / kTM * ((n_tiles_all + tpc - 1) / tpc);
    return (int)std::max<int64_t>(1, std::min<int64_t>(kSms / blocks, 8));
}

int tc_fwd_columns(const Consts& c, bool tf) { return fwd_shape(c.n_band, tf).bn; }
size_t tc_adj_smem(bool tf) {
    return (tf ? Ring<kAdjBN, 2, true>::kBytes : Ring<kAdjBN, kAdjStages, false>::kBytes) + 256 +
           4 * 32 * kTrPitch * sizeof(float) + 1024;
}

cudaError_t launch_fwd_tc(const TcMaps& tm, bool tf, const Consts& c, const Grid& grid, const Galaxies& g,
                          const float* theta, const int32_t* gal_idx, const int32_t* perm, const uint32_t* hull,
                          int64_t n, float* cJ, int nsplit, int* err, cudaStream_t s, float* cJz) {
    if (cJz) return launch_fwd_tc_z(tm, tf, c, grid, g, theta, gal_idx, perm, hull, n, cJ, nsplit, err, s, cJz);
    return fwd_tc_launch<false>(tm, tf, c, grid, g, theta, gal_idx, perm, hull, n, cJ, nsplit, err, s, nullptr);
}

cudaError_t launch_adj_tc(const TcMaps& tm, bool tf, const Consts& c, const Grid& grid, int64_t n,
                          const uint32_t* hull, float* Wbar, int nsplit, int* err, cudaStream_t s) {
    if (n <= 0) return cudaSuccess;
    const int n_tiles_all = (c.K + kAdjBN - 1) / kAdjBN;
    const int tpc = adj_tpc(c, n);
    const int groups = (n_tiles_all + tpc - 1) / tpc;
    const dim3 blocks((unsigned)(((n + kTM - 1) / kTM) * groups), nsplit);
    const size_t smem = tc_adj_smem(tf);
    cudaError_t e;
    if (tf) {
        e = cudaFuncSetAttribute(k_adj_tc<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_adj_tc<true><<<blocks, kThreadsTC, smem, s>>>(tm, c, grid, n, hull, Wbar, err, tpc);
    } else {
        e = cudaFuncSetAttribute(k_adj_tc<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
        k_adj_tc<false><<<blocks, kThreadsTC, smem, s>>>(tm, c, grid, n, hull, Wbar, err, tpc);
    }
    return cudaGetLastError();
}

cudaError_t launch_wait_probe(int ready, uint32_t limit, int* err, cudaStream_t s) {
    k_wait_probe<<<1, 64, 0, s>>>(ready, limit, err);
    return cudaGetLastError();
}

}  // namespace sps
