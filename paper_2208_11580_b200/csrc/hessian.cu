// Layer Hessian H = 2 X X^T (Section 3 of "Optimal Brain Compression": Hessian of each row's least-squares
// problem; identical for all rows; further calibration chunks are accumulated into it).
//
// X is d x n with the calibration axis contiguous, so both GEMM operands are K-major.  Only tiles on or
// below the diagonal are computed (SYRK); the calibration axis is split into slices whose partial sums are
// combined in a fixed order by the finalize kernel, which also applies the factor 2, mirrors the lower
// triangle (exactly symmetric output) and adds to the previous H when accumulating.  Deterministic.
//
// This file holds the FP32 CUDA-core path (OBC_PREC_FP32), the slice/finalize machinery, and the dispatch
// to the tensor-core paths.
#include "gemm_fp32.cuh"

namespace obc {

int hessian_splits(int d, int64_t n) {
    const int T = (d + 127) / 128;
    const int ntiles = T * (T + 1) / 2;
    int64_t s = (444 + ntiles - 1) / ntiles;
    const int64_t by_len = (n + 2047) / 2048;      // short accumulation chains: partial sums are combined in FP32 RN
    if (by_len > s) s = by_len;
    if (s > 32) s = 32;
    if (s * 64 > n) s = n / 64;
    if (s < 1) s = 1;
    return (int)s;
}

// FP32 path: tile and slices.  64 x 64 tiles (four blocks per SM) waste less on the diagonal and on ragged edges;
// 128 x 128 tiles (two blocks per SM) halve the traffic from L2, which matters once the padding no longer does.
// Slices bound the rounding: s chains of n / s products, added in c chains, err by about sqrt(n / s^2 + s / c) roundings of the result
// (64 x 64 tiles add even and odd k apart: 2 s chains; the finalize kernel adds this path's slices in four).  Where that is more
// than one chain of the tensor-core paths' slices would give, more slices are taken: 1024 x 8192 with 8 slices erred by 2.5e-7, with
// 13 by 1.9e-7.
static bool fp32_small_tile(int d) { return d <= 640; }
static int fp32_splits(int d, int64_t n) {
    const int tile = fp32_small_tile(d) ? 64 : 128;
    const int64_t T = (d + tile - 1) / tile, ntiles = T * (T + 1) / 2;
    const int64_t resident = B200_SMS * (tile == 64 ? F32<64>::BLOCKS : F32<128>::BLOCKS);
    int64_t s = resident / ntiles;                                      // one full wave ...
    const int64_t by_len = (n + 2047) / 2048;                           // ... or chains of at most 2048 products
    if (by_len > s) s = (by_len * ntiles + resident - 1) / resident * resident / ntiles;      // (whole waves)
    if (s * 128 > n) s = n / 128;                                       // slices of 128 or more
    if (s < 1) s = 1;
    const double tc = hessian_splits(d, n), chains = (tile == 64 ? 2.0 : 1.0) * s;
    if (n / (chains * chains) + s / 4.0 > n / (tc * tc) + tc) {
        s = (int64_t)(tile == 64 ? (tc + 1) / 2 : tc);
        if (s * ntiles > resident) s = (s * ntiles + resident - 1) / resident * resident / ntiles;
    }
    if (s > 512) s = 512;
    return (int)s;
}

size_t hessian_tc_extra_bytes(int d, int64_t n);

size_t hessian_workspace_bytes(int d, int64_t n) {      // partial sums + what the tensor-core paths add
    const size_t tc = round_up((size_t)hessian_splits(d, n) * d * d * sizeof(float), 256) + hessian_tc_extra_bytes(d, n);
    const size_t fp32 = round_up((size_t)fp32_splits(d, n) * d * d * sizeof(float), 256);
    return tc > fp32 ? tc : fp32;
}

// partial[z][i][j] = sum_{k in slice z} X[i][k] X[j][k]   for tiles with bj <= bi
template <int TILE>
__global__ void __launch_bounds__(F32<TILE>::THREADS, F32<TILE>::BLOCKS) syrk_fp32_kernel(const float* __restrict__ X, int d, int64_t n,
                                                                                            int64_t ldx, int64_t slice, float* __restrict__ partial) {
    extern __shared__ __align__(16) float fsm[];
    int bi = 0, t = blockIdx.x;                            // lower-triangular tile pairs
    while (t > bi) { t -= bi + 1; ++bi; }
    const int bj = t;
    const int64_t kb = (int64_t)blockIdx.y * slice;
    const int64_t ke = kb + slice < n ? kb + slice : n;
    float* P = partial + (size_t)blockIdx.y * d * d;
    f32_tile_product<TILE, true>(fsm, X, ldx, d, bi * TILE, X, ldx, d, bj * TILE, kb, ke, [&](int i, int j, float v) {
        const int gi = bi * TILE + i, gj = bj * TILE + j;
        if (gi < d && gj <= gi) P[(size_t)gi * d + gj] = v;
    });
}

// H[i][j] = H[j][i] = (accumulate ? H[i][j] : 0) + 2 * sum_z partial[z][i][j]     for j <= i
// err (nullable): a non-zero flag from the producing kernel (a bounded wait that expired) turns the whole result
// into NaN; info (nullable) receives 0 or OBC_ERR_TIMEOUT accordingly.
// A block takes a 32 x 32 tile on or below the diagonal; the mirror image goes through shared memory, so that both copies are
// written along rows (column writes of single values took as long as the partial sums of 32 slices).
// CHAINS = 4: every fourth slice in a sum of its own, for the many slices of the FP32 path (512 slices in one chain are 512 more
// roundings of the result; in FP64 the additions took longer than the loads, 64 x 65536 133 -> 567 us).
template <int CHAINS>
__global__ void __launch_bounds__(256) hessian_finalize_kernel(const float* __restrict__ partial, int splits, int d,
                                                               float* __restrict__ H, int ldh, int accumulate,
                                                               const int* __restrict__ err, int32_t* __restrict__ info) {
    __shared__ float tile[32][33];
    const int bi = blockIdx.y, bj = blockIdx.x;
    const bool failed = err && *err != 0;
    if (info && bi == 0 && bj == 0 && threadIdx.x == 0) info[0] = failed ? (int32_t)OBC_ERR_TIMEOUT : 0;
    if (bj > bi) return;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    const int j = bj * 32 + tx;
    float s[CHAINS][4] = {};
    constexpr int AHEAD = CHAINS == 4 ? 8 : 4;            // slices read together: 16 or 32 loads in flight, added in order
    for (int z0 = 0; z0 < splits; z0 += AHEAD) {
        float v[AHEAD][4];
#pragma unroll
        for (int q = 0; q < AHEAD; ++q)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int i = bi * 32 + ty + 8 * r;
                v[q][r] = z0 + q < splits && i < d && j <= i ? __ldcs(partial + (size_t)(z0 + q) * d * d + (size_t)i * d + j) : 0.f;
            }
#pragma unroll
        for (int q = 0; q < AHEAD; ++q)
#pragma unroll
            for (int r = 0; r < 4; ++r) s[q % CHAINS][r] += v[q][r];
    }
    if (CHAINS == 4) {
#pragma unroll
        for (int r = 0; r < 4; ++r) s[0][r] = (s[0][r] + s[1 % CHAINS][r]) + (s[2 % CHAINS][r] + s[3 % CHAINS][r]);
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int i = bi * 32 + ty + 8 * r;
        if (i < d && j <= i) {
            float v = 2.f * s[0][r];
            if (accumulate) v += H[(size_t)i * ldh + j];
            if (failed) v = __int_as_float(0x7fc00000);
            H[(size_t)i * ldh + j] = v;
            s[0][r] = v;
        }
        tile[ty + 8 * r][tx] = s[0][r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < 4; ++r) {                         // (row, column) of the mirror image: j0 + .., i0 + ..
        const int mi = bj * 32 + ty + 8 * r, mj = bi * 32 + tx;
        if (mj < d && mi < mj) H[(size_t)mi * ldh + mj] = tile[tx][ty + 8 * r];
    }
}

template <int CHAINS>
static obc_status finalize_launch(const float* partial, int splits, int d, float* H, int ldh, int accumulate, const int* err,
                                  int32_t* info, cudaStream_t stream) {
    const int T = (d + 31) / 32;
    hessian_finalize_kernel<CHAINS><<<dim3(T, T), 256, 0, stream>>>(partial, splits, d, H, ldh, accumulate, err, info);
    count_launch();
    OBC_CUDA_TRY(cudaGetLastError());
    return OBC_OK;
}

obc_status hessian_finalize_launch(const float* partial, int splits, int d, float* H, int ldh, int accumulate,
                                   const int* err, int32_t* info, cudaStream_t stream) {
    return finalize_launch<1>(partial, splits, d, H, ldh, accumulate, err, info, stream);
}

obc_status hessian_fp32_launch(const float* X, int d, int64_t n, int64_t ldx, float* H, int ldh, int accumulate,
                               int32_t* info, void* ws, cudaStream_t stream) {
    const int splits = fp32_splits(d, n);
    int64_t slice = (n + splits - 1) / splits;
    slice = (slice + 31) / 32 * 32;
    const int tile = fp32_small_tile(d) ? 64 : 128;
    const int T = (d + tile - 1) / tile;
    dim3 grid(T * (T + 1) / 2, splits);
    float* partial = reinterpret_cast<float*>(ws);
    if (tile == 64) {
        OBC_CUDA_TRY(cudaFuncSetAttribute(syrk_fp32_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, F32<64>::SMEM));
        syrk_fp32_kernel<64><<<grid, F32<64>::THREADS, F32<64>::SMEM, stream>>>(X, d, n, ldx, slice, partial);
    } else {
        OBC_CUDA_TRY(cudaFuncSetAttribute(syrk_fp32_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, F32<128>::SMEM));
        syrk_fp32_kernel<128><<<grid, F32<128>::THREADS, F32<128>::SMEM, stream>>>(X, d, n, ldx, slice, partial);
    }
    count_launch();
    OBC_CUDA_TRY(cudaGetLastError());
    return finalize_launch<4>(partial, splits, d, H, ldh, accumulate, nullptr, info, stream);
}

}  // namespace obc
