// Dense refit for sequential compression (appendix "Sequential Quantization with OBQ" of "Optimal Brain
// Compression"): when a layer's inputs X are those of the already compressed model, the dense weights are first
// re-optimised in closed form, W^T = (X X^T)^-1 X Y^T with Y the dense model's outputs, so that they are a
// minimiser again before the layer is compressed.  Two steps, both accumulating like the Hessian:
//     G (+)= Y X^T                       (tensor cores for TF32 / BF16X3, CUDA cores for FP32)
//     W  = 2 G Hinv,  Hinv = inv(2 X X^T + lambda I)   (the dampened inverse the solver uses anyway)
// This file holds the FP32 CUDA-core product C = alpha A B^T used by both steps.
#include "gemm_fp32.cuh"

namespace obc {

// C (M x N, ldc) = alpha * A (M x K, lda) * B^T (B is N x K, ldb) + beta * C; row-major FP32.  A cluster of blocks shares one
// tile, each with a slice of K; the slices are added in order through distributed shared memory (the entry points have no
// workspace for partial sums).
template <int TILE, bool VEC>
__global__ void __launch_bounds__(F32<TILE>::THREADS, F32<TILE>::BLOCKS) sgemm_nt_kernel(int M, int N, int64_t K, int64_t slice, float alpha,
                                                                                         const float* __restrict__ A, int64_t lda,
                                                                                         const float* __restrict__ B, int64_t ldb, float beta,
                                                                                         float* __restrict__ C, int ldc) {
    extern __shared__ __align__(16) float fsm[];
    namespace cg = cooperative_groups;
    cg::cluster_group cluster = cg::this_cluster();
    const int parts = (int)cluster.num_blocks(), part = (int)cluster.block_rank();
    // (clusters are numbered along x alone: the other grid dimensions end at 65535 tiles)
    const int tile = blockIdx.x / parts, rows = (M + TILE - 1) / TILE;
    const int i0 = tile % rows * TILE, j0 = tile / rows * TILE;
    const int64_t kb = (int64_t)part * slice, ke = kb + slice < K ? kb + slice : K;
    static_assert(F32<TILE>::SMEM >= TILE * TILE * 4 || TILE == 64, "the partial tile takes the place of the stages");
    f32_tile_product<TILE, VEC>(fsm, A, lda, M, i0, B, ldb, N, j0, kb, ke, [&](int i, int j, float v) { fsm[i * TILE + j] = v; });
    cluster.sync();
    for (int e = part * F32<TILE>::THREADS + threadIdx.x; e < TILE * TILE; e += parts * F32<TILE>::THREADS) {
        float s = 0.f;
        for (int z = 0; z < parts; ++z) s += cluster.map_shared_rank(fsm, z)[e];
        const int gi = i0 + e / TILE, gj = j0 + e % TILE;
        if (gi < M && gj < N) {
            float* c = C + (size_t)gi * ldc + gj;
            *c = (beta == 0.f ? 0.f : beta * *c) + alpha * s;
        }
    }
    cluster.sync();                                        // no block leaves while its tile is read
}

template <int TILE, bool VEC>
static obc_status sgemm_nt_tiles(int M, int N, int64_t K, float alpha, const float* A, int64_t lda, const float* B, int64_t ldb, float beta,
                                 float* C, int ldc, cudaStream_t stream) {
    const int64_t tiles = (int64_t)((M + TILE - 1) / TILE) * ((N + TILE - 1) / TILE);
    // parts of K: as long as all blocks still fit at once, slices of 256 or more
    int parts = 1;
    while (parts < 8 && tiles * parts * 2 <= B200_SMS * F32<TILE>::BLOCKS && K / (parts * 2) >= 256) parts *= 2;
    int64_t slice = (K + parts - 1) / parts;
    slice = (slice + 31) / 32 * 32;
    auto kernel = sgemm_nt_kernel<TILE, VEC>;
    OBC_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, F32<TILE>::SMEM));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(tiles * parts));
    cfg.blockDim = dim3(F32<TILE>::THREADS);
    cfg.dynamicSmemBytes = F32<TILE>::SMEM;
    cfg.stream = stream;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = parts; attr.val.clusterDim.y = 1; attr.val.clusterDim.z = 1;
    cfg.attrs = &attr; cfg.numAttrs = 1;
    OBC_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, M, N, K, slice, alpha, A, lda, B, ldb, beta, C, ldc));
    count_launch();
    return OBC_OK;
}

obc_status sgemm_nt_launch(int M, int N, int64_t K, float alpha, const float* A, int64_t lda, const float* B, int64_t ldb,
                           float beta, float* C, int ldc, cudaStream_t stream) {
    // the larger tile where it fills the SMs with the help of at most two parts of K
    if ((int64_t)((M + 127) / 128) * ((N + 127) / 128) >= 96)
        return sgemm_nt_tiles<128, false>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, stream);
    if (aligned16(A) && aligned16(B) && lda % 4 == 0 && ldb % 4 == 0)
        return sgemm_nt_tiles<64, true>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, stream);
    return sgemm_nt_tiles<64, false>(M, N, K, alpha, A, lda, B, ldb, beta, C, ldc, stream);
}

}  // namespace obc
