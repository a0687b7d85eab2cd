// FP32 CUDA-core product A B^T of two row-major operands with the contraction along their rows: the Hessian's FP32 path
// (lower tile pairs of one matrix, partial sums per slice of the contraction) and the FP32 products of the dense refit.
//
// Bound by the FMA pipe (FP32 FMAs from registers reach 53 TFLOP/s on this part).  Two tiles:
//   128 x 128, 256 threads with 8 x 8 outputs: four 128-bit shared-memory loads feed 32 packed FMAs (fma.f32x2 on pairs of
//     columns).  A stage is 16 k deep and k-major, so that a thread's operands are contiguous; cp.async copies single values
//     into place, groups of four rows are permuted by k so that the copies meet few bank conflicts.  3072 x 65536 (SYRK): 15.0 ->
//     13.5 ms (46 TFLOP/s) against synchronous staging.
//   64 x 64, 128 threads with 8 x 4 outputs: less padding for short matrices and four times the blocks.  Rows are kept as they
//     are in memory (16-byte cp.async, 32 k per stage, rows padded to 36 floats so that the 8 rows a warp reads at once fall on
//     different banks) and the packed FMAs take even and odd k: single-value copies would cost a third of the time here
//     (147 x 50173: 134 us against 101 us; 202 us with 128 x 128 tiles and synchronous staging).
#pragma once
#include "common.cuh"
#include <cooperative_groups.h>

namespace obc {

template <int TILE> struct F32 {
    static constexpr int THREADS = TILE == 128 ? 256 : 128;
    static constexpr int BLOCKS = TILE == 128 ? 2 : 4;                         // per SM
    static constexpr int K = TILE == 128 ? 16 : 32;                            // k per stage
    static constexpr int STAGES = TILE == 128 ? 4 : 3;
    static constexpr int STAGE_FLOATS = TILE == 128 ? 2 * 128 * 16 : 2 * 64 * 36;
    static constexpr int SMEM = STAGES * STAGE_FLOATS * 4;
};

// emit(i, j, s) for this thread's elements of the tile: s = sum over k in [kb, ke) of A[i0 + i][k] B[j0 + j][k]; rows past rows_a /
// rows_b read as 0.  VEC: rows start on 16-byte boundaries (64 x 64 tiles only; else 4-byte copies).
template <int TILE, bool VEC, typename Emit>
__device__ __forceinline__ void f32_tile_product(float* smem, const float* __restrict__ A, int64_t lda, int rows_a, int i0,
                                                 const float* __restrict__ B, int64_t ldb, int rows_b, int j0, int64_t kb, int64_t ke, Emit emit) {
    using C = F32<TILE>;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t sbase = (uint32_t)__cvta_generic_to_shared(smem);
    const int steps = ke > kb ? (int)((ke - kb + C::K - 1) / C::K) : 0;
    // a warp covers 4 x 8 threads of the thread grid
    const int ty = (warp % 2) * 4 + (lane >> 3) + (TILE == 128 ? ((warp >> 1) % 2) * 8 : 0);
    const int tx = (TILE == 128 ? warp >> 2 : warp >> 1) * 8 + (lane & 7);

    auto stage_copy = [&](int s, int64_t k0) {
        if (TILE == 128) {
            const int ck = tid % 16, crow = tid / 16;
            const uint32_t base = sbase + (uint32_t)(s * C::STAGE_FLOATS + ck * 128) * 4;
            const bool kin = k0 + ck < ke;
#pragma unroll
            for (int c = 0; c < 16; ++c) {
                const bool second = c >= 8;
                const int r = crow + 16 * (c & 7);
                const int gi = (second ? j0 : i0) + r;
                const bool in = kin && gi < (second ? rows_b : rows_a);
                const float* src = second ? B + (int64_t)gi * ldb : A + (int64_t)gi * lda;
                const uint32_t dst = base + (uint32_t)((second ? 128 * 16 : 0) + ((((r >> 2) ^ (ck & 7)) << 2) | (r & 3))) * 4;
                asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(in ? src + k0 + ck : A), "r"(in ? 4 : 0));
            }
        } else {
            const uint32_t base = sbase + (uint32_t)(s * C::STAGE_FLOATS) * 4;
#pragma unroll
            for (int c = tid; c < 2 * 64 * 8; c += 128) {
                const int row = c >> 3, kq = (c & 7) * 4;
                const bool second = row >= 64;
                const int gi = second ? j0 + row - 64 : i0 + row;
                const bool in = gi < (second ? rows_b : rows_a);
                const float* src = (second ? B + (int64_t)(in ? gi : 0) * ldb : A + (int64_t)(in ? gi : 0) * lda);
                const uint32_t dst = base + (uint32_t)(row * 36 + kq) * 4;
                const int64_t left = in ? ke - (k0 + kq) : 0;          // values of this piece inside the slice
                if (VEC) {
                    const int bytes = left >= 4 ? 16 : (left > 0 ? (int)left * 4 : 0);
                    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(bytes ? src + k0 + kq : src), "r"(bytes));
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int bytes = left > q ? 4 : 0;
                        asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst + 4 * q), "l"(bytes ? src + k0 + kq + q : src), "r"(bytes));
                    }
                }
            }
        }
        asm volatile("cp.async.commit_group;");
    };
    float2 acc[8][4];
#pragma unroll
    for (int q = 0; q < 8; ++q)
#pragma unroll
        for (int p = 0; p < 4; ++p) acc[q][p] = make_float2(0.f, 0.f);
#pragma unroll
    for (int s = 0; s < C::STAGES - 1; ++s) {
        if (s < steps) stage_copy(s, kb + (int64_t)s * C::K);
        else asm volatile("cp.async.commit_group;");
    }
    for (int st = 0; st < steps; ++st) {
        asm volatile("cp.async.wait_group %0;" ::"n"(C::STAGES - 2));
        __syncthreads();
        if (st + C::STAGES - 1 < steps) stage_copy((st + C::STAGES - 1) % C::STAGES, kb + (int64_t)(st + C::STAGES - 1) * C::K);
        else asm volatile("cp.async.commit_group;");
        const float* S = smem + (size_t)(st % C::STAGES) * C::STAGE_FLOATS;
        if (TILE == 128) {
            const float4* As = reinterpret_cast<const float4*>(S);
            const float4* Bs = As + 128 * 16 / 4;
#pragma unroll
            for (int k = 0; k < 16; ++k) {
                const int x = k & 7;
                const float4 a0 = As[k * 32 + (ty ^ x)], a1 = As[k * 32 + ((ty + 16) ^ x)];
                const float4 b0 = Bs[k * 32 + (tx ^ x)], b1 = Bs[k * 32 + ((tx + 16) ^ x)];
                const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
                const float2 b[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w), make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
                for (int q = 0; q < 8; ++q)
#pragma unroll
                    for (int p = 0; p < 4; ++p) acc[q][p] = __ffma2_rn(make_float2(a[q], a[q]), b[p], acc[q][p]);
            }
        } else {
            const float* As = S + ty * 36;
            const float* Bs = S + (64 + tx) * 36;
#pragma unroll 2
            for (int k = 0; k < 32; k += 4) {
                float4 b[4];
#pragma unroll
                for (int p = 0; p < 4; ++p) b[p] = *reinterpret_cast<const float4*>(Bs + p * 16 * 36 + k);
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    const float4 a = *reinterpret_cast<const float4*>(As + q * 8 * 36 + k);
#pragma unroll
                    for (int p = 0; p < 4; ++p) {
                        acc[q][p] = __ffma2_rn(make_float2(a.x, a.y), make_float2(b[p].x, b[p].y), acc[q][p]);
                        acc[q][p] = __ffma2_rn(make_float2(a.z, a.w), make_float2(b[p].z, b[p].w), acc[q][p]);
                    }
                }
            }
        }
    }
    asm volatile("cp.async.wait_group 0;");
    __syncthreads();                                       // the stages are free (emit may use them)
#pragma unroll
    for (int q = 0; q < 8; ++q) {
        const int i = TILE == 128 ? 4 * ty + (q & 3) + (q >> 2) * 64 : ty + 8 * q;
#pragma unroll
        for (int p = 0; p < 4; ++p) {
            if (TILE == 128) {
                const int j = 4 * tx + 2 * (p & 1) + (p >> 1) * 64;
                emit(i, j, acc[q][p].x);
                emit(i, j + 1, acc[q][p].y);
            } else {
                emit(i, tx + 16 * p, acc[q][p].x + acc[q][p].y);
            }
        }
    }
}

}  // namespace obc
