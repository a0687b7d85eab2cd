// The rank-B update of the blocked row engine for long rows on the 5th-generation tensor cores: H -= sum_b z_b z_b^T over the
// compacted lower triangle of one row's private inverse Hessian (B <= 64 pending vectors), one 512-thread block per SM.
//
// A pass reads and writes every element of the triangle once (8 bytes); a tile takes about 2600 cycles of its SM's pipeline of copy,
// products, subtraction and store, which is the copy rate of HBM when all SMs pass at once (16 rows of 4608 alone: 51 ms of passes,
// 128 rows: 56 ms).  Everything but that traffic is kept off the warps: TMA brings tiles of 128 rows x 64 columns of H into shared memory and takes them back,
// tcgen05.mma (kind::f16) forms the tile's increment in tensor memory, and eight warps only subtract one from the other.
// The products cost nothing beside the traffic, so a pass takes as many pending vectors as tensor memory holds partial sums
// for; most of them wait in L2 (the mma.sync form spent half of a warp's time multiplying, so more vectors per pass bought it
// little).  48 or 64 of them by the row's length (blk_plan): the steps between two passes read them all.  During a pass the space of the FP32
// pending vectors is free and holds the tiles and operands.
//
// Operands.  Before the pass every pending vector is written as two FP16 planes, z * 2^e = hi + lo (hi rounded to 11 bits, lo
// the rounded rest: 22 significant bits), to global memory (they stay in L2).  The power of two takes the largest entry to
// [2^13, 2^14); an entry's error is then 2^-23 of itself or, where lo is subnormal, 2^-39 of the largest entry.  Where the diagonal
// (the live one, or the squares of the largest entries) spans more than 2^24 every slot has a power of its own (zexp), so that
// small rows of the matrix keep their own precision.  lo*hi + hi*lo + hi*hi is formed; the
// missing lo*lo is below 2^-22 of a product.  Boxes of 16 G vectors x 64 slots go into 128B-swizzled shared memory as
// MN-major operands.
//
// Rounding.  The tensor core truncates its FP32 accumulator after every instruction (measured: -0.46 units in the last
// place on average for one 16-deep product).  Every group of 16 vectors therefore has an accumulator of its own, the two
// small products are added first, and the groups are added in FP32 round-to-nearest with the last mantissa bit of each
// set, which turns "truncated" into "right on average" (+0.07; +0.15 after three chained products).
//
// Every wait is bounded.  When one expires the block abandons the pass: once all its threads have stopped, the issuing ones wait
// (with the built-in limit) for their copies and products in flight, and the row is reported with -OBC_ERR_TIMEOUT.
#pragma once
#include "engine.cuh"
#include "tensor_map.cuh"
#include <cuda_fp16.h>

namespace obc {

constexpr int FT_M = 128, FT_N = 64;              // tile
constexpr int FT_GMAX = 4;                        // groups of 16 pending vectors (two tiles' accumulators in tensor memory)
constexpr int FT_COLS = 512;
constexpr int FT_EW = 8;                          // warps that subtract: 32 rows x 32 columns each; four more issue
constexpr int FT_WAIT_LIMIT = 1 << 22;            // polls before a wait gives up
constexpr int FT_GROUP_BYTES = 16 * 128;          // one plane of 16 vectors x 64 slots of FP16
constexpr int FT_TILE_BYTES = FT_M * FT_N * 4;

// Tensor maps: the planes (slots, 64 vectors, hi / lo of every block) by groups of 16 vectors in the copied box, and the
// private triangles (32 columns, rows, column groups of all buffers) in boxes of a whole tile and of 32 columns x 32 rows.
struct FlushMaps { CUtensorMap z[FT_GMAX]; CUtensorMap h128, h32; };

struct FlushBars {                                // in shared memory; the barriers are re-initialised before every pass
    unsigned long long full_a[2], free_a[2], full_b[2], free_b[2], full_h[4], ready[4], free_h[4], done[2], free_d[2];
    uint32_t tmem; int abort;
};

// Buffers of a pass over g groups of 16 vectors in `bytes` of shared memory: row operands, column operands, tiles.
struct FlushBufs { int n_a, n_b, n_h; };
__host__ __device__ inline int ft_stage_bytes(int g, FlushBufs f) { return 2 * g * FT_GROUP_BYTES * (2 * f.n_a + f.n_b) + f.n_h * FT_TILE_BYTES; }
__host__ __device__ inline FlushBufs ft_bufs(int g, int bytes) {
    FlushBufs f{2, 2, 4};
    if (ft_stage_bytes(g, f) > bytes) f = FlushBufs{2, 1, 4};
    if (ft_stage_bytes(g, f) > bytes) f = FlushBufs{2, 2, 3};
    if (ft_stage_bytes(g, f) > bytes) f = FlushBufs{2, 1, 3};
    if (ft_stage_bytes(g, f) > bytes) f = FlushBufs{2, 1, 2};
    if (ft_stage_bytes(g, f) > bytes) f = FlushBufs{1, 1, 2};
    if (ft_stage_bytes(g, f) > bytes) f = FlushBufs{1, 1, 1};
    return f;
}

__device__ __forceinline__ uint32_t ft_smem(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void ft_bar_init(unsigned long long* b, int count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(ft_smem(b)), "r"(count) : "memory");
}
__device__ __forceinline__ void ft_bar_arrive(unsigned long long* b) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(ft_smem(b)) : "memory");
}
__device__ __forceinline__ void ft_expect(unsigned long long* b, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(ft_smem(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool ft_test(unsigned long long* b, int parity) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(ft_smem(b)), "r"(parity) : "memory");
    return ok != 0;
}
// false when the limit is reached or another thread of the block has given up
__device__ __forceinline__ bool ft_wait(unsigned long long* b, int parity, FlushBars* fb) {
    for (int i = 0; i < FT_WAIT_LIMIT; ++i) {
        if (ft_test(b, parity)) return true;
        if ((i & 15) == 15) {
            if (*(volatile int*)&fb->abort) return false;
            if (i >= 64) __nanosleep(32);
        }
    }
    *(volatile int*)&fb->abort = 1;
    return false;
}
__device__ __forceinline__ void ft_drain(unsigned long long* b, int parity) {
    for (int i = 0; i < FT_WAIT_LIMIT && !ft_test(b, parity); ++i) __nanosleep(32);
}
__device__ __forceinline__ void ft_load(uint32_t dst, const CUtensorMap* map, unsigned long long* bar, int x, int y, int z) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
                 ::"r"(dst), "l"(map), "r"(ft_smem(bar)), "r"(x), "r"(y), "r"(z) : "memory");
}
// the triangles are streamed past L2's other contents (evict first)
__device__ __forceinline__ uint64_t ft_stream_policy() {
    uint64_t p;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
    return p;
}
__device__ __forceinline__ void ft_load_stream(uint32_t dst, const CUtensorMap* map, unsigned long long* bar, int x, int y, int z, uint64_t pol) {
    asm volatile("cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;"
                 ::"r"(dst), "l"(map), "r"(ft_smem(bar)), "r"(x), "r"(y), "r"(z), "l"(pol) : "memory");
}
__device__ __forceinline__ void ft_store_stream(uint32_t src, const CUtensorMap* map, int x, int y, int z, uint64_t pol) {
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.bulk_group.L2::cache_hint [%1, {%2, %3, %4}], [%0], %5;"
                 ::"r"(src), "l"(map), "r"(x), "r"(y), "r"(z), "l"(pol) : "memory");
}
// MN-major operand, 128B swizzle: 64-slot blocks `block` bytes apart, groups of 8 vectors 1024 bytes apart
__device__ __forceinline__ uint64_t ft_desc(uint32_t addr, uint32_t block) {
    uint64_t d = (uint64_t)((addr >> 4) & 0x3fffu);
    d |= (uint64_t)(block >> 4) << 16;
    d |= (uint64_t)(1024 >> 4) << 32;
    d |= (uint64_t)1 << 46;
    d |= (uint64_t)2 << 61;
    return d;
}
__device__ __forceinline__ void ft_mma(uint32_t d, uint64_t a, uint64_t b, uint32_t acc) {
    constexpr uint32_t idesc = (1u << 4) | (1u << 15) | (1u << 16) | ((uint32_t)(FT_N >> 3) << 17) | ((uint32_t)(FT_M >> 4) << 24);
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
                 "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
                 ::"r"(d), "l"(a), "l"(b), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void ft_commit(unsigned long long* bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(ft_smem(bar)) : "memory");
}
// 32 rows (lanes) x 16 columns
__device__ __forceinline__ void ft_tmem_ld(uint32_t addr, uint32_t (&v)[16]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                   "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
                 : "r"(addr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}
// 2^-e of a slot's own power (wide diagonals only)
__device__ __forceinline__ float ft_unscale(const signed char* zexp, int slot) { return __int_as_float((127 - zexp[slot]) << 23); }

__device__ __forceinline__ void ft_alloc(FlushBars* fb) {
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(ft_smem(&fb->tmem)), "r"(FT_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::);
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void ft_free(FlushBars* fb) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(fb->tmem), "r"(FT_COLS));
    }
}
// One thread, before / after a pass.
__device__ __forceinline__ void ft_init_bars(FlushBars* fb) {
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        ft_bar_init(&fb->full_a[q], 1); ft_bar_init(&fb->free_a[q], 1); ft_bar_init(&fb->full_b[q], 1); ft_bar_init(&fb->free_b[q], 1);
        ft_bar_init(&fb->done[q], 1); ft_bar_init(&fb->free_d[q], FT_EW);
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        ft_bar_init(&fb->full_h[q], 1); ft_bar_init(&fb->ready[q], FT_EW); ft_bar_init(&fb->free_h[q], 1);
    }
    fb->abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void ft_inval_bars(FlushBars* fb) {
    unsigned long long* b = fb->full_a;
#pragma unroll
    for (int q = 0; q < (int)(offsetof(FlushBars, tmem) / 8); ++q) asm volatile("mbarrier.inval.shared::cta.b64 [%0];" ::"r"(ft_smem(b + q)) : "memory");
}

// Tile sequence of a pass: column blocks of 64 in order, down the rows from the diagonal -- the order of memory (along the rows
// instead, every tile is in other pages: 128 x 4608 153 against 149 ms).
__device__ __forceinline__ void ft_next_tile(int& rb, int& c, int m1) {
    if (++rb * FT_M >= m1) { c += FT_N; rb = c / FT_M; }
}
// A position in a ring of n buffers and how often it has gone round.
struct Ring {
    int at = 0, round = 0;
    __device__ __forceinline__ void next(int n) { if (++at == n) { at = 0; ++round; } }
};
struct FlushGeom {                                // of a pass
    const FlushMaps* maps; int plane, buf, G, T, m1; FlushBufs nb; uint32_t sa, sb, sh, tmem;
};
// The parts of tile (rb, c) that hold data, each as f(map, 32-column group, first row inside the tile): the whole tile
// below the diagonal, on it the 32 x 32 parts that reach it.
template <typename F>
__device__ __forceinline__ void ft_parts(const FlushGeom& q, int rb, int c, F f) {
    if (c < rb * FT_M) f(&q.maps->h128, 0, 0);
    else {
#pragma unroll
        for (int cg = 0; cg < FT_N / 32; ++cg)
            for (int r = 0; r < FT_M; r += 32)
                if (c + 32 * cg <= rb * FT_M + r && rb * FT_M + r < q.m1) f(&q.maps->h32, cg, r);
    }
}
// Copies of the tile of H at (rb, c).  One thread.
__device__ __forceinline__ bool ft_copy_tile(const FlushGeom& q, FlushBars* fb, Ring& h, int rb, int c, uint64_t pol) {
    if (h.round > 0 && !ft_wait(&fb->free_h[h.at], (h.round - 1) & 1, fb)) return false;
    uint32_t bytes = FT_TILE_BYTES;
    if (c >= rb * FT_M) { bytes = 0; ft_parts(q, rb, c, [&](const CUtensorMap*, int, int) { bytes += 32 * 128; }); }
    ft_expect(&fb->full_h[h.at], bytes);
    ft_parts(q, rb, c, [&](const CUtensorMap* m, int cg, int r) {
        ft_load_stream(q.sh + h.at * FT_TILE_BYTES + cg * (FT_M * 128) + r * 128, m, &fb->full_h[h.at], 0, rb * FT_M + r, q.buf + (c >> 5) + cg, pol);
    });
    h.next(q.nb.n_h);
    return true;
}
// Copies of the vectors at the tile's rows and, first tile of a column block, at its columns.  One thread (another one: the
// operands run ahead of the tiles, whose buffers are held until they are back in memory).
__device__ __forceinline__ bool ft_copy_operands(const FlushGeom& q, FlushBars* fb, Ring& b, Ring& a, int rb, int c) {
    const uint32_t blk = q.G * 2 * FT_GROUP_BYTES;    // both planes of 64 slots
    const CUtensorMap* zm = &q.maps->z[q.G - 1];
    if (rb == c / FT_M) {
        if (b.round > 0 && !ft_wait(&fb->free_b[b.at], (b.round - 1) & 1, fb)) return false;
        ft_expect(&fb->full_b[b.at], blk);
        ft_load(q.sb + b.at * blk, zm, &fb->full_b[b.at], c, 0, q.plane);
        b.next(q.nb.n_b);
    }
    if (a.round > 0 && !ft_wait(&fb->free_a[a.at], (a.round - 1) & 1, fb)) return false;
    ft_expect(&fb->full_a[a.at], 2 * blk);
    ft_load(q.sa + a.at * 2 * blk, zm, &fb->full_a[a.at], rb * FT_M, 0, q.plane);
    ft_load(q.sa + (a.at * 2 + 1) * blk, zm, &fb->full_a[a.at], rb * FT_M + 64, 0, q.plane);
    a.next(q.nb.n_a);
    return true;
}
// Products of tile t; first / last: of its column block.  One thread.
template <int GM>
__device__ __forceinline__ bool ft_multiply(const FlushGeom& q, FlushBars* fb, int t, Ring& b, Ring& a, bool first, bool last) {
    const uint32_t blk = q.G * 2 * FT_GROUP_BYTES;
    const int buf = t & 1;
    if (first && !ft_wait(&fb->full_b[b.at], b.round & 1, fb)) return false;
    if (!ft_wait(&fb->full_a[a.at], a.round & 1, fb)) return false;
    if (t > 1 && !ft_wait(&fb->free_d[buf], ((t >> 1) - 1) & 1, fb)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint64_t da = ft_desc(q.sa + a.at * 2 * blk, blk), db = ft_desc(q.sb + b.at * blk, blk);
    const uint32_t d = q.tmem + buf * (GM * FT_N);
    constexpr uint64_t STEP = FT_GROUP_BYTES >> 4;
    const uint64_t LO = q.G * STEP;
#pragma unroll
    for (int k = 0; k < GM; ++k) if (k < q.G) ft_mma(d + k * FT_N, da + LO + k * STEP, db + k * STEP, 0u);
#pragma unroll
    for (int k = 0; k < GM; ++k) if (k < q.G) ft_mma(d + k * FT_N, da + k * STEP, db + LO + k * STEP, 1u);
#pragma unroll
    for (int k = 0; k < GM; ++k) if (k < q.G) ft_mma(d + k * FT_N, da + k * STEP, db + k * STEP, 1u);
    ft_commit(&fb->done[buf]);
    ft_commit(&fb->free_a[a.at]);
    a.next(q.nb.n_a);
    if (last) { ft_commit(&fb->free_b[b.at]); b.next(q.nb.n_b); }
    return true;
}
// The last n uses of a ring of `len` barriers are over (all of them, if there were fewer).
__device__ __forceinline__ void ft_ring_over(unsigned long long* bars, Ring r, int len, int n) {
    const int used = r.round * len + r.at;
    for (int x = max(0, used - n); x < used; ++x) ft_drain(&bars[x % len], (x / len) & 1);
}
// The products of `tiles` tiles and all that they signal are over; b, a: the operand rings as ft_multiply left them.
__device__ __forceinline__ void ft_products_over(const FlushGeom& q, FlushBars* fb, int tiles, Ring b, Ring a) {
    if (tiles > 0) ft_drain(&fb->done[(tiles - 1) & 1], ((tiles - 1) >> 1) & 1);
    ft_ring_over(fb->free_a, a, q.nb.n_a, 1);
    ft_ring_over(fb->free_b, b, q.nb.n_b, 1);
}
// Takes the tile at (rb, c) back to memory once every warp has finished its part.  One thread (of all tiles).
__device__ __forceinline__ bool ft_store(const FlushGeom& q, FlushBars* fb, Ring& h, int rb, int c, uint64_t pol) {
    if (!ft_wait(&fb->ready[h.at], h.round & 1, fb)) return false;
    ft_parts(q, rb, c, [&](const CUtensorMap* m, int cg, int r) {
        ft_store_stream(q.sh + h.at * FT_TILE_BYTES + cg * (FT_M * 128) + r * 128, m, 0, rb * FT_M + r, q.buf + (c >> 5) + cg, pol);
    });
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
    asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    ft_bar_arrive(&fb->free_h[h.at]);
    h.next(q.nb.n_h);
    return true;
}
// A warp's 32 x 32 part of tile t: H minus the increment, in shared memory.
template <int GM>
__device__ __forceinline__ bool ft_subtract(const FlushGeom& q, FlushBars* fb, int t, Ring& hq, int rb, int c, float unscale, const signed char* zexp) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int h = hq.at, buf = t & 1;
    const int cg = warp >> 2, r0 = rb * FT_M + 32 * (warp & 3), col = c + 32 * cg;
    bool ok = ft_wait(&fb->full_h[h], hq.round & 1, fb);
    ok = ok && ft_wait(&fb->done[buf], (t >> 1) & 1, fb);
    if (!__all_sync(0xffffffffu, ok)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const bool any = r0 < q.m1 && col <= r0;
    const uint32_t row = q.sh + h * FT_TILE_BYTES + cg * (FT_M * 128) + (32 * (warp & 3) + lane) * 128;
    const uint32_t d = q.tmem + buf * (GM * FT_N) + 32 * cg + ((uint32_t)(32 * (warp & 3)) << 16);
    const float rs = zexp && any && r0 + lane < q.m1 ? -ft_unscale(zexp, r0 + lane) : -unscale;
#pragma unroll
    for (int v = 0; v < 2; ++v) {                     // 16 columns at a time
        if (any) {
            uint32_t x[16];
            float acc[16];
            ft_tmem_ld(d + 16 * v, x);
#pragma unroll
            for (int e = 0; e < 16; ++e) acc[e] = __uint_as_float(x[e] | 1u);
            for (int k = 1; k < q.G; ++k) {
                ft_tmem_ld(d + k * FT_N + 16 * v, x);
#pragma unroll
                for (int e = 0; e < 16; e += 2) {
                    const float2 s = __fadd2_rn(make_float2(acc[e], acc[e + 1]), make_float2(__uint_as_float(x[e] | 1u), __uint_as_float(x[e + 1] | 1u)));
                    acc[e] = s.x; acc[e + 1] = s.y;
                }
            }
            if (zexp) {
#pragma unroll
                for (int e = 0; e < 16; ++e) acc[e] *= col + 16 * v + e < q.m1 ? ft_unscale(zexp, col + 16 * v + e) : 0.f;
            }
#pragma unroll
            for (int e = 0; e < 4; ++e) {
                const uint32_t at = row + ((uint32_t)((4 * v + e) ^ (lane & 7)) << 4);
                float4 o;
                asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(o.x), "=f"(o.y), "=f"(o.z), "=f"(o.w) : "r"(at) : "memory");
                o.x = fmaf(rs, acc[4 * e], o.x); o.y = fmaf(rs, acc[4 * e + 1], o.y);
                o.z = fmaf(rs, acc[4 * e + 2], o.z); o.w = fmaf(rs, acc[4 * e + 3], o.w);
                asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(at), "f"(o.x), "f"(o.y), "f"(o.z), "f"(o.w) : "memory");
            }
        }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if (lane == 0) { ft_bar_arrive(&fb->free_d[buf]); ft_bar_arrive(&fb->ready[h]); }
    hq.next(q.nb.n_h);
    return true;
}

// One pass over the triangle whose first column group is `tri` in the maps, already compacted to m1 rows.  Before it: the planes are in the new
// slot numbering and zero up to a multiple of 16 vectors, the barriers are initialised, plain accesses are fenced against
// the copies, and the block has synchronised.
//   plane     first of the block's two planes (hi, lo) in the maps
//   unscale   2^-2e of the planes' power, or zexp: the slots' own powers
//   GM        most groups of 16 vectors that the kernel takes
//   stop      tile (from 1) at which the products give up, for tests; 0: never
template <int GM>
__device__ __forceinline__ bool blk_flush_tc(const FlushMaps* maps, int plane, int tri, unsigned char* stage, int stage_bytes, FlushBars* fb, int m1,
                                             int nb, float unscale, const signed char* zexp, int stop) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    FlushGeom q;
    q.maps = maps; q.plane = plane; q.buf = tri; q.m1 = m1;
    q.G = (nb + 15) >> 4;
    q.nb = ft_bufs(q.G, stage_bytes);
    q.sh = ft_smem(stage);
    q.sa = q.sh + q.nb.n_h * FT_TILE_BYTES;
    q.sb = q.sa + q.nb.n_a * 4 * q.G * FT_GROUP_BYTES;
    q.tmem = fb->tmem;
    const int n_rb = (m1 + FT_M - 1) / FT_M;
    q.T = (n_rb - 1) * n_rb / 2 * (FT_M / FT_N) + (m1 + FT_N - 1) / FT_N;
    Ring h, b, a;
    int rb = 0, c = 0, t = 0;
    if (warp < FT_EW) {
        for (; t < q.T; ++t) {
            if (!ft_subtract<GM>(q, fb, t, h, rb, c, unscale, zexp)) break;
            ft_next_tile(rb, c, m1);
        }
    } else if (warp == FT_EW && lane == 0) {
        const uint64_t pol = ft_stream_policy();
        for (; t < q.T; ++t) {
            if (!ft_copy_tile(q, fb, h, rb, c, pol)) break;
            ft_next_tile(rb, c, m1);
        }
    } else if (warp == FT_EW + 3 && lane == 0) {
        for (; t < q.T; ++t) {
            if (!ft_copy_operands(q, fb, b, a, rb, c)) break;
            ft_next_tile(rb, c, m1);
        }
    } else if (warp == FT_EW + 1 && lane == 0) {
        for (; t < q.T; ++t) {
            if (t + 1 == stop) {                      // (as if a wait had expired: constant limits keep the waits short)
                *(volatile int*)&fb->abort = 1;
                break;
            }
            int nrb = rb, nc = c;
            ft_next_tile(nrb, nc, m1);
            if (!ft_multiply<GM>(q, fb, t, b, a, rb == c / FT_M, nc != c)) break;
            rb = nrb; c = nc;
        }
    } else if (warp == FT_EW + 2 && lane == 0) {
        const uint64_t pol = ft_stream_policy();
        for (; t < q.T; ++t) {
            if (!ft_store(q, fb, h, rb, c, pol)) break;
            ft_next_tile(rb, c, m1);
        }
        asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
    }
    __syncwarp();
    __syncthreads();
    // Nothing may land or be signalled after the block has moved on.  The products' last signals may be under way in any case; copies
    // are all consumed unless the pass was abandoned, which is only certain now: another thread's wait may have expired
    // after this one's last copy.
    const bool aborted = *(volatile int*)&fb->abort != 0;
    if (warp == FT_EW + 1 && lane == 0) ft_products_over(q, fb, t, b, a);
    if (aborted && warp == FT_EW && lane == 0) ft_ring_over(fb->full_h, h, q.nb.n_h, q.nb.n_h);
    if (aborted && warp == FT_EW + 3 && lane == 0) {
        ft_ring_over(fb->full_b, b, q.nb.n_b, q.nb.n_b);
        ft_ring_over(fb->full_a, a, q.nb.n_a, q.nb.n_a);
    }
    __syncwarp();
    __syncthreads();
    asm volatile("fence.proxy.async;" ::: "memory");  // the copies' writes before the plain accesses that follow
    if (threadIdx.x == 0) ft_inval_bars(fb);
    __syncthreads();
    return !aborted;
}

}  // namespace obc
