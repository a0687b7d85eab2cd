// Row elimination engine with deferred Lemma-1 updates (Algorithm 1 / Algorithm 3 of "Optimal Brain
// Compression"), one thread block per weight-matrix row, several rows per SM.
//
// A greedy step needs only three things from the row's inverse Hessian: its diagonal (for the scores), the
// pivot column (for the weight update, Eq. 3 / Eq. 7) and, later, everything else.  Lemma 1 is a rank-1
// update, so B of them can be held back as vectors z_b = H[:,p_b] / sqrt([H]_pp) (each taken from the matrix
// as it would be at its own step) and applied together:
//       H_true = H_stored - sum_b z_b z_b^T .
// The pivot column of a step is then one column of H_stored corrected by the pending vectors (m x B work),
// and the m x m matrix is read and written once per B steps instead of once per step.  Picks, weights and
// losses are the same as with step-by-step updates up to the order of the FP32 roundings.
//
// Layout.  The private copy keeps the lower triangle only (the matrix stays symmetric).  Slots [0, m0) are
// fixed between two flushes; eliminated slots are marked dead (perm = -1).  The flush applies the pending
// vectors and compacts at the same time: a dead slot h below the new size m1 is taken over by a live slot
// s >= m1, i.e. element (i, j) of the new triangle is read from (max(si, sj), min(si, sj)) of the old one.
// All such foreign reads come from rows >= m1, which the flush never writes, so it runs in place.
// The flush is a rank-B update and runs on the tensor cores: with 512 threads per row on tcgen05 with the triangle moved by TMA
// (flush_tc.cuh; pending vectors beyond shared memory wait in a global buffer that stays in L2), with several rows per SM by
// mma.sync (warp tiles of 16 rows x 64 columns on packed FP16 planes, see blk_flush_f16): there the passes of one row
// overlap the steps of another, and tensor memory and tile buffers would have to be shared.  The O(m) selection state (weights,
// diagonal) is FP64, as in the streaming engine.  Once the live triangle fits into the shared memory of the pending
// vectors, the row finishes on chip: one slot per thread with its state in registers, eight updates deferred.
//
// Shares of rows.  When a launch has more rows than resident blocks and the rows do not divide evenly, whole waves
// would leave most SMs idle through the last one.  Instead every block gets the same amount of work: the rows
// are laid end to end and cut into gridDim.x equal pieces.  A row that straddles a cut is started by the block before
// the cut -- as that block's FIRST item -- up to a flush boundary near the cut, where its state (weights, diagonal,
// slot map; the triangle stays in a buffer of its own) is saved, and it is finished by the next block as that
// block's LAST item.  The state is complete long before it is needed; the reader still checks a flag with a bounded
// wait (a cooperative launch keeps all blocks resident) and reports a row it could not pick up through row_status.
//
// Step protocol.  Between two flushes every slot belongs to one thread (groups of 4 consecutive slots per
// thread), which is the only one to touch wd[j], dg[j], perm[j] and its entries of the pending vectors; the
// update phase also leaves an FP32 estimate of each own slot's next score in registers.  The warps publish one record each
// (their smallest estimate, and whether another one is near it), and after the single barrier of the step every warp reads the
// records and derives the same winner (fast_pick).  Only where another slot's estimate is within 1e-4 of the smallest is the
// choice made on FP64 scores, with a second barrier (thread_best, block_pick): ties to the last bit go by original index.
// Records alternate between two buffers by step parity.
// What bounds a step is the latency of this chain (scores, pick, pivot column, corrections, state), not its arithmetic.
#pragma once
#include "flush_tc.cuh"
#include <type_traits>

namespace obc {

constexpr int BLK_MAXB = 64;
constexpr int BLK_REC_BYTES = 640;            // one record buffer: 16 warps x fast record, 16 warps x (s, key, slot, orig)
constexpr int BLK_OFF_BC = 1280;              // Bcast (grid parameters, flush bookkeeping)
constexpr int BLK_OFF_PV = 1536;              // int pv[64]   slots eliminated since the last flush
constexpr int BLK_OFF_HL = 1792;              // int hl[64]   holes (dead slots below the new size)
constexpr int BLK_OFF_MV = 2048;              // int mv[64]   live slots that move into the holes
constexpr int BLK_OFF_CM = 2304;
constexpr int BLK_OFF_RF = 2944;              // float rf[64]  min/max reduction of the compound grid
constexpr int BLK_OFF_GRP = 3200;             // forced groups: int slot[4], float M[4][4] (pivot columns at the pivot slots)
constexpr int BLK_OFF_SCHED = 3280;           // shares of rows: int[4] of the item in work, address of its triangle
constexpr int BLK_OFF_FB = 3328;              // FlushBars
constexpr int BLK_FIXED = 3584;
static_assert(BLK_OFF_FB + sizeof(FlushBars) <= BLK_FIXED, "");
constexpr int BLK_GS = 4;                     // forced eliminations taken together

// Per-row state in shared memory: perm (int32), srcm (uint16); optional: the row in original order (weight trace), one byte
// per block of the N:M pattern, off-diagonals of block pruning; wd and dg (FP64): first, or, where passes run on
// tcgen05, last, next to the pending vectors -- such a pass parks them in global memory and uses their space too.
// (block pruning, bc = block size 4 or 8: the 6 or 28 off-diagonal entries of every block's c x c diagonal block, FP64)
__host__ __device__ inline size_t blk_state_bytes(int cap, bool wfull, bool nm = false, int bc = 0) {
    return (size_t)20 * cap + (((size_t)2 * cap + 15) & ~(size_t)15) + (wfull ? (size_t)4 * cap : 0) +
           (nm ? (((size_t)(cap >> 1) + 15) & ~(size_t)15) : 0) + (bc == 8 ? (size_t)28 * cap : (bc ? (size_t)12 * cap : 0));
}
// Stride of the pending vectors for a row of m slots: = 4 (mod 32), so that the tensor-core fragments of the flush (every second
// row of 4 pairs of vectors x 8 consecutive slots per load) touch 32 different banks.
__host__ __device__ inline int blk_ldz(int m) { return ((m + 12 + 31) & ~31) + 4; }     // >= m + 16
// Updates that a row of m slots defers between two passes: as many vectors as there is room for.  pairs: passes by mma.sync on packed
// planes, which hold two vectors each (fewer than 512 threads; no overflow vectors there).
__host__ __device__ inline int blk_updates(int m, int panel_floats, int max_pending, int g_vectors, bool pairs) {
    const int fit = panel_floats / blk_ldz(m), n = !pairs ? fit + g_vectors : fit < 2 ? 2 : fit & ~1;
    return n < max_pending ? n : max_pending;
}
// On chip: TAIL_B deferred updates as two arrays per slot (column entries v, v / [H]_pp; TAIL_LD floats apart: 128-bit accesses
// of consecutive slots meet no bank twice), then the lower triangle, its rows end to end: column p of 32 rows from a multiple of
// 32 on touches 32 different banks (triangular numbers mod 32 are a permutation).
constexpr int TAIL_B = 8, TAIL_LD = 12;
__host__ __device__ __forceinline__ int tail_at(int i, int j) { return i * (i + 1) / 2 + j; }      // j <= i
static size_t blk_tail_bytes(int ms) { return (size_t)8 * TAIL_LD * ms + (size_t)4 * tail_at(ms, 0); }

// ---- shares of rows ------------------------------------------------------------------------------------------------
constexpr int BLK_SPLIT_WAIT_LIMIT = 1 << 22;  // polls (256 ns apart) before a block gives up on a row its neighbour started
struct SplitHeader {                          // what the block that started a row leaves for the one that finishes it
    int s_cut;                                // steps done (0: the row was not started)
    int m0;                                   // live slots, all in [0, m0), nothing pending
    int done;                                 // 1: nothing is left to do (the row was finished, or failed and was reported)
    int pad[61];
};
// followed by: double wd[cap], double dg[cap], int perm[cap], float wfull[cap]
__host__ __device__ inline size_t blk_split_stride(int cap) { return sizeof(SplitHeader) + (size_t)28 * cap + 256; }

// Work model of a row, in units of "half a matrix element moved by a flush": a pass over the compacted triangle of m
// slots costs m^2 / 2, a deferred-update step costs as much as blk_step_cost of those, a step on chip 0.6 of that.  Fitted when every pass
// ran by mma.sync (1.1 - 1.3e-10 s per m^2; a step 7 us with one 512-thread row per SM, 3.4 us with several smaller blocks per SM) and a
// step on chip took 8000 cycles (1500 now).  Passes and steps have become shorter since and the values were not fitted again: 256 rows x
// 2304 of 25 ms each on 148 SMs take 43.5 ms, which is 256 / 148 of a row.
__host__ __device__ inline double blk_step_cost(int nt) { return nt >= 512 ? 30000.0 : 14000.0; }

// The flush boundary of a row's schedule at which about num/den of the row's work is done (0: before the first
// boundary; total: the share reaches into the on-chip end of the row, which is then left to the starting block).
// Every thread of a block computes the same value from the same arguments.
static __device__ __noinline__ int blk_cut_step(int d, int ms, int total, int panel_floats, int max_pending, int g_vectors,
                                        bool pairs, int num, int den, double step_cost) {
    double all = 0.0, at = 0.0;
    int cut = 0;
    for (int pass = 0; pass < 2; ++pass) {
        int m = d, s = 0;
        double cost = 0.0;
        while (s < total && m > ms) {
            int b = blk_updates(m, panel_floats, max_pending, g_vectors, pairs);
            b = max(1, min(b, min(m - ms, total - s)));
            cost += step_cost * b;
            s += b; m -= b;
            if (s >= total) break;
            cost += 0.5 * (double)m * (double)m;                  // the pass over the compacted triangle
            if (pass == 1 && m > ms && cost <= at) cut = s;       // last boundary not beyond the share
        }
        cost += step_cost * 0.6 * (total - s);                    // steps on chip
        if (pass == 0) { all = cost; at = all * (double)num / (double)den; }
    }
    return cut;
}

// The it-th item of block `blk` out of `ng` when `rows` rows are shared out: false when there is none.  Without
// shares: whole rows blk, blk + ng, ...  With shares: positions in units of 1/ng of a row, row r covers
// [r ng, (r+1) ng) and the block covers [blk rows, (blk+1) rows); the row that straddles the upper cut is started first
// (head_num/ng of it), the one that straddles the lower cut is finished last.  Plain integer arithmetic, recomputed
// per item so that nothing of it stays in registers during a row.
enum { ITEM_FULL = 0, ITEM_HEAD = 1, ITEM_TAIL = 2 };
__device__ __forceinline__ bool blk_item(bool split, int blk, int ng, int rows, int it, int* rr, int* kind, int* head_num) {
    *kind = ITEM_FULL; *head_num = 0;
    if (!split) { *rr = blk + it * ng; return *rr < rows; }
    const long long a0 = (long long)blk * rows, a1 = a0 + rows;
    const int r_first = (int)(a0 / ng), tail_num = (int)(a0 - (long long)r_first * ng);
    const int r_last = (int)((a1 - 1) / ng);
    int hn = (int)(a1 - (long long)r_last * ng);
    if (hn == ng) hn = 0;                                          // the row ends at the cut: a whole row
    const int full_lo = tail_num ? r_first + 1 : r_first, full_hi = hn ? r_last : r_last + 1;
    const int n_items = (hn ? 1 : 0) + (full_hi - full_lo) + (tail_num ? 1 : 0);
    if (it >= n_items) return false;
    if (hn && it == 0) { *rr = r_last; *kind = ITEM_HEAD; *head_num = hn; }
    else if (tail_num && it == n_items - 1) { *rr = r_first; *kind = ITEM_TAIL; }
    else *rr = full_lo + it - (hn ? 1 : 0);
    return true;
}

// The cold paths of the hand-over are kept out of line, so that the register allocation of a row's loop is the
// same with and without them.
// Thread 0: wait (bounded) for the flag of the block that started the row; returns 1 when it is set.
static __device__ __noinline__ int blk_wait_flag(int* flag) {
    int ok = 0;
    for (int spin = 0; spin < BLK_SPLIT_WAIT_LIMIT; ++spin) {
        if (atomicAdd(flag, 0) != 0) { ok = 1; break; }
        __nanosleep(256);
    }
    __threadfence();
    return ok;
}
// Thread 0: publish the header of the row this block started (or declined to start), then the flag.
static __device__ __noinline__ void blk_publish(char* state, int* flag, int s_cut, int m0, int done) {
    SplitHeader* sh = reinterpret_cast<SplitHeader*>(state);
    sh->s_cut = s_cut; sh->m0 = m0; sh->done = done;
    __threadfence();
    atomicExch(flag, 1);
}
// All threads: state of a row between shared memory and the hand-over record (save = true: to the record).
static __device__ __noinline__ void blk_state_copy(bool save, char* state, int cap, int d, int m, int nt, double* wd, double* dg,
                                            int* perm, unsigned short* srcm, float* wfull) {
    char* base = state + sizeof(SplitHeader);
    double* swd = reinterpret_cast<double*>(base);
    double* sdg = swd + cap;
    int* sperm = reinterpret_cast<int*>(sdg + cap);
    float* swf = reinterpret_cast<float*>(sperm + cap);
    const int tid = threadIdx.x;
    if (save) {
        for (int j = tid; j < m; j += nt) { swd[j] = wd[j]; sdg[j] = dg[j]; sperm[j] = perm[j]; }
        if (wfull) for (int j = tid; j < d; j += nt) swf[j] = wfull[j];
        __threadfence();                   // state, triangle and outputs of every thread before the flag
    } else {
        for (int j = tid; j < cap; j += nt) {
            const bool in = j < m;
            wd[j] = in ? swd[j] : 0.0; dg[j] = in ? sdg[j] : 0.0; perm[j] = in ? sperm[j] : -1;
            srcm[j] = (unsigned short)j;
            if (wfull && j < d) wfull[j] = swf[j];
        }
    }
}

// Place of element (i, j), j <= i, of a private triangle: groups of columns one after the other, ld rows each.  A column is then one
// strip of consecutive lines instead of a line per row of the matrix.
// One row per SM (WIDE): 32 columns, rows of 128 bytes, so that a 128-row tile of a group is contiguous.  Else 4 columns, rows of 16
// bytes: a warp's 32 rows of a pivot column are 4 lines instead of 32 (one L1 tag look-up each, which the step's other accesses
// queued behind), 768 x 768 2:4 8.55 -> 8.06 ms, 3072 x 768 compound 85.2 -> 82.7.  With one long row per SM the smaller groups lose
// more in the passes and the holes than the columns gain: with passes on tcgen05 256 x 2304 OBQ 43.6 -> 46.2 ms, 128 x 1152 blocks of 4 7.74 ->
// 8.53; blocks of 8, whose passes are by mma.sync, 32 x 3072 88.4 -> 92.8, 64 x 2304 40.9 -> 41.8, 64 x 1536 15.0 -> 15.3.
template <bool WIDE> __device__ __forceinline__ int tri_at(int ld, int i, int j) {
    return WIDE ? ((j >> 5) * ld + i) * 32 + (j & 31) : ((j >> 2) * ld + i) * 4 + (j & 3);
}
__host__ __device__ inline size_t tri_floats(int cap) { return (size_t)((cap + 63) & ~63) * cap; }      // (an even number of groups)

struct Records {                              // views into one record buffer
    uint4* fast; unsigned* key; int* slot; int* orig; double* s;
};
__device__ __forceinline__ Records rec_view(char* scratch, int parity) {
    char* b = scratch + parity * BLK_REC_BYTES;
    Records r;
    r.fast = reinterpret_cast<uint4*>(b);     // [16]
    r.s = reinterpret_cast<double*>(b + 256); // [16]
    r.key = reinterpret_cast<unsigned*>(r.s + 16);
    r.slot = reinterpret_cast<int*>(r.key + 16);
    r.orig = r.slot + 16;
    return r;
}

// Monotone map of a float to an unsigned key (smaller float -> smaller key); NaN never reaches it.
__device__ __forceinline__ unsigned float_key(float x) {
    const unsigned u = __float_as_uint(x);
    return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float key_float(unsigned k) { return __uint_as_float((k & 0x80000000u) ? k & 0x7fffffffu : ~k); }
constexpr unsigned KEY_NONE = 0xFFFFFFFFu;
constexpr float NEAR = 1e-4f;                 // estimates this close (relative) are told apart by their FP64 scores

struct Pick { int slot; int orig; double s; };

// The block's smallest estimate.  m1: the thread's smallest (slot, orig: its slot; slot < 0: none), m2: its second smallest.
// `sure`: no other estimate of the block is near it and it is well inside the FP32 range, so its slot has the smallest FP64
// score too (an estimate is off by a few 1e-7).  One barrier.
template <int NT>
__device__ __forceinline__ Pick fast_pick(float m1, float m2, int slot, int orig, const Records& rec, bool* sure) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned key = slot >= 0 ? float_key(m1) : KEY_NONE;
    const unsigned kmin = __reduce_min_sync(0xffffffffu, key);
    const float v = key_float(kmin), t = v + NEAR * fabsf(v);
    const unsigned near = __ballot_sync(0xffffffffu, slot >= 0 && m1 <= t), two = __ballot_sync(0xffffffffu, m2 <= t);
    const bool many = kmin == KEY_NONE || two != 0u || __popc(near) != 1;
    if (many ? lane == 0 : m1 <= t && slot >= 0) rec.fast[warp] = make_uint4(kmin, (unsigned)slot, (unsigned)orig, many ? 1u : 0u);
    __syncthreads();
    uint4 q = make_uint4(KEY_NONE, 0u, 0u, 0u);
    if (lane < NW) q = rec.fast[lane];
    const unsigned kg = __reduce_min_sync(0xffffffffu, q.x);
    const float vg = key_float(kg), tg = vg + NEAR * fabsf(vg);
    const unsigned at = __ballot_sync(0xffffffffu, q.x == kg);
    const unsigned others = __ballot_sync(0xffffffffu, q.x != kg && q.x <= float_key(tg));
    const uint4 w = rec.fast[(__ffs(at) - 1) & (NW - 1)];
    *sure = others == 0u && __popc(at) == 1 && w.w == 0u && vg >= 1e-30f && vg <= 1e30f;
    Pick p;
    p.slot = kg == KEY_NONE ? -1 : (int)w.y; p.orig = (int)w.z; p.s = 0.0;
    return p;
}
// A slot that is known: its owner names it, the others have slot < 0.  One barrier.
template <int NT>
__device__ __forceinline__ Pick known_pick(int slot, int orig, const Records& rec) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const unsigned has = __ballot_sync(0xffffffffu, slot >= 0);
    if (has ? slot >= 0 : lane == 0) rec.fast[warp] = make_uint4(has ? 0u : KEY_NONE, (unsigned)slot, (unsigned)orig, 0u);
    __syncthreads();
    const unsigned at = __ballot_sync(0xffffffffu, lane < NW && rec.fast[lane & (NW - 1)].x == 0u);
    const uint4 w = rec.fast[at ? __ffs(at) - 1 : 0];
    Pick p;
    p.slot = at ? (int)w.y : -1; p.orig = (int)w.z; p.s = 0.0;
    return p;
}

// Combines one candidate per lane into the lane holding the smallest (s, orig); key = float_key((float)s)
// orders all but near-equal candidates, which are then compared exactly.  Returns the winning lane or -1.
__device__ __forceinline__ int warp_winner(unsigned key, double s, int orig) {
    const unsigned kmin = __reduce_min_sync(0xffffffffu, key);
    if (kmin == KEY_NONE) return -1;
    const unsigned cand = __ballot_sync(0xffffffffu, key == kmin);
    if (__popc(cand) == 1) return __ffs(cand) - 1;
    double bs = (key == kmin) ? s : CUDART_INF;
    int bo = (key == kmin) ? orig : 0x7fffffff;
    int bl = threadIdx.x & 31;
#pragma unroll
    for (int off = 16; off; off >>= 1) {
        const double s2 = __shfl_xor_sync(0xffffffffu, bs, off);
        const int o2 = __shfl_xor_sync(0xffffffffu, bo, off);
        const int l2 = __shfl_xor_sync(0xffffffffu, bl, off);
        if (key_less(s2, o2, bs, bo)) { bs = s2; bo = o2; bl = l2; }
    }
    return bl;
}

// Every thread holds at most one candidate (slot < 0: none).  Publishes the warp's best in the record buffer,
// then, after the barrier, every warp derives the block's best from the records.
template <int NT>
__device__ __forceinline__ Pick block_pick(unsigned key, double s, int slot, int orig, const Records& rec) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (slot < 0) key = KEY_NONE;
    const int wl = warp_winner(key, s, orig);
    if (wl < 0) { if (lane == 0) rec.key[warp] = KEY_NONE; }
    else if (lane == wl) {
        rec.key[warp] = key; rec.slot[warp] = slot; rec.orig[warp] = orig;
        rec.s[warp] = s;
    }
    __syncthreads();
    const bool in = lane < NW;
    const unsigned k2 = in ? rec.key[lane] : KEY_NONE;
    const double s2 = (in && k2 != KEY_NONE) ? rec.s[lane] : CUDART_INF;
    const int o2 = (in && k2 != KEY_NONE) ? rec.orig[lane] : 0x7fffffff;
    const int ww = warp_winner(k2, s2, o2);
    Pick p;
    p.slot = -1; p.orig = -1; p.s = 0.0;
    if (ww >= 0) { p.slot = rec.slot[ww]; p.orig = rec.orig[ww]; p.s = rec.s[ww]; }
    return p;
}

// Slot ownership between two flushes: thread t owns the slots 4t .. 4t+3 of every group of 4 NT slots, i.e.
// slot(k) = (k / 4) * 4 NT + 4 t + (k % 4) for k < KMAX, so that its entries of a pending vector, of a matrix
// row and of the state arrays are 16 contiguous bytes.
template <int NT>
__device__ __forceinline__ int own_slot(int k) { return (k >> 2) * (4 * NT) + (threadIdx.x << 2) + (k & 3); }

// err = q(w) - w on the row's grid.  Kept out of line: it is reached once per slot and step in the OBQ kernels,
// and inlining it at every use multiplies the code size of a kernel whose instruction footprint already matters
// (several rows in different phases share one SM's instruction cache).
static __device__ __noinline__ double grid_error(double w, double sc, double isc, double ze, double mq) {
    double code;
    return grid_q_fast(w, sc, isc, ze, mq, &code) - w;
}

// The grid of a row as the estimates use it: the codes' integer range without the zero point.  lo > hi: a zero point whose
// sum with a code is not exact, or a scale far outside the range of ordinary weights; there every estimate is 0, which leaves the
// choice to the FP64 scores of all slots.
struct GridRange { int lo, hi; };
__device__ __forceinline__ GridRange grid_range(double sc, double ze, double mq) {
    const double fine = ze * 1073741824.0;                     // (a multiple of 2^-30 below 1e5 plus a code: 48 bits)
    const bool exact = (ze == rint(ze) && fabs(ze) < 1e9) || (fine == rint(fine) && fabs(ze) < 1e5);
    const bool plain = exact && fabs(sc) > 1e-30 && fabs(sc) < 1e30;      // (false for NaN)
    GridRange g;
    g.lo = plain ? (int)ceil(-ze) : 1;
    g.hi = plain ? (int)floor(mq - ze) : 0;
    return g;
}

// FP32 estimate of the score of a slot (relative error of a few 1e-7): it only screens candidates, slots that are near the best
// estimate are told apart by FP64 scores.  On a grid the distance to the nearest code's value is taken in FP64, as the exact score
// takes it: a small distance is what wins, and weights may lie on the grid already.  x + 1.5 * 2^52 - 1.5 * 2^52 rounds x to an
// integer whose low 32 bits are the sum's (rint, the clamps and the conversions take four times as many slots of the FP64
// and conversion pipes).
template <bool Q>
__device__ __forceinline__ float score_estimate(double w, double dgv, bool quant, double sc, double isc, double ze, double mq,
                                                const GridRange& gr) {
    float ef;
    if (Q && quant) {
        constexpr double M = 6755399441055744.0;
        const double t = w * isc, u = t + M;
        const int r = __double2loint(u);
        // (the high word says whether the integer fits 32 bits: it has to agree with the low word's sign.)  Next to a rounding
        // boundary the two possible codes give the same |err| to ~1e-16, which is all an estimate needs
        double c = u - M;
        if (__double2hiint(u) != 0x43380000 + (r >> 31) || r < gr.lo || r > gr.hi) c = t < -ze ? -ze : mq - ze;
        ef = gr.lo > gr.hi ? 0.f : __double2float_rn(fma(c, sc, -w));
    } else {
        ef = __double2float_rn(w);
    }
    return ef * __fdividef(ef, __double2float_rn(dgv));
}

// Estimates of all own slots from the state arrays (NaN for dead or unused slots).
// N:M pattern: blkcnt (nullable) holds per block of 2^nm_lg original columns the number of weights eliminated so
// far; a slot whose block has reached nm_prune is no candidate (NaN estimate).  cntw receives the counts of the
// own slots' blocks, one byte per slot, which the update phase then keeps current in registers.
template <int NT, int KMAX, bool Q>
__device__ __forceinline__ void estimate_own(float (&sa)[KMAX], const double* wd, const double* dg, const int* perm,
                                             int m0, bool quant, double sc, double isc, double ze, double mq, const GridRange& gr,
                                             const unsigned char* blkcnt, int nm_lg, int nm_prune,
                                             unsigned (&cntw)[KMAX / 4]) {
#pragma unroll
    for (int g = 0; g < KMAX / 4; ++g) cntw[g] = 0u;
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        const int j = own_slot<NT>(k);
        sa[k] = CUDART_NAN_F;
        if (j < m0 && perm[j] >= 0) {
            unsigned c = 0u;
            if (blkcnt) { c = blkcnt[perm[j] >> nm_lg]; cntw[k >> 2] |= c << (8 * (k & 3)); }
            if (!blkcnt || (int)c < nm_prune) sa[k] = score_estimate<Q>(wd[j], dg[j], quant, sc, isc, ze, mq, gr);
        }
    }
}

// The thread's two smallest estimates and the slot of the first (-1: none); NaN estimates are no candidates.
template <int NT, int KMAX>
__device__ __forceinline__ void smallest_own(const float (&sa)[KMAX], float* m1, float* m2, int* slot) {
    float a = CUDART_INF_F, b = CUDART_INF_F;
    int ka = -1;
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        const bool lt = sa[k] < a;
        b = lt ? a : fminf(b, sa[k]);                                   // (fminf ignores NaN)
        a = lt ? sa[k] : a;
        ka = lt ? k : ka;
    }
    *m1 = a; *m2 = b; *slot = ka < 0 ? -1 : own_slot<NT>(ka);
}

// The thread's best live slot among its own by (score, original index), given the estimates: only the slots
// within 1e-4 of the thread's best estimate take the FP64 division, so the result (ties included) is the
// exact FP64 choice.  The candidates are first collected in a bit mask and then scored in one loop, so the
// exact scoring exists once in the code and the lanes of a warp take it together.
// With the outlier rule (Section 4, "Quantization Outliers") a slot whose error exceeds Delta/2 wins by
// largest error; such candidates get negative scores, below every regular one.
template <int NT, int KMAX, bool Q>
__device__ __forceinline__ void thread_best(const float (&sa)[KMAX], const double* wd, const double* dg,
                                            const int* perm, bool quant, bool outliers, double sc, double isc,
                                            double ze, double mq, unsigned* key, double* s_out, int* slot_out) {
    float smin = CUDART_INF_F;
#pragma unroll
    for (int k = 0; k < KMAX; ++k) smin = fminf(smin, sa[k]);           // fminf ignores NaN estimates
    const float thr = smin + NEAR * fabsf(smin);
    unsigned cand = 0u, valid = 0u;
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        if (sa[k] <= thr || sa[k] == smin) cand |= 1u << k;             // false for NaN estimates
        if (sa[k] == sa[k]) valid |= 1u << k;
    }
    double bs = CUDART_INF, oe = -1.0;
    int bo = 0x7fffffff, bslot = -1, oo = 0x7fffffff, oslot = -1;
    unsigned todo = (Q && outliers) ? valid : cand;
    while (todo) {
        const int k = __ffs(todo) - 1;
        todo &= todo - 1;
        const int j = own_slot<NT>(k);
        const double w = wd[j];
        double err = -w;
        if (Q && quant) err = grid_error(w, sc, isc, ze, mq);
        const int o = perm[j];
        if ((cand >> k) & 1u) {
            const double s = err * err / dg[j];
            if (key_less(s, o, bs, bo)) { bs = s; bo = o; bslot = j; }
        }
        if (Q && outliers) {
            const double a = fabs(err);
            if (a > 0.5 * sc && (a > oe || (a == oe && o < oo))) { oe = a; oo = o; oslot = j; }
        }
    }
    *key = KEY_NONE; *s_out = bs; *slot_out = bslot;
    if (bslot >= 0) *key = float_key(__double2float_rn(bs));
    if (Q && outliers && oslot >= 0) { *s_out = -oe; *slot_out = oslot; *key = float_key(__double2float_rn(-oe)); }
}

// The flush applies the nb pending vectors Z[b][.] (already in the new slot numbering) to the triangle and compacts it
// to m1 rows.  srcm[i] = old slot whose data new slot i takes (i itself unless i is a hole).  The triangle is far
// larger than L2 and touched once per flush, so it is loaded and stored with the evict-first hint and leaves L2 to
// the overflow part of the pending vectors.
// ---- flush on the tensor cores -----------------------------------------------------------------------------------
// The flush is a rank-nb update, H -= Z^T Z with nb <= 64: a dense contraction.  A warp takes tiles of 16 rows x
// 64 columns; the increment of a tile is formed by mma.sync m16n8k8 (TF32 inputs, FP32 accumulation over 8 pending
// vectors at a time, the partial sums added up in FP32 registers) with every FP32 operand split into two TF32 parts, z = hi + lo, and the three products
// hi*hi + hi*lo + lo*hi (the missing lo*lo term is below 2^-22 of each product, and the products of one update are
// about 1/d_col of the element they change).  The tile of H is fetched afterwards (a prefetch cursor has pulled it
// into L2); the increment is subtracted in FP32 -- one rounding of the matrix element per flush -- and stored.
// Register layout: lane (g, t) = (lane / 4, lane % 4) holds rows g and g + 8 and, of every 16-column group u, the
// four columns 16u + 4t .. + 3 (one 128-bit access per row and group).  The two 8-column MMA tiles of a group take
// its even and its odd columns: tile 2u, n = 2t + e  <->  column 16u + 4t + 2e;  tile 2u+1: that + 1.  Their B
// fragments (n = g) are then the adjacent pair 16u + 2g, + 1 of a pending vector: one 64-bit shared-memory load.
// The leading part is rounded to nearest (on the magnitude, ties away): truncation would leave every product short
// by a part of the same sign, a bias that adds up over the d_col updates of an element instead of averaging out.
__device__ __forceinline__ uint32_t tf32_rn(float x) { return (__float_as_uint(x) + 0x1000u) & 0xFFFFE000u; }
__device__ __forceinline__ void tf32_split(float x, uint32_t& hi, uint32_t& lo) {
    hi = tf32_rn(x);                                        // 11 significant bits
    // the difference is exact in FP32 and has either sign; the tensor core reads its leading 11 bits (truncation of
    // a part whose sign is random is no bias; rounding it too was measured and changes nothing)
    lo = __float_as_uint(x - __uint_as_float(hi));
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

// GP: pending vectors nbs .. nb - 1 are rows of G (global memory, stride gld: the overflow part, resident in L2).  Their
// row operands are copied once per row group into the warp's staging block zstage (16 floats per vector); their column
// operands are read from L2 in the fragment layout, 8 vectors at a time.
// first product of a chain: the accumulator operand is zero
__device__ __forceinline__ void mma_tf32_z(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
// two values at once: the integer part of the split per value, the subtraction as one packed FP32 instruction
__device__ __forceinline__ void tf32_split2(float2 x, uint32_t& hi0, uint32_t& hi1, uint32_t& lo0, uint32_t& lo1) {
    hi0 = tf32_rn(x.x); hi1 = tf32_rn(x.y);
    const float2 l = __ffma2_rn(make_float2(__uint_as_float(hi0), __uint_as_float(hi1)), make_float2(-1.f, -1.f), x);
    lo0 = __float_as_uint(l.x); lo1 = __float_as_uint(l.y);
}

// A tile of H (16 rows x 64 columns from c0; in L2 by now: the cursor passed it two tiles ago) minus the increment acc * unscale.
template <bool STREAM, bool WIDE>
__device__ __forceinline__ void blk_flush_store(float* __restrict__ Hp, int ldp, int c0, int ngroups, const int (&rr)[2], const bool (&in)[2],
                                                const int (&sr)[2], int t, const float (&acc)[8][4], float unscale,
                                                const unsigned short* srcm, const uint32_t* colmask) {
    // ---- the tile of H (in L2 by now: the cursor passed it two tiles ago), minus the increment -----------
    float4 hv[4][2];
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            hv[u][h] = make_float4(0.f, 0.f, 0.f, 0.f);
            const int j = c0 + (u << 4) + (t << 2);
            if (u < ngroups && in[h] && j <= rr[h]) {
                const float4* src = reinterpret_cast<const float4*>(Hp + tri_at<WIDE>(ldp, sr[h], j));
                hv[u][h] = STREAM ? __ldcs(src) : *src;
            }
        }
    // columns of this lane that are holes: their data sits in the mover's row
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (u < ngroups) {
            const int j = c0 + (u << 4) + (t << 2);
            const uint32_t my4 = (colmask[j >> 5] >> (j & 31)) & 0xFu;
            if (my4) {
#pragma unroll
                for (int comp = 0; comp < 4; ++comp) {
                    if (!((my4 >> comp) & 1u)) continue;
                    const int jj = j + comp;
                    const int sj = (int)srcm[jj];
#pragma unroll
                    for (int h = 0; h < 2; ++h) {
                        if (in[h] && jj <= rr[h]) {
                            const float val = Hp[tri_at<WIDE>(ldp, max(sr[h], sj), min(sr[h], sj))];
                            if (comp == 0) hv[u][h].x = val; else if (comp == 1) hv[u][h].y = val;
                            else if (comp == 2) hv[u][h].z = val; else hv[u][h].w = val;
                        }
                    }
                }
            }
        }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) {
        if (u < ngroups) {
            const int j = c0 + (u << 4) + (t << 2);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
                if (in[h] && j <= rr[h]) {
                    float4 o = hv[u][h];
                    o.x = fmaf(-unscale, acc[2 * u][2 * h], o.x);     o.z = fmaf(-unscale, acc[2 * u][2 * h + 1], o.z);
                    o.y = fmaf(-unscale, acc[2 * u + 1][2 * h], o.y); o.w = fmaf(-unscale, acc[2 * u + 1][2 * h + 1], o.w);
                    float4* dst = reinterpret_cast<float4*>(Hp + tri_at<WIDE>(ldp, rr[h], j));
                    if (STREAM) __stcs(dst, o); else *dst = o;
                }
            }
        }
    }
}

template <int NT, bool STREAM, bool GP, bool WIDE>
__device__ __forceinline__ void blk_flush_mma(float* __restrict__ Hp, int ldp, int m1, int nb, int nbs, const float* Z, int ldz,
                                              const float* __restrict__ G, int gld, float* zstage,
                                              const unsigned short* srcm, const uint32_t* colmask) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int nrg = (m1 + 15) >> 4;
    const int ksteps = ((GP ? nbs : nb) + 7) >> 3;
    const int nbg = GP ? nb - nbs : 0;
    const int ksteps_g = (nbg + 7) >> 3;
    // The products are cheap next to the latency of memory, and a warp has one tile (4 KB) in registers at a time:
    // a cursor runs FLUSH_AHEAD tiles ahead of the warp through its sequence of tiles and pulls them into L2
    // (measured at d_col = 2304: 12 % off the pass with a distance of 1 or 2 tiles, less with 4, a loss from 8 on).
    constexpr int FLUSH_AHEAD = 2;
    int prg = warp, pc0 = 0;
    auto prefetch_next = [&]() {
        if (prg >= nrg) return;
        // 16 rows x 2 lines of 128 bytes, or 16 column groups x 2 lines of 8 rows
        const int row = (prg << 4) + (WIDE ? lane >> 1 : (lane & 1) << 3), col = pc0 + (WIDE ? (lane & 1) << 5 : (lane >> 1) << 2);
        if (row < m1 && col <= row + (WIDE ? 0 : 7))
            asm volatile("prefetch.global.L2 [%0];" ::"l"(Hp + tri_at<WIDE>(ldp, srcm[row], col)));
        pc0 += 64;
        if (pc0 >= min((prg << 4) + 16, m1)) { pc0 = 0; prg += NW; }
    };
#pragma unroll
    for (int a = 0; a < FLUSH_AHEAD; ++a) prefetch_next();
    for (int rg = warp; rg < nrg; rg += NW) {
        const int i0 = rg << 4;
        const int jend = min(i0 + 16, m1);                     // columns [0, jend) hold data of this row group
        const int rr[2] = {i0 + g, i0 + g + 8};                // the lane's two rows
        const bool in[2] = {rr[0] < m1, rr[1] < m1};
        const int sr[2] = {in[0] ? (int)srcm[rr[0]] : 0, in[1] ? (int)srcm[rr[1]] : 0};
        if (GP && nbg > 0) {                                   // row operands of the overflow vectors -> staging block
            __syncwarp();
            for (int e = lane; e < nbg * 4; e += 32) {
                const int v = e >> 2, q = e & 3;
                *reinterpret_cast<float4*>(zstage + v * 16 + 4 * q) =
                    *reinterpret_cast<const float4*>(G + (size_t)v * gld + i0 + 4 * q);
            }
            __syncwarp();
        }
        for (int c0 = 0; c0 < jend; c0 += 64) {
            const int ngroups = min(4, (jend - c0 + 15) >> 4);
            prefetch_next();
            // ---- the tile's increment: sum over the pending vectors of z[row] * z[column] -------------------------
            float acc[8][4];
#pragma unroll
            for (int n = 0; n < 8; ++n) { acc[n][0] = 0.f; acc[n][1] = 0.f; acc[n][2] = 0.f; acc[n][3] = 0.f; }
            // one step: 8 pending vectors (this lane: vectors k0 = 8 ks + t and k0 + 4) times the tile's rows and columns
            auto kstep = [&](const float (&av)[4], const float2 (&b0)[4], const float2 (&b1)[4]) {
                uint32_t ah[4], al[4];
#pragma unroll
                for (int q = 0; q < 4; ++q) tf32_split(av[q], ah[q], al[q]);
                uint32_t bh[8][2], bl[8][2];                              // the 8 MMA tiles: (k0, k1) parts
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    tf32_split2(b0[u], bh[2 * u][0], bh[2 * u + 1][0], bl[2 * u][0], bl[2 * u + 1][0]);
                    tf32_split2(b1[u], bh[2 * u][1], bh[2 * u + 1][1], bl[2 * u][1], bl[2 * u + 1][1]);
                }
                // The tensor core rounds every result toward zero (measured: the products of one instruction are
                // summed with guard bits, then truncated to FP32).  On a running accumulator that is a bias of about
                // 2^-25 of the accumulator per instruction, of the same sign for all d_col / 8 instructions of an
                // element.  So the three products of 8 pending vectors are summed from zero, the two small ones
                // first -- one truncation at the size of that partial sum -- and the partial sums are added to the
                // running increment in FP32 with round-to-nearest.  A product into an accumulator is issued eight
                // products after the previous one into it: their latency is long.
                float dk[8][4];
#pragma unroll
                for (int n = 0; n < 8; ++n) mma_tf32_z(dk[n], al, bh[n][0], bh[n][1]);
#pragma unroll
                for (int n = 0; n < 8; ++n) mma_tf32(dk[n], ah, bl[n][0], bl[n][1]);
#pragma unroll
                for (int n = 0; n < 8; ++n) mma_tf32(dk[n], ah, bh[n][0], bh[n][1]);
                // That one truncation per partial sum still shortens every increment by half a unit in the last place on
                // average, the same way for every element and pass -- a uniform scaling of all Lemma-1 updates, which the
                // last steps of a row (the few remaining entries carry everything eliminated before) amplify: measured
                // on a 2304-column layer, the final loss was off by 1.7e-4 with it and 1.3e-5 without.  Setting the last
                // mantissa bit turns "truncated" into "truncated + 0 or 1 unit", which is right on average.
#pragma unroll
                for (int n = 0; n < 8; ++n)
#pragma unroll
                    for (int e = 0; e < 4; e += 2) {                     // (two additions per instruction)
                        const float2 r = __fadd2_rn(make_float2(acc[n][e], acc[n][e + 1]),
                                                    make_float2(__uint_as_float(__float_as_uint(dk[n][e]) | 1u),
                                                                __uint_as_float(__float_as_uint(dk[n][e + 1]) | 1u)));
                        acc[n][e] = r.x; acc[n][e + 1] = r.y;
                    }
            };
            // column operands of an overflow step, straight from L2; issued one step ahead of their use
            float2 pb0[4], pb1[4];
            auto load_g = [&](int kg) {
                const int k0 = (kg << 3) + t, k1 = k0 + 4;
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int c = c0 + (u << 4) + (g << 1);               // < round_up(m1, 16) <= gld
                    pb0[u] = make_float2(0.f, 0.f); pb1[u] = pb0[u];
                    if (u < ngroups && k0 < nbg) pb0[u] = *reinterpret_cast<const float2*>(G + (size_t)k0 * gld + c);
                    if (u < ngroups && k1 < nbg) pb1[u] = *reinterpret_cast<const float2*>(G + (size_t)k1 * gld + c);
                }
            };
            if (GP && ksteps_g > 0) load_g(0);                            // in flight during the shared-memory steps
            for (int ks = 0; ks < ksteps; ++ks) {
                const int k0 = (ks << 3) + t, k1 = k0 + 4;
                const bool v0 = k0 < (GP ? nbs : nb), v1 = k1 < (GP ? nbs : nb);
                const float* z0 = Z + (size_t)k0 * ldz;
                const float* z1 = Z + (size_t)k1 * ldz;
                const float av[4] = {v0 && in[0] ? z0[rr[0]] : 0.f, v0 && in[1] ? z0[rr[1]] : 0.f,
                                     v1 && in[0] ? z1[rr[0]] : 0.f, v1 && in[1] ? z1[rr[1]] : 0.f};
                float2 b0[4], b1[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    const int c = c0 + (u << 4) + (g << 1);               // < m1 + 16 <= ldz
                    b0[u] = make_float2(0.f, 0.f); b1[u] = b0[u];         // (a group past the end multiplies zeros)
                    if (u < ngroups && v0) b0[u] = *reinterpret_cast<const float2*>(z0 + c);
                    if (u < ngroups && v1) b1[u] = *reinterpret_cast<const float2*>(z1 + c);
                }
                kstep(av, b0, b1);
            }
            if (GP) for (int kg = 0; kg < ksteps_g; ++kg) {
                const int k0 = (kg << 3) + t, k1 = k0 + 4;
                const bool v0 = k0 < nbg, v1 = k1 < nbg;
                const float av[4] = {v0 ? zstage[k0 * 16 + g] : 0.f, v0 ? zstage[k0 * 16 + g + 8] : 0.f,      // (rows past m1
                                     v1 ? zstage[k1 * 16 + g] : 0.f, v1 ? zstage[k1 * 16 + g + 8] : 0.f};     // are never stored)
                float2 b0[4], b1[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) { b0[u] = pb0[u]; b1[u] = pb1[u]; }
                if (kg + 1 < ksteps_g) load_g(kg + 1);
                kstep(av, b0, b1);
            }
            blk_flush_store<STREAM, WIDE>(Hp, ldp, c0, ngroups, rr, in, sr, t, acc, 1.f, srcm, colmask);
        }
    }
}

// ---- a pass on tcgen05 (flush_tc.cuh): what the block prepares for it ----------------------------------------------------
// A triangle that TMA stores write is read past L1.
template <bool TC> __device__ __forceinline__ float ld_tri(const float* p) { return TC ? __ldcg(p) : *p; }
template <bool TC> __device__ __forceinline__ float4 ld_tri4(const float* p) {
    return TC ? __ldcg(reinterpret_cast<const float4*>(p)) : *reinterpret_cast<const float4*>(p);
}
template <int BYTES> __device__ __forceinline__ void copy_async(float* to, const float* from) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from), "n"(BYTES) : "memory");
}
__device__ __forceinline__ float pow2f(int e) { return __int_as_float((127 + e) << 23); }
// the power of two that takes v (> 0, finite) to [2^13, 2^14), within what a float power of two and its square hold
__device__ __forceinline__ int plane_power(float v) { return min(60, max(-50, 13 - ((int)(__float_as_uint(v) >> 23) - 127))); }

// The power of two that takes the pending vectors' largest entry to [2^13, 2^14), and whether the diagonal spans more than 2^24.
template <int NT, int KMAX>
__device__ __forceinline__ int blk_plane_range(const float* panel, int ldz, int scap, const float* G, int gld, int nb, int m0, int m1,
                                               const double* dg, const int* perm, float* rf, bool* wide) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    auto vec = [&](int b) { return b < scap ? panel + (size_t)b * ldz : G + (size_t)(b - scap) * gld; };
    float zmax = 0.f, dmax = 0.f, dmin = CUDART_INF_F;
#pragma unroll 2
    for (int b = 0; b < nb; ++b) {
        const float* z = vec(b);
#pragma unroll
        for (int g = 0; g < KMAX / 4; ++g) {
            const int jb = own_slot<NT>(4 * g);
            if (jb < m1) {
                const float4 v = *reinterpret_cast<const float4*>(z + jb);
                zmax = fmaxf(fmaxf(fmaxf(zmax, fabsf(v.x)), fmaxf(fabsf(v.y), fabsf(v.z))), fabsf(v.w));
            }
        }
    }
#pragma unroll
    for (int k = 0; k < KMAX; ++k) {
        const int j = own_slot<NT>(k);
        if (j < m0 && perm[j] >= 0) { const float x = fmaxf((float)dg[j], 0.f); dmax = fmaxf(dmax, x); dmin = fminf(dmin, x); }
    }
    zmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(zmax)));
    dmax = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(dmax)));
    dmin = __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(dmin)));
    if (lane == 0) { rf[warp] = zmax; rf[NW + warp] = dmax; rf[2 * NW + warp] = dmin; }
    __syncthreads();
#pragma unroll
    for (int w = 0; w < NW; ++w) { zmax = fmaxf(zmax, rf[w]); dmax = fmaxf(dmax, rf[NW + w]); dmin = fminf(dmin, rf[2 * NW + w]); }
    // the planes hold vectors of the diagonal before the pending eliminations: zmax^2 is what it had been (at least) where it has
    // collapsed since
    *wide = dmin < fmaxf(dmax, zmax * zmax) * 5.9604645e-8f;             // 2^-24
    return plane_power(zmax);
}

// The pending vectors (b < scap in shared memory, the rest in G), already in the new slot numbering, as FP16 planes hi, lo
// (64 rows each); rows nb .. of the last group of 16 become zero.  Returns the planes' power of two, or 99 where every slot has
// its own (zexp).  Every thread of the block calls it; the caller synchronises before the planes are read.
template <int NT, int KMAX>
__device__ __forceinline__ int blk_make_planes(const float* panel, int ldz, int scap, const float* G, int gld, int nb, int m0, int m1,
                                               const double* dg, const int* perm, float* rf, __half* planes, int zld, signed char* zexp) {
    auto vec = [&](int b) { return b < scap ? panel + (size_t)b * ldz : G + (size_t)(b - scap) * gld; };
    bool wide;
    const int power = blk_plane_range<NT, KMAX>(panel, ldz, scap, G, gld, nb, m0, m1, dg, perm, rf, &wide);
    const int nb16 = (nb + 15) & ~15;
#pragma unroll
    for (int g = 0; g < KMAX / 4; ++g) {
        const int jb = own_slot<NT>(4 * g);
        if (jb >= m1) continue;
        float sc[4] = {pow2f(power), pow2f(power), pow2f(power), pow2f(power)};
        if (wide) {
            float mx[4] = {0.f, 0.f, 0.f, 0.f};
            for (int b = 0; b < nb; ++b) {
                const float4 v = *reinterpret_cast<const float4*>(vec(b) + jb);
                mx[0] = fmaxf(mx[0], fabsf(v.x)); mx[1] = fmaxf(mx[1], fabsf(v.y)); mx[2] = fmaxf(mx[2], fabsf(v.z)); mx[3] = fmaxf(mx[3], fabsf(v.w));
            }
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int e = plane_power(mx[q]);
                sc[q] = pow2f(e);
                zexp[jb + q] = (signed char)e;
            }
        }
        __half* p = planes + jb;
#pragma unroll 4
        for (int b = 0; b < nb16; ++b) {
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (b < nb) v = *reinterpret_cast<const float4*>(vec(b) + jb);
            v.x *= sc[0]; v.y *= sc[1]; v.z *= sc[2]; v.w *= sc[3];
            const __half2 h0 = __floats2half2_rn(v.x, v.y), h1 = __floats2half2_rn(v.z, v.w);
            const float2 f0 = __half22float2(h0), f1 = __half22float2(h1);
            const __half2 l0 = __floats2half2_rn(v.x - f0.x, v.y - f0.y), l1 = __floats2half2_rn(v.z - f1.x, v.w - f1.y);
            *reinterpret_cast<uint2*>(p + (size_t)b * zld) =
                make_uint2(*reinterpret_cast<const unsigned*>(&h0), *reinterpret_cast<const unsigned*>(&h1));
            *reinterpret_cast<uint2*>(p + (size_t)(64 + b) * zld) =
                make_uint2(*reinterpret_cast<const unsigned*>(&l0), *reinterpret_cast<const unsigned*>(&l1));
        }
    }
    return wide ? 99 : power;
}

// The same planes in the vectors' own place in shared memory, for the flush by mma.sync: rows 2b and 2b + 1 become the hi and the lo
// halves of vectors 2b and 2b + 1, two FP16 to a word (a fragment register of m16n8k16).  Row nb is there when nb is odd.
template <int NT, int KMAX>
__device__ __forceinline__ void blk_pack_planes(float* panel, int ldz, int nb, int m1, float scale) {
#pragma unroll
    for (int g = 0; g < KMAX / 4; ++g) {
        const int jb = own_slot<NT>(4 * g);
        if (jb >= m1) continue;
#pragma unroll 4
        for (int b = 0; b < nb; b += 2) {
            float* z = panel + (size_t)b * ldz + jb;
            const float4 u = *reinterpret_cast<const float4*>(z);
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (b + 1 < nb) v = *reinterpret_cast<const float4*>(z + ldz);
            const float x0[4] = {u.x * scale, u.y * scale, u.z * scale, u.w * scale}, x1[4] = {v.x * scale, v.y * scale, v.z * scale, v.w * scale};
            unsigned hi[4], lo[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const __half2 h = __floats2half2_rn(x0[q], x1[q]);
                const float2 f = __half22float2(h);
                const __half2 l = __floats2half2_rn(x0[q] - f.x, x1[q] - f.y);
                hi[q] = *reinterpret_cast<const unsigned*>(&h); lo[q] = *reinterpret_cast<const unsigned*>(&l);
            }
            *reinterpret_cast<uint4*>(z) = make_uint4(hi[0], hi[1], hi[2], hi[3]);
            *reinterpret_cast<uint4*>(z + ldz) = make_uint4(lo[0], lo[1], lo[2], lo[3]);
        }
    }
}

__device__ __forceinline__ void mma_f16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_f16_z(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
        : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3]) : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}

// The flush by mma.sync on packed planes (blk_pack_planes): tiles, register layout, compaction and the treatment of the partial sums as
// in blk_flush_mma, with m16n8k16 on FP16 planes instead of m16n8k8 on TF32 parts: half the products per vector, and the operands
// are split once per flush instead of in every tile (3072 x 768 replay and OBQ 82.7 -> 75.7 ms, 768 x 768 2:4 8.06 -> 7.41).  Partial sums are
// over 16 vectors, scaled by `unscale` = 2^-2e of the planes.  What bounds it is the latency of a warp's one tile in flight: read, products,
// subtraction, store.  Rows whose diagonal is too wide for a common power of two, and rows with overflow vectors (blocks of 8),
// take the TF32 form.
template <int NT, bool WIDE>
__device__ __forceinline__ void blk_flush_f16(float* __restrict__ Hp, int ldp, int m1, int nb, const float* Z, int ldz, float unscale,
                                              const unsigned short* srcm, const uint32_t* colmask) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    const int nrg = (m1 + 15) >> 4;
    const int pairs = (nb + 1) >> 1, ksteps = (pairs + 7) >> 3;
    const uint32_t* W = reinterpret_cast<const uint32_t*>(Z);
    constexpr int FLUSH_AHEAD = 2;                             // as in blk_flush_mma
    int prg = warp, pc0 = 0;
    auto prefetch_next = [&]() {
        if (prg >= nrg) return;
        // 16 rows x 2 lines of 128 bytes, or 16 column groups x 2 lines of 8 rows
        const int row = (prg << 4) + (WIDE ? lane >> 1 : (lane & 1) << 3), col = pc0 + (WIDE ? (lane & 1) << 5 : (lane >> 1) << 2);
        if (row < m1 && col <= row + (WIDE ? 0 : 7))
            asm volatile("prefetch.global.L2 [%0];" ::"l"(Hp + tri_at<WIDE>(ldp, srcm[row], col)));
        pc0 += 64;
        if (pc0 >= min((prg << 4) + 16, m1)) { pc0 = 0; prg += NW; }
    };
#pragma unroll
    for (int a = 0; a < FLUSH_AHEAD; ++a) prefetch_next();
    for (int rg = warp; rg < nrg; rg += NW) {
        const int i0 = rg << 4;
        const int jend = min(i0 + 16, m1);                     // columns [0, jend) hold data of this row group
        const int rr[2] = {i0 + g, i0 + g + 8};                // the lane's two rows
        const bool in[2] = {rr[0] < m1, rr[1] < m1};
        const int sr[2] = {in[0] ? (int)srcm[rr[0]] : 0, in[1] ? (int)srcm[rr[1]] : 0};
        for (int c0 = 0; c0 < jend; c0 += 64) {
            const int ngroups = min(4, (jend - c0 + 15) >> 4);
            prefetch_next();
            float acc[8][4];
#pragma unroll
            for (int n = 0; n < 8; ++n) { acc[n][0] = 0.f; acc[n][1] = 0.f; acc[n][2] = 0.f; acc[n][3] = 0.f; }
            for (int ks = 0; ks < ksteps; ++ks) {
                // this lane: pairs 8 ks + t and + 4; past the last pair zeros
                const int p0 = (ks << 3) + t, p1 = p0 + 4;
                const bool v0 = p0 < pairs, v1 = p1 < pairs;
                const uint32_t* z0 = W + (size_t)(2 * p0) * ldz;
                const uint32_t* z1 = W + (size_t)(2 * p1) * ldz;
                uint32_t ah[4], al[4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    ah[h] = v0 && in[h] ? z0[rr[h]] : 0u;     al[h] = v0 && in[h] ? z0[ldz + rr[h]] : 0u;
                    ah[2 + h] = v1 && in[h] ? z1[rr[h]] : 0u; al[2 + h] = v1 && in[h] ? z1[ldz + rr[h]] : 0u;
                }
#pragma unroll
                for (int half = 0; half < 2; ++half) {         // two column groups at a time
                    if (2 * half >= ngroups) break;
                    uint2 bh0[2], bl0[2], bh1[2], bl1[2];
#pragma unroll
                    for (int x = 0; x < 2; ++x) {
                        const int u = 2 * half + x, c = c0 + (u << 4) + (g << 1);      // < m1 + 16 <= ldz
                        bh0[x] = bl0[x] = bh1[x] = bl1[x] = make_uint2(0u, 0u);
                        if (u < ngroups && v0) { bh0[x] = *reinterpret_cast<const uint2*>(z0 + c); bl0[x] = *reinterpret_cast<const uint2*>(z0 + ldz + c); }
                        if (u < ngroups && v1) { bh1[x] = *reinterpret_cast<const uint2*>(z1 + c); bl1[x] = *reinterpret_cast<const uint2*>(z1 + ldz + c); }
                    }
                    float dk[4][4];
#pragma unroll
                    for (int x = 0; x < 2; ++x) { mma_f16_z(dk[2 * x], al, bh0[x].x, bh1[x].x); mma_f16_z(dk[2 * x + 1], al, bh0[x].y, bh1[x].y); }
#pragma unroll
                    for (int x = 0; x < 2; ++x) { mma_f16(dk[2 * x], ah, bl0[x].x, bl1[x].x); mma_f16(dk[2 * x + 1], ah, bl0[x].y, bl1[x].y); }
#pragma unroll
                    for (int x = 0; x < 2; ++x) { mma_f16(dk[2 * x], ah, bh0[x].x, bh1[x].x); mma_f16(dk[2 * x + 1], ah, bh0[x].y, bh1[x].y); }
#pragma unroll
                    for (int n = 0; n < 4; ++n)
#pragma unroll
                        for (int e = 0; e < 4; e += 2) {
                            const float2 r = __fadd2_rn(make_float2(acc[4 * half + n][e], acc[4 * half + n][e + 1]),
                                                        make_float2(__uint_as_float(__float_as_uint(dk[n][e]) | 1u),
                                                                    __uint_as_float(__float_as_uint(dk[n][e + 1]) | 1u)));
                            acc[4 * half + n][e] = r.x; acc[4 * half + n][e + 1] = r.y;
                        }
                }
            }
            blk_flush_store<true, WIDE>(Hp, ldp, c0, ngroups, rr, in, sr, t, acc, unscale, srcm, colmask);
        }
    }
}

// The triangle's part of the compaction: the movers' rows and columns into the holes.  They come from rows >= m1, which
// nothing here writes.  srcm[j] = old slot whose data new slot j takes.
template <int NT>
__device__ __forceinline__ void blk_fill_holes(float* H, int ldp, int m1, int nh, const int* hl, const int* mv, const unsigned short* srcm) {
    for (int j = threadIdx.x; j < m1; j += NT) {
        const int sj = srcm[j];
        for (int q0 = 0; q0 < nh; q0 += 16) {                  // sixteen loads in flight per thread
            float v[16];
#pragma unroll
            for (int q = 0; q < 16; ++q)
                if (q0 + q < nh) { const int sh = mv[q0 + q]; v[q] = __ldcg(H + tri_at<true>(ldp, max(sh, sj), min(sh, sj))); }
#pragma unroll
            for (int q = 0; q < 16; ++q)
                if (q0 + q < nh) { const int h = hl[q0 + q]; H[tri_at<true>(ldp, max(h, j), min(h, j))] = v[q]; }
        }
    }
}

// The deferred updates of the on-chip triangle S (m slots): S[i][j] -= sum_b v_b[i] u_b[j].  A warp takes 8 rows and 32 columns at a
// time; rows of eliminated slots are left out.
template <int NT>
__device__ __forceinline__ void tail_flush(float* S, int m, const float* vt, const float* ut, const int* perm) {
    constexpr int NW = NT / 32;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    for (int i0 = 8 * warp; i0 < m; i0 += 8 * NW)
        for (int c0 = 0; c0 < min(i0 + 8, m); c0 += 32) {
            const int j = c0 + lane;
            const float4* uj = reinterpret_cast<const float4*>(ut + min(j, m - 1) * TAIL_LD);
            const float4 u0 = uj[0], u1 = uj[1];
#pragma unroll 4
            for (int i = i0; i < min(i0 + 8, m); ++i) {
                if (perm[i] < 0) continue;
                const float4* vi = reinterpret_cast<const float4*>(vt + i * TAIL_LD);
                const float4 v0 = vi[0], v1 = vi[1];
                if (j <= i) {
                    float x = v0.x * u0.x;
                    x = fmaf(v0.y, u0.y, x); x = fmaf(v0.z, u0.z, x); x = fmaf(v0.w, u0.w, x);
                    x = fmaf(v1.x, u1.x, x); x = fmaf(v1.y, u1.y, x); x = fmaf(v1.z, u1.z, x); x = fmaf(v1.w, u1.w, x);
                    S[tail_at(i, j)] -= x;
                }
            }
        }
}

// Block pruning (Section 3, "Block-Sparsity", Eq. 5), blocks of 4: score w_P^T ((Hinv)_P)^-1 w_P of one 4-slot group
// from its weights w, the diagonal a_ii and the off-diagonals o = (a01, a02, a03, a12, a13, a23) of its 4 x 4 block, by
// an LDL^T factorisation: the score is sum_i y_i^2 / d_i, which is also the sum of the four single-weight losses
// when the members are eliminated in this order.  Returns NaN if the block is not positive definite.
__device__ __forceinline__ double block4_score(const double* w, const double* a, const double* o) {
    const double d0 = a[0], r0 = 1.0 / d0;
    const double l10 = o[0] * r0, l20 = o[1] * r0, l30 = o[2] * r0;
    const double d1 = a[1] - l10 * o[0], r1 = 1.0 / d1;
    const double t21 = o[3] - l20 * o[0], t31 = o[4] - l30 * o[0];
    const double l21 = t21 * r1, l31 = t31 * r1;
    const double d2 = a[2] - l20 * o[1] - l21 * t21, r2 = 1.0 / d2;
    const double t32 = o[5] - l30 * o[1] - l31 * t21;
    const double l32 = t32 * r2;
    const double d3 = a[3] - l30 * o[2] - l31 * t31 - l32 * t32, r3 = 1.0 / d3;
    const double y0 = w[0];
    const double y1 = w[1] - l10 * y0;
    const double y2 = w[2] - l20 * y0 - l21 * y1;
    const double y3 = w[3] - l30 * y0 - l31 * y1 - l32 * y2;
    if (!(d0 > 0.0) || !(d1 > 0.0) || !(d2 > 0.0) || !(d3 > 0.0)) return CUDART_NAN;
    return y0 * y0 * r0 + y1 * y1 * r1 + y2 * y2 * r2 + y3 * y3 * r3;
}

// Blocks of 8: the same score by Gaussian elimination of the members in ascending order on a copy of the 8 x 8 block
// (diagonal a, off-diagonals o packed by rows of the upper triangle: (0,1) .. (0,7), (1,2) .. (6,7)): the sum of the
// eight single-weight losses w_i^2 / a_ii met on the way.  Returns NaN if a pivot is not positive.
__device__ __forceinline__ int block8_index(int i, int j) { return i * (15 - i) / 2 + (j - i - 1); }      // i < j
static __device__ __noinline__ double block8_score(const double* w, const double* a, const double* o) {
    double m[8][8], y[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        y[i] = w[i]; m[i][i] = a[i];
#pragma unroll
        for (int j = i + 1; j < 8; ++j) m[i][j] = o[block8_index(i, j)];
    }
    double sc = 0.0;
    bool ok = true;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const double dii = m[i][i], r = 1.0 / dii;
        ok = ok && (dii > 0.0);
        sc += y[i] * y[i] * r;
#pragma unroll
        for (int j = i + 1; j < 8; ++j) {
            const double l = m[i][j] * r;
            y[j] -= l * y[i];
#pragma unroll
            for (int k = j; k < 8; ++k) m[j][k] -= l * m[i][k];
        }
    }
    return ok ? sc : CUDART_NAN;
}

// Q = the kernel contains the OBQ code (modes QUANT and REPLAY_QUANT); the pruning kernels are built without it.
// BC = 4 or 8: block pruning in blocks of that many consecutive columns (pruning kernels only), 0: single weights.
// FG = the kernel takes forced eliminations (replay of a known order) four at a time: their order is known, so the
// four pivot columns are fetched and corrected together, the 4 x 4 block of the columns at the pivot slots is
// broadcast, and every thread carries out the four Lemma-1 eliminations on its own slots in registers -- two
// barriers per four steps, each pending vector read once for four columns.  Same arithmetic per element as four
// single steps, but for the order in which the four members' own corrections are added.
// Block pruning in blocks of 4 does the same with the four members of the block it has picked (BG).
// NM = N:M pruning; the other kernels are built without that code.
// GPV = the kernel can keep further pending vectors in global memory (long rows, 512 threads only).
// SH = the kernel takes shares of rows (a row may be started by one block and finished by the next); launches whose
// rows divide evenly over the blocks run the kernel built without that code.
// Passes on tcgen05: one block per SM (blocks of 8 keep 28 bytes more per slot and may lack the room for its tiles).  Only
// those kernels take the tensor maps.
template <int NT, int BC> constexpr bool blk_tc = NT >= 512 && BC != 8;
struct NoMaps {};
template <int NT, int BC> using BlkMaps = std::conditional_t<blk_tc<NT, BC>, FlushMaps, NoMaps>;

template <int NT, int KMAX, bool Q, int BC, bool FG, bool GPV, bool SH, bool NM>
__global__ void __launch_bounds__(NT, 512 / NT) blocked_engine_kernel(const __grid_constant__ BlkMaps<NT, BC> zmaps,
                                                                      const __grid_constant__ EngineArgs a) {
    extern __shared__ __align__(16) char smem[];
    constexpr int NW = NT / 32;
    constexpr int BCD = BC ? BC : 1;                           // divisor that is never zero
    constexpr bool TC = blk_tc<NT, BC>, WIDE = NT >= 512;      // (WIDE: the triangle in groups of 32 columns)
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int d = a.d, cap = a.cap, ms = a.ms;
    char* scratch = smem;
    Bcast* bc = reinterpret_cast<Bcast*>(smem + BLK_OFF_BC);
    int* pv = reinterpret_cast<int*>(smem + BLK_OFF_PV);
    int* hl = reinterpret_cast<int*>(smem + BLK_OFF_HL);
    int* mv = reinterpret_cast<int*>(smem + BLK_OFF_MV);
    float* rf = reinterpret_cast<float*>(smem + BLK_OFF_RF);
    uint32_t* colmask = reinterpret_cast<uint32_t*>(smem + BLK_OFF_CM);
    // wd and dg (FP64) come first or, with passes on tcgen05, last (blk_state_bytes)
    double* wd = reinterpret_cast<double*>(smem + BLK_FIXED);
    double* dg = wd + cap;
    int* perm = TC ? reinterpret_cast<int*>(smem + BLK_FIXED) : reinterpret_cast<int*>(dg + cap);
    const int before_state = TC ? 16 * cap : 0;
    unsigned short* srcm = reinterpret_cast<unsigned short*>(perm + cap);
    const bool has_wfull = a.w_trace != nullptr;
    float* wfull = reinterpret_cast<float*>(smem + BLK_FIXED + blk_state_bytes(cap, false) - before_state);
    // N:M pattern: at most nm_prune eliminations per block.  (Decided at run time in the replay kernels too, where it is always
    // false: compiled without that code they are 2 - 4 % slower, 16 x 1536 4.18 -> 4.30 ms.)
    const bool has_nm = (NM || (FG && !Q)) && a.nm_prune > 0;
    const int nm_lg = a.nm_lg, nm_prune = a.nm_prune;
    unsigned char* blkcnt = reinterpret_cast<unsigned char*>(smem + BLK_FIXED + blk_state_bytes(cap, has_wfull) - before_state);
    double* boff = reinterpret_cast<double*>(smem + BLK_FIXED + blk_state_bytes(cap, has_wfull, has_nm) - before_state);
    float* panel = reinterpret_cast<float*>(smem + BLK_FIXED + blk_state_bytes(cap, has_wfull, has_nm, BC));
    if (TC) { wd = reinterpret_cast<double*>(panel) - 2 * cap; dg = wd + cap; }
    // tail views (the end of a row in shared memory) share the panel's space
    float* vt = panel;
    float* ut = vt + TAIL_LD * ms;
    float* S = ut + TAIL_LD * ms;
    const int ldp = a.ldp;
    float* const Hp0 = a.Hws ? a.Hws + (size_t)blockIdx.x * tri_floats(cap) : nullptr;      // the block's own triangle
#define HP (SH ? *reinterpret_cast<float**>(smem + BLK_OFF_SCHED + 16) : Hp0)
    // overflow of the pending vectors: gB more of them in global memory (sized to stay in L2), stride gld
    // (only the one-row-per-SM configuration uses it; the other kernels are built without that code)
    constexpr bool GP = GPV;
    constexpr bool BG = BC == 4 && KMAX == 4;                  // (the kernels with more slots per thread have no registers for it)
    enum { COLS_REGS, COLS_SMEM, COLS_SUBTRACT };              // where the columns of four eliminations wait for their corrections
    constexpr int COLS = KMAX == 4 ? COLS_REGS : (TC ? COLS_SUBTRACT : COLS_SMEM);
    const int gB = (GP && a.Gpan) ? a.g_vectors : 0, gld = a.g_ld;
    // (recomputed at every use instead of held in registers: the kernels with the overflow code have none to spare)
#define GVEC (a.Gpan + (size_t)blockIdx.x * a.g_vectors * a.g_ld)
#define ZSTAGE (panel + a.panel_floats + (size_t)warp * a.g_vectors * 16)      /* per warp: g_vectors x 16 floats */

    FlushBars* fb = reinterpret_cast<FlushBars*>(smem + BLK_OFF_FB);
    if (TC && d > ms) ft_alloc(fb);

    // ---- this block's items: whole rows, plus (shares of rows) the start of one row and the rest of another -------
    int* sched = reinterpret_cast<int*>(smem + BLK_OFF_SCHED);
    if (SH) {                                  // the item counter lives in shared memory too
        if (tid == 0) sched[3] = 0;
        __syncthreads();
    }
    for (int it_reg = 0;; ++it_reg) {
        int rr, kind, head_num;
        const int it = SH ? sched[3] : it_reg;
        if (SH) { __syncthreads(); if (tid == 0) sched[3] = it + 1; __syncthreads(); }    // read by all, then moved on
        if (!blk_item(SH, blockIdx.x, gridDim.x, a.row_count, it, &rr, &kind, &head_num)) break;
        const int NG = gridDim.x;
        const int r = a.row_begin + rr;
        // the triangle of the row in work: buffer blk for whole rows, ng + blk for the row this block starts, ng + blk - 1
        // for the row it finishes (kept in shared memory and re-read where needed, not in registers)
        int hbuf = kind == ITEM_FULL ? (int)blockIdx.x : (kind == ITEM_HEAD ? NG + (int)blockIdx.x : NG + (int)blockIdx.x - 1);
        int n_forced = 0, n_free = 0;
        bool quant = false;
        if (a.mode == MODE_PRUNE) { n_free = a.steps; }
        else if (a.mode == MODE_REPLAY) { n_forced = a.forced_counts[r]; }
        else if (a.mode == MODE_QUANT) { n_free = d; quant = Q; }
        else { n_forced = a.forced_counts[r]; n_free = d - n_forced; quant = Q; }
        if (n_forced < 0) n_forced = 0;
        if (n_forced > d) n_forced = d;
        if (n_free > d - n_forced) n_free = d - n_forced;
        const int total = n_forced + n_free;
        const bool outliers = Q && quant && (a.flags & OBC_FLAG_OUTLIERS);

        // ---- shares of rows: where this item stops, and what a continued row starts from -----------------
        int s_stop = total;                // steps [s_begin, s_stop) of the row are this item's
        int s_begin = 0, m_begin = d;
        if (kind == ITEM_HEAD) s_stop = blk_cut_step(d, ms, total, a.panel_floats, a.max_pending, gB, !(GP || TC), head_num, NG, blk_step_cost(NT));
        if (kind == ITEM_HEAD && s_stop <= 0) {
            // too small a share to be worth a start: the neighbour takes the whole row
            if (tid == 0) blk_publish(a.split_state + (size_t)blockIdx.x * a.split_stride, a.split_flags + blockIdx.x, 0, d, 0);
            continue;
        }
        if (kind == ITEM_TAIL) {
            const SplitHeader* sh = reinterpret_cast<const SplitHeader*>(a.split_state + (size_t)(blockIdx.x - 1) * a.split_stride);
            if (tid == 0) bc->nh = blk_wait_flag(a.split_flags + blockIdx.x - 1);
            __syncthreads();
            const int ok = bc->nh;
            __syncthreads();
            if (!ok) {                     // the start of this row never arrived: report it, touch nothing else
                if (tid == 0) a.row_status[r] = -(int)OBC_ERR_TIMEOUT;
                continue;
            }
            if (sh->done) continue;        // finished (or failed and reported) by the block that started it
            s_begin = sh->s_cut; m_begin = sh->m0;
            if (s_begin == 0) { kind = ITEM_FULL; hbuf = (int)blockIdx.x; }    // never started: a whole row
        }

        if (SH) {                              // read during and after the row
            if (tid == 0) {
                sched[0] = kind; sched[1] = s_stop; sched[2] = hbuf;
                *reinterpret_cast<float**>(smem + BLK_OFF_SCHED + 16) = a.Hws + (size_t)hbuf * tri_floats(cap);
            }
            __syncthreads();
        }

        // ---- row set-up ------------------------------------------------------------------------------
        if (kind == ITEM_TAIL) {
            // continue a row: state as saved at the flush boundary s_begin (slots [0, m_begin) all live, nothing pending)
            blk_state_copy(false, a.split_state + (size_t)(blockIdx.x - 1) * a.split_stride, cap, d, m_begin, NT, wd, dg, perm, srcm,
                           has_wfull ? wfull : nullptr);
            for (int k = tid; k < 160; k += NT) colmask[k] = 0u;
            if (tid == 0) {
                bc->sc = 1.0; bc->ze = 0.0; bc->mq = 0.0;
                if (a.mode == MODE_QUANT || (a.mode == MODE_REPLAY_QUANT && s_begin > n_forced)) {
                    bc->sc = (double)a.scale[r]; bc->ze = (double)a.zero[r];
                    bc->mq = (double)grid_maxq(a.bits, a.symmetric);
                }
            }
        } else {
            for (int j = tid; j < d; j += NT) {
                const float w = a.W[(size_t)r * a.ldw + j];
                wd[j] = (double)w;
                dg[j] = (double)a.Hinv[(size_t)j * a.ldhi + j];
                perm[j] = j;
                srcm[j] = (unsigned short)j;
                if (has_wfull) wfull[j] = w;
                if (a.codes) a.codes[(size_t)r * d + j] = -1;
                if (a.mask) a.mask[(size_t)r * d + j] = 1;
            }
            if (has_nm) for (int b = tid; b < (d >> nm_lg); b += NT) blkcnt[b] = 0;
            if (BC == 8) {
                for (int e = tid; e < (d >> 3) * 28; e += NT) {
                    const int g = e / 28, k = e - g * 28;
                    int ia = 0, rest = k;
                    while (rest >= 7 - ia) { rest -= 7 - ia; ++ia; }
                    const int ib = ia + 1 + rest;
                    boff[e] = (double)a.Hinv[(size_t)(8 * g + ia) * a.ldhi + 8 * g + ib];
                }
            } else if (BC) {
                for (int e = tid; e < (d >> 2) * 6; e += NT) {
                    const int g = e / 6, k = e - g * 6;
                    const int ia = k < 3 ? 0 : (k < 5 ? 1 : 2), ib = k < 3 ? k + 1 : (k < 5 ? k - 1 : 3);
                    boff[e] = (double)a.Hinv[(size_t)(4 * g + ia) * a.ldhi + 4 * g + ib];
                }
            }
            for (int k = tid; k < 160; k += NT) colmask[k] = 0u;
            for (int j = d + tid; j < cap; j += NT) perm[j] = -1;
            if (tid == 0) {
                bc->sc = 1.0; bc->ze = 0.0; bc->mq = 0.0;
                if (a.mode == MODE_QUANT) {
                    bc->sc = (double)a.scale[r]; bc->ze = (double)a.zero[r];
                    bc->mq = (double)grid_maxq(a.bits, a.symmetric);
                }
                a.row_status[r] = first_status(a, r);
            }
            if (a.w_trace)
                for (int j = tid; j < d; j += NT)
                    a.w_trace[((size_t)r * (a.trace_steps + 1)) * d + j] = a.W[(size_t)r * a.ldw + j];
        }
        if (kind != ITEM_TAIL && d > ms && total > 0) {
            if constexpr (!WIDE) {
                // a warp takes 8 rows, 4 lanes a row: 64 contiguous bytes read of each, 128 written to each of 4 column groups
                for (int i0 = 8 * warp; i0 < d; i0 += 8 * NW) {
                    const int i = i0 + (lane >> 2);
                    const float4* s4 = reinterpret_cast<const float4*>(a.Hinv + (size_t)i * a.ldhi);
                    float* dst = HP;
                    const int n4 = i < d ? (i >> 2) + 1 : 0;
                    for (int j0 = lane & 3; j0 < n4; j0 += 16) {       // four loads in flight per lane
                        float4 t[4];
#pragma unroll
                        for (int k = 0; k < 4; ++k) if (j0 + 4 * k < n4) t[k] = __ldg(s4 + j0 + 4 * k);
#pragma unroll
                        for (int k = 0; k < 4; ++k) if (j0 + 4 * k < n4) *reinterpret_cast<float4*>(dst + tri_at<WIDE>(ldp, i, 4 * (j0 + 4 * k))) = t[k];
                    }
                }
            } else {
                for (int i = warp; i < d; i += NW) {
                    const float4* s4 = reinterpret_cast<const float4*>(a.Hinv + (size_t)i * a.ldhi);
                    float* dst = HP;
                    auto put = [&](int j4, float4 v) { *reinterpret_cast<float4*>(dst + tri_at<WIDE>(ldp, i, 4 * j4)) = v; };
                    const int n4 = (i >> 2) + 1;
                    if (GP || FG) {                 // (kernels with no registers to spare: one load in flight)
                        for (int j4 = lane; j4 < n4; j4 += 32) put(j4, s4[j4]);
                    } else {
                        for (int j0 = lane; j0 < n4; j0 += 128) {      // four loads in flight per lane
                            float4 t[4];
#pragma unroll
                            for (int k = 0; k < 4; ++k) if (j0 + 32 * k < n4) t[k] = __ldg(s4 + j0 + 32 * k);
#pragma unroll
                            for (int k = 0; k < 4; ++k) if (j0 + 32 * k < n4) put(j0 + 32 * k, t[k]);
                        }
                    }
                }
            }
        }
        __syncthreads();
        double gsc = bc->sc, gze = bc->ze, gmq = bc->mq;       // grid parameters of the row (registers)
        GridRange gr = grid_range(gsc, gze, gmq);

        int m0 = m_begin;                // slots in use (tail phase: number of live slots)
        int nb = 0;                      // pending vectors
        int ldz = blk_ldz(m0);
        int scap = a.panel_floats / ldz;     // pending vectors that fit into shared memory at this row length
        int bcur = blk_updates(m0, a.panel_floats, a.max_pending, gB, !(GP || TC));
        if (BC) bcur &= ~(BC - 1);           // whole blocks between two flushes, so that 4-slot groups stay together
        int s = s_begin;
        bool failed = false, timed_out = false;
        int blk_base = 0, blk_orig = 0;  // block pruning: first slot, its column and the score of the block being eliminated
        double blk_score = 0.0;
        float sa[KMAX];                  // score estimates of the own slots, kept up to date by the update phase
        unsigned cntw[KMAX / 4];         // N:M: eliminations so far in the block of each own slot (one byte per slot)
#pragma unroll
        for (int g = 0; g < KMAX / 4; ++g) cntw[g] = 0u;
        bool sa_valid = false;
        unsigned alive = 0u;             // own slots that are live
        bool alive_valid = false;
        double gisc = 1.0 / gsc;
        // The block of columns to go next (block pruning).
        auto pick_block = [&](const Records& rec) {
            // block boundary: exact FP64 score of every own live group (its four slots are all live here)
            if (BC == 8) __syncwarp();       // the second half's state and some off-diagonals were written by the neighbouring lane
            double bs = CUDART_INF;
            int bo = 0x7fffffff, cslot = -1;
#pragma unroll
            for (int g = 0; g < KMAX / 4; ++g) {
                const int jb = own_slot<NT>(4 * g);
                if (BC == 8 && (jb & 7) != 0) continue;      // a block of 8 is scored by the owner of its first half
                if (jb < m0 && perm[jb] >= 0) {
                    const double sc4 = BC == 8 ? block8_score(wd + jb, dg + jb, boff + (jb >> 3) * 28)
                                               : block4_score(wd + jb, dg + jb, boff + (jb >> 2) * 6);
                    const int o = perm[jb];
                    if (key_less(sc4, o, bs, bo)) { bs = sc4; bo = o; cslot = jb; }
                }
            }
            const Pick pk = block_pick<NT>(cslot >= 0 ? float_key(__double2float_rn(bs)) : KEY_NONE, bs, cslot, cslot >= 0 ? perm[cslot] : -1, rec);
            blk_base = pk.slot; blk_orig = pk.orig; blk_score = pk.s;
            return pk;
        };
        // (every thread: the smallest and largest weight of its survivors)
        auto survivors_grid = [&](float lo, float hi) {
#pragma unroll
            for (int off = 16; off; off >>= 1) {
                lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, off));
                hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, off));
            }
            if (lane == 0) { rf[warp] = lo; rf[32 + warp] = hi; }
            __syncthreads();
            for (int k = 0; k < NW; ++k) { lo = fminf(lo, rf[k]); hi = fmaxf(hi, rf[32 + k]); }
            float sc, ze;
            grid_from_range(lo, hi, a.bits, a.symmetric, &sc, &ze);
            if (tid == 0) { a.scale[r] = sc; a.zero[r] = ze; }
            gsc = (double)sc; gze = (double)ze; gmq = (double)grid_maxq(a.bits, a.symmetric);
            gisc = 1.0 / gsc;
            gr = grid_range(gsc, gze, gmq);
            __syncthreads();                                   // rf is reused by the next row's grid
        };
        for (; s < total; ++s) {
            if (d > ms && nb > 0 && (nb == bcur || m0 - nb <= ms || (SH && s == sched[1]))) {
                // ---- flush: apply the pending vectors and compact to m1 slots ------------------------
                __syncthreads();                           // the last step's vector and perm updates
                const int m1 = m0 - nb;
                if (warp == 0) {
                    // holes (dead slots below the new size) and, as many, live slots above it, paired by rank
                    int nh = 0, nm = 0;
#pragma unroll
                    for (int q = 0; q < 2; ++q) {
                        const int b = lane + 32 * q;
                        const int h = b < nb ? pv[b] : 0x7fffffff;
                        const unsigned hm = __ballot_sync(0xffffffffu, h < m1);
                        if (h < m1) hl[nh + __popc(hm & ((1u << lane) - 1u))] = h;
                        nh += __popc(hm);
                        const bool lv = b < nb && perm[m1 + b] >= 0;
                        const unsigned lm = __ballot_sync(0xffffffffu, lv);
                        if (lv) mv[nm + __popc(lm & ((1u << lane) - 1u))] = m1 + b;
                        nm += __popc(lm);
                    }
                    if (lane == 0) bc->nh = nh;
                } else if (TC && tid == 32) {
                    ft_init_bars(fb);
                }
                __syncthreads();
                const int nh = bc->nh;
                for (int idx = tid; idx < nh * nb; idx += NT) {
                    const int q = idx / nb, b = idx - q * nb;
                    float* zr = (!GP || b < scap) ? panel + (size_t)b * ldz : GVEC + (size_t)(b - scap) * gld;
                    zr[hl[q]] = zr[mv[q]];
                }
                if (tid < nh) {
                    const int h = hl[tid];
                    srcm[h] = (unsigned short)mv[tid];
                    if (!TC) atomicOr(&colmask[h >> 5], 1u << (h & 31));
                }
                __syncthreads();
                if constexpr (TC) {
                    blk_fill_holes<NT>(HP, ldp, m1, nh, hl, mv, srcm);
                    signed char* zexp = a.zexp + (size_t)blockIdx.x * cap;
                    const int power = blk_make_planes<NT, KMAX>(panel, ldz, GP ? scap : nb, GP ? GVEC : nullptr, gld, nb, m0, m1, dg, perm, rf,
                                                                a.Zws + (size_t)blockIdx.x * 128 * a.zld, a.zld, zexp);
                    // the FP64 state gives its space to the pass (d_col = 4608: three tile buffers instead of two)
                    double2* park = a.park + (size_t)blockIdx.x * cap;
                    for (int j = tid; j < cap; j += NT) park[j] = reinterpret_cast<const double2*>(wd)[j];      // (wd and dg: 2 cap doubles)
                    asm volatile("fence.proxy.async;" ::: "memory");            // plain accesses before the copies
                    __syncthreads();
                    unsigned char* stage = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(wd) + 1023) & ~(uintptr_t)1023);
                    const int stage_bytes = (int)(reinterpret_cast<unsigned char*>(panel + a.panel_floats) - stage);
                    const bool fine = blk_flush_tc<(KMAX > 8 ? 3 : FT_GMAX)>(&zmaps, blockIdx.x * 2, (SH ? sched[2] : (int)blockIdx.x) * (((cap + 63) & ~63) >> 5), stage, stage_bytes, fb, m1, nb,
                                      power == 99 ? 1.f : pow2f(-2 * power), power == 99 ? zexp : nullptr, a.stop_tile);
                    for (int j = tid; j < cap; j += NT) reinterpret_cast<double2*>(wd)[j] = __ldcg(park + j);
                    __syncthreads();
                    if (!fine) { timed_out = true; break; }
                } else if (!GP) {                              // (evict-first at every row length: ~1 %)
                    bool wide;
                    const int power = blk_plane_range<NT, KMAX>(panel, ldz, nb, nullptr, 0, nb, m0, m1, dg, perm, rf, &wide);
                    if (!wide) {
                        blk_pack_planes<NT, KMAX>(panel, ldz, nb, m1, pow2f(power));
                        __syncthreads();
                        blk_flush_f16<NT, WIDE>(HP, ldp, m1, nb, panel, ldz, pow2f(-2 * power), srcm, colmask);
                    } else {                                   // small rows of the matrix keep their own precision
                        blk_flush_mma<NT, true, false, WIDE>(HP, ldp, m1, nb, nb, panel, ldz, nullptr, 0, nullptr, srcm, colmask);
                    }
                }
                else
                    blk_flush_mma<NT, true, true, WIDE>(HP, ldp, m1, nb, min(nb, scap), panel, ldz, GVEC, gld, ZSTAGE, srcm, colmask);
                __syncthreads();
                if (tid < nh) {
                    const int h = hl[tid], sv = mv[tid];
                    wd[h] = wd[sv]; dg[h] = dg[sv]; perm[h] = perm[sv];
                    if (BC == 4 && (h & 3) == 0)      // holes and movers are whole aligned groups in block mode
                        for (int k = 0; k < 6; ++k) boff[(h >> 2) * 6 + k] = boff[(sv >> 2) * 6 + k];
                    if (BC == 8 && (h & 7) == 0)
                        for (int k = 0; k < 28; ++k) boff[(h >> 3) * 28 + k] = boff[(sv >> 3) * 28 + k];
                    srcm[h] = (unsigned short)h;
                    if (!TC) colmask[h >> 5] = 0u;
                }
                m0 = m1; nb = 0;
                sa_valid = false; alive_valid = false;
#pragma unroll
                for (int k = 0; k < KMAX; ++k) sa[k] = CUDART_NAN_F;      // slots changed hands: not carried over
#pragma unroll
                for (int g = 0; g < KMAX / 4; ++g) cntw[g] = 0u;
                ldz = blk_ldz(m0);
                scap = a.panel_floats / ldz;
                bcur = blk_updates(m0, a.panel_floats, a.max_pending, gB, !(GP || TC));
                if (BC) bcur &= ~(BC - 1);
                __syncthreads();
            }
            if (SH && s == sched[1]) break;      // (shares of rows) the row is handed over here, everything applied
            if (m0 <= ms) break;                 // on chip from here
            const bool forced = s < n_forced;
            const bool q_now = Q && quant && !forced;
            if ((BG && !has_wfull && (s - n_forced) % BCD == 0 && (!GP || nb + BLK_GS <= scap)) ||
                (FG && forced && !has_wfull && !has_nm && s + BLK_GS <= (SH ? min(n_forced, sched[1]) : n_forced) && nb + BLK_GS <= bcur &&
                 (!GP || nb + BLK_GS <= scap))) {
                // ======================= four forced eliminations together ================================
                constexpr int GS = BLK_GS;
                if (BG) pick_block(rec_view(scratch, s & 1));
                int* gslot = reinterpret_cast<int*>(smem + BLK_OFF_GRP);
                float* gM = reinterpret_cast<float*>(smem + BLK_OFF_GRP + 16);
                int fo[GS];
#pragma unroll
                for (int g = 0; g < GS; ++g) fo[g] = BG ? blk_orig + g : a.forced_order[(size_t)r * d + s + g];
                unsigned live = 0u;
#pragma unroll
                for (int g4 = 0; g4 < KMAX / 4; ++g4) {
                    const int jb = own_slot<NT>(4 * g4);
                    if (jb >= m0) continue;
                    const int4 pm = *reinterpret_cast<const int4*>(perm + jb);
                    const int pq[4] = {pm.x, pm.y, pm.z, pm.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (jb + q < m0 && pq[q] >= 0) {
                            live |= 1u << (4 * g4 + q);
#pragma unroll
                            for (int g = 0; g < GS; ++g)
                                if (!BG && pq[q] == fo[g]) gslot[g] = jb + q;
                        }
                }
                if (!BG) __syncthreads();
                int p4[GS];
                bool ok = true;
#pragma unroll
                for (int g = 0; g < GS; ++g) {
                    p4[g] = BG ? blk_base + g : gslot[g];
                    // (a stale slot is dead, perm = -1, or holds another column)
                    ok = ok && fo[g] >= 0 && p4[g] >= 0 && p4[g] < m0 && perm[p4[g]] == fo[g];
                }
                ok = ok && p4[0] != p4[1] && p4[0] != p4[2] && p4[0] != p4[3] && p4[1] != p4[2] && p4[1] != p4[3] &&
                     p4[2] != p4[3];
                if (ok) {
                    double wp4[GS], dp4[GS];
#pragma unroll
                    for (int g = 0; g < GS; ++g) { wp4[g] = wd[p4[g]]; dp4[g] = dg[p4[g]]; }
                    // the four pivot columns of the stored matrix at the own slots, minus the pending vectors' part (all of them
                    // in shared memory here).  The part is summed first and subtracted once, as a single step does: taken
                    // from the column product by product, every product is rounded at the size of the column's entry (rms error
                    // of the loss 1.2 times as large for blocks of 4, 1.7 times for a replay before OBQ at 960 columns).  The
                    // columns wait in registers of their own or, where there are none, in shared memory at the place of the
                    // vectors to come; only the kernels with more slots and passes on tcgen05, whose stores a copy by way of L1
                    // might miss, subtract product by product.
                    const float* const tri = HP;
                    float v[GS][KMAX], cols[COLS == COLS_REGS ? GS : 1][COLS == COLS_REGS ? KMAX : 1];
                    float* const wait = panel + (size_t)nb * ldz;
#pragma unroll
                    for (int g4 = 0; g4 < KMAX / 4; ++g4) {
                        const int jb = own_slot<NT>(4 * g4);
                        auto stored = [&](int g, int k) -> float& { return COLS == COLS_REGS ? cols[COLS == COLS_REGS ? g : 0][COLS == COLS_REGS ? k : 0] : v[g][k]; };
#pragma unroll
                        for (int g = 0; g < GS; ++g)
#pragma unroll
                            for (int q = 0; q < 4; ++q) { v[g][4 * g4 + q] = 0.f; stored(g, 4 * g4 + q) = 0.f; }
                        if (jb >= m0) continue;
#pragma unroll
                        for (int g = 0; g < GS; ++g) {
                            const int p = p4[g];
                            if (jb + 3 <= p) {
                                const float* from = tri + tri_at<WIDE>(ldp, p, jb);
                                if (COLS == COLS_SMEM) copy_async<16>(wait + (size_t)g * ldz + jb, from);
                                else {
                                    const float4 t = ld_tri4<TC>(from);
                                    stored(g, 4 * g4) = t.x; stored(g, 4 * g4 + 1) = t.y; stored(g, 4 * g4 + 2) = t.z; stored(g, 4 * g4 + 3) = t.w;
                                }
                            } else {
#pragma unroll
                                for (int q = 0; q < 4; ++q) {
                                    const int j = jb + q;
                                    if (!((live >> (4 * g4 + q)) & 1u)) continue;
                                    const float* from = tri + ((j <= p) ? tri_at<WIDE>(ldp, p, j) : tri_at<WIDE>(ldp, j, p));
                                    if (COLS == COLS_SMEM) copy_async<4>(wait + (size_t)g * ldz + j, from);
                                    else stored(g, 4 * g4 + q) = ld_tri<TC>(from);
                                }
                            }
                        }
                    }
                    for (int b = 0; b < nb; ++b) {
                        const float* zo = panel + (size_t)b * ldz;
                        float zp[GS];
#pragma unroll
                        for (int g = 0; g < GS; ++g) zp[g] = zo[p4[g]];
#pragma unroll
                        for (int g4 = 0; g4 < KMAX / 4; ++g4) {
                            if ((live >> (4 * g4)) & 0xFu) {
                                const float4 z = *reinterpret_cast<const float4*>(zo + own_slot<NT>(4 * g4));
#pragma unroll
                                for (int g = 0; g < GS; ++g) {
                                    v[g][4 * g4] = fmaf(-z.x, zp[g], v[g][4 * g4]);
                                    v[g][4 * g4 + 1] = fmaf(-z.y, zp[g], v[g][4 * g4 + 1]);
                                    v[g][4 * g4 + 2] = fmaf(-z.z, zp[g], v[g][4 * g4 + 2]);
                                    v[g][4 * g4 + 3] = fmaf(-z.w, zp[g], v[g][4 * g4 + 3]);
                                }
                            }
                        }
                    }
                    if (COLS == COLS_REGS) {
#pragma unroll
                        for (int g = 0; g < GS; ++g)
#pragma unroll
                            for (int k = 0; k < KMAX; ++k) v[g][k] += cols[COLS == COLS_REGS ? g : 0][COLS == COLS_REGS ? k : 0];
                    } else if (COLS == COLS_SMEM) {
                        asm volatile("cp.async.wait_all;" ::: "memory");       // own copies only: no barrier
#pragma unroll
                        for (int g4 = 0; g4 < KMAX / 4; ++g4) {
                            if (!((live >> (4 * g4)) & 0xFu)) continue;
#pragma unroll
                            for (int g = 0; g < GS; ++g) {
                                const float4 t = *reinterpret_cast<const float4*>(wait + (size_t)g * ldz + own_slot<NT>(4 * g4));
                                v[g][4 * g4] += t.x; v[g][4 * g4 + 1] += t.y; v[g][4 * g4 + 2] += t.z; v[g][4 * g4 + 3] += t.w;
                            }
                        }
                    }
                    // the columns at the four pivot slots, from the owners of those slots
#pragma unroll
                    for (int k = 0; k < KMAX; ++k) {
                        if (!((live >> k) & 1u)) continue;
                        const int j = own_slot<NT>(k);
#pragma unroll
                        for (int g2 = 0; g2 < GS; ++g2)
                            if (j == p4[g2]) {
#pragma unroll
                                for (int g = 0; g < GS; ++g) gM[g * GS + g2] = v[g][k];
                            }
                    }
                    __syncthreads();
                    // the four eliminations at the pivot slots themselves (every thread, same values)
                    float zz[GS][GS];                      // vector e at pivot slot x
                    double idp[GS], fg[GS];
                    float rsq[GS];
                    bool fine = true;
#pragma unroll
                    for (int g = 0; g < GS; ++g) {
                        float mc[GS];
#pragma unroll
                        for (int x = 0; x < GS; ++x) {
                            mc[x] = gM[g * GS + x];
#pragma unroll
                            for (int e = 0; e < g; ++e) mc[x] = fmaf(-zz[e][x], zz[e][g], mc[x]);
                        }
                        const double dpp = dp4[g], w = wp4[g];
                        if (!(dpp > 0.0) || !isfinite(dpp) || !isfinite(w)) fine = false;
                        idp[g] = 1.0 / dpp;
                        fg[g] = w * idp[g];
                        rsq[g] = __frsqrt_rn((float)dpp);
#pragma unroll
                        for (int x = 0; x < GS; ++x) zz[g][x] = mc[x] * rsq[g];
#pragma unroll
                        for (int x = g + 1; x < GS; ++x) {
                            wp4[x] -= fg[g] * (double)mc[x];
                            dp4[x] -= (double)mc[x] * (double)mc[x] * idp[g];
                        }
                    }
                    if (fine) {
#pragma unroll
                        for (int g4 = 0; g4 < KMAX / 4; ++g4) {
                            const int jb = own_slot<NT>(4 * g4);
                            if (jb >= m0) continue;
                            float zv[GS][4], vv[BG ? GS : 1][4];
#pragma unroll
                            for (int q = 0; q < 4; ++q) {
                                const int k = 4 * g4 + q, j = jb + q;
#pragma unroll
                                for (int g = 0; g < GS; ++g) zv[g][q] = 0.f;
                                if (!((live >> k) & 1u)) continue;
                                int gm = GS;                   // this slot is the gm-th pivot (GS: none of them)
#pragma unroll
                                for (int g = 0; g < GS; ++g) if (j == p4[g]) gm = g;
                                double nw = wd[j], nd = dg[j];
#pragma unroll
                                for (int g = 0; g < GS; ++g) {
                                    if (g < gm) {
                                        float vj = v[g][k];
#pragma unroll
                                        for (int e = 0; e < g; ++e) vj = fmaf(-zv[e][q], zz[e][g], vj);
                                        nw -= fg[g] * (double)vj;
                                        nd -= (double)vj * (double)vj * idp[g];
                                        zv[g][q] = vj * rsq[g];
                                        if (BG) vv[BG ? g : 0][q] = vj;
                                    }
                                }
                                if (gm < GS) perm[j] = -1;
                                else { wd[j] = nw; dg[j] = nd; }
                            }
#pragma unroll
                            for (int g = 0; g < GS; ++g)
                                *reinterpret_cast<float4*>(panel + (size_t)(nb + g) * ldz + jb) =
                                    make_float4(zv[g][0], zv[g][1], zv[g][2], zv[g][3]);
                            if (BG && ((live >> (4 * g4)) & 0xFu) == 0xFu && jb != p4[0]) {
                                // Lemma 1 on the group's own 4 x 4 diagonal block, member by member (off-diagonal part)
                                double* o = boff + (jb >> 2) * 6;
#pragma unroll
                                for (int g = 0; g < GS; ++g) {
                                    const double v0 = (double)vv[BG ? g : 0][0], v1 = (double)vv[BG ? g : 0][1];
                                    const double v2 = (double)vv[BG ? g : 0][2], v3 = (double)vv[BG ? g : 0][3];
                                    o[0] -= v0 * v1 * idp[g]; o[1] -= v0 * v2 * idp[g]; o[2] -= v0 * v3 * idp[g];
                                    o[3] -= v1 * v2 * idp[g]; o[4] -= v1 * v3 * idp[g]; o[5] -= v2 * v3 * idp[g];
                                }
                            }
                        }
                        if (BG) {
                            if (tid < GS) {
                                pv[nb + tid] = blk_base + tid;
                                const int t = s - n_forced + tid;
                                if (a.W_out) a.W_out[(size_t)r * a.ldwo + blk_orig + tid] = 0.f;
                                if (a.mask) a.mask[(size_t)r * d + blk_orig + tid] = 0;
                                if (a.order) a.order[(size_t)r * d + t] = blk_orig + tid;
                                if (a.loss) a.loss[(size_t)r * d + t] = tid ? 0.f : (float)blk_score;
                            }
                        } else if (tid < GS) {
                            pv[nb + tid] = p4[tid];
                            if (a.W_out) a.W_out[(size_t)r * a.ldwo + fo[tid]] = 0.f;
                            if (a.mask) a.mask[(size_t)r * d + fo[tid]] = 0;
                        }
                        nb += GS;
                        s += GS - 1;
                        sa_valid = false; alive_valid = false;
#pragma unroll
                        for (int k = 0; k < KMAX; ++k) sa[k] = CUDART_NAN_F;
                        continue;
                    }
                }
                // an entry of the order that names no live column, or a pivot that is not positive: the single steps below
                // meet it again and report it
            }
            // ---- grid of the compound path: built from the survivors when the replay is over -----------
            if (Q && a.mode == MODE_REPLAY_QUANT && s == n_forced) {
                float lo = 0.f, hi = 0.f;
#pragma unroll
                for (int k = 0; k < KMAX; ++k) {               // own slots: their owner is the only writer
                    const int j = own_slot<NT>(k);
                    if (j < m0 && perm[j] >= 0) { const float w = (float)wd[j]; lo = fminf(lo, w); hi = fmaxf(hi, w); }
                }
                survivors_grid(lo, hi);
                sa_valid = false;
            }
            // ---- pick the slot ---------------------------------------------------------------------------
            const Records rec = rec_view(scratch, s & 1);
            Pick pk;
            bool sure = true;
            if (forced) {
                const int f = a.forced_order[(size_t)r * d + s];
                int cslot = -1;
#pragma unroll
                for (int k = 0; k < KMAX; ++k) {
                    const int j = own_slot<NT>(k);
                    if (j < m0 && f >= 0 && perm[j] == f) cslot = j;      // (perm = -1: a dead slot)
                }
                pk = known_pick<NT>(cslot, f, rec);
            } else if (BC && (s - n_forced) % BCD != 0) {
                // the next member of the block chosen at the last block boundary: a block's slots hold consecutive columns
                __syncthreads();
                pk.slot = blk_base + (s - n_forced) % BCD; pk.orig = blk_orig + (s - n_forced) % BCD; pk.s = 0.0;
            } else if (BC) {
                pk = pick_block(rec);
            } else {
                if (!sa_valid || outliers)
                    estimate_own<NT, KMAX, Q>(sa, wd, dg, perm, m0, q_now, gsc, gisc, gze, gmq, gr, has_nm ? blkcnt : nullptr,
                                           nm_lg, nm_prune, cntw);
                if (!(Q && outliers)) {
                    float e1, e2;
                    int cslot;
                    smallest_own<NT, KMAX>(sa, &e1, &e2, &cslot);
                    pk = fast_pick<NT>(e1, e2, cslot, cslot >= 0 ? perm[cslot] : -1, rec, &sure);
                } else {
                    sure = false;
                }
                if (!sure) {                                   // (the same for every thread of the block)
                    unsigned key = KEY_NONE;
                    double cs = 0.0;
                    int cslot = -1;
                    thread_best<NT, KMAX, Q>(sa, wd, dg, perm, q_now, outliers, gsc, gisc, gze, gmq, &key, &cs, &cslot);
                    pk = block_pick<NT>(key, cs, cslot, cslot >= 0 ? perm[cslot] : -1, rec);
                }
            }
            const int p = pk.slot, op = pk.orig;
            const double dpp = p < 0 ? 0.0 : dg[p], wp = p < 0 ? 0.0 : wd[p];      // (a pivot's state is not written again)
            if (p < 0 || !(dpp > 0.0) || !isfinite(dpp) || !isfinite(wp)) { failed = true; break; }
            double qp = 0.0, code = -1.0;
            if (Q && q_now) qp = grid_q_fast(wp, gsc, gisc, gze, gmq, &code);
            const double e = wp - qp;
            // ======================= deferred-update step ==============================================
            float* zb = (!GP || nb < scap) ? panel + (size_t)nb * ldz : GVEC + (size_t)(nb - scap) * gld;
            // pivot column of the stored matrix (own slots), corrected by the pending vectors
            const float* const tri = HP;
            float c[KMAX], corr[KMAX];
            if (!alive_valid) {
                alive = 0u;
#pragma unroll
                for (int g = 0; g < KMAX / 4; ++g) {
                    const int jb = own_slot<NT>(4 * g);
                    if (jb >= m0) continue;
                    const int4 pm = *reinterpret_cast<const int4*>(perm + jb);
                    const int pq[4] = {pm.x, pm.y, pm.z, pm.w};
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (jb + q < m0 && pq[q] >= 0) alive |= 1u << (4 * g + q);
                }
                alive_valid = true;
            }
            const bool owner = ((p >> 2) & (NT - 1)) == tid;
            if (owner) alive &= ~(1u << ((p >> 2) / NT * 4 + (p & 3)));
#pragma unroll
            for (int g = 0; g < KMAX / 4; ++g) {
                const int jb = own_slot<NT>(4 * g);
#pragma unroll
                for (int q = 0; q < 4; ++q) { c[4 * g + q] = 0.f; corr[4 * g + q] = 0.f; }
                if (jb >= m0) continue;
                if (jb + 3 <= p) {
                    const float4 v = ld_tri4<TC>(tri + tri_at<WIDE>(ldp, p, jb));
                    c[4 * g] = v.x; c[4 * g + 1] = v.y; c[4 * g + 2] = v.z; c[4 * g + 3] = v.w;
                } else {
#pragma unroll
                    for (int q = 0; q < 4; ++q) {
                        const int j = jb + q;
                        if ((alive >> (4 * g + q)) & 1u) c[4 * g + q] = ld_tri<TC>(tri + ((j <= p) ? tri_at<WIDE>(ldp, p, j) : tri_at<WIDE>(ldp, j, p)));
                    }
                }
            }
            const double idpp = 1.0 / dpp;
            const double f = e * idpp;
            const float rs = __frsqrt_rn((float)dpp);
            const int nbs = GP ? min(nb, scap) : nb;
            for (int b = 0; b < nbs; ++b) {
                const float* zo = panel + (size_t)b * ldz;
                const float zp = zo[p];
#pragma unroll
                for (int g = 0; g < KMAX / 4; ++g) {
                    if ((alive >> (4 * g)) & 0xFu) {
                        const float4 z = *reinterpret_cast<const float4*>(zo + own_slot<NT>(4 * g));
                        corr[4 * g] = fmaf(z.x, zp, corr[4 * g]);
                        corr[4 * g + 1] = fmaf(z.y, zp, corr[4 * g + 1]);
                        corr[4 * g + 2] = fmaf(z.z, zp, corr[4 * g + 2]);
                        corr[4 * g + 3] = fmaf(z.w, zp, corr[4 * g + 3]);
                    }
                }
            }
            if (GP)
#pragma unroll 4
            for (int b = nbs; b < nb; ++b) {               // the overflow vectors, from L2
                const float* zo = GVEC + (size_t)(b - scap) * gld;
                const float zp = zo[p];
#pragma unroll
                for (int g = 0; g < KMAX / 4; ++g) {
                    if ((alive >> (4 * g)) & 0xFu) {
                        const float4 z = *reinterpret_cast<const float4*>(zo + own_slot<NT>(4 * g));
                        corr[4 * g] = fmaf(z.x, zp, corr[4 * g]);
                        corr[4 * g + 1] = fmaf(z.y, zp, corr[4 * g + 1]);
                        corr[4 * g + 2] = fmaf(z.z, zp, corr[4 * g + 2]);
                        corr[4 * g + 3] = fmaf(z.w, zp, corr[4 * g + 3]);
                    }
                }
            }
            // state update of the own slots (Eq. 3 / Eq. 7), the new pending vector, and the score
            // estimates the next free step starts from
            const bool est_next = !BC && (s + 1 >= n_forced) && !outliers;
            const bool q_next = Q && quant && (s + 1 >= n_forced);
#pragma unroll
            for (int g = 0; g < KMAX / 4; ++g) {
                const int jb = own_slot<NT>(4 * g);
                if (jb >= m0) continue;
                int pq[4] = {0, 0, 0, 0};
                if (has_nm || has_wfull) {
                    const int4 pm = *reinterpret_cast<const int4*>(perm + jb);
                    pq[0] = pm.x; pq[1] = pm.y; pq[2] = pm.z; pq[3] = pm.w;
                }
                float zv[4];
                // the group's FP64 state as 128-bit accesses: a warp's 64-bit accesses at this stride (32 bytes
                // between lanes) would meet four to a bank; dead slots keep the value they had
                double2* wq = reinterpret_cast<double2*>(wd + jb);
                double2* dq = reinterpret_cast<double2*>(dg + jb);
                const double2 w01 = wq[0], w23 = wq[1], d01 = dq[0], d23 = dq[1];
                double wv[4] = {w01.x, w01.y, w23.x, w23.y}, dv[4] = {d01.x, d01.y, d23.x, d23.y};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const int k = 4 * g + q;
                    zv[q] = 0.f;
                    sa[k] = CUDART_NAN_F;
                    if (!((alive >> k) & 1u)) continue;
                    const float vj = c[k] - corr[k];
                    const double nw = wv[q] - f * (double)vj;
                    const double nd = dv[q] - (double)vj * (double)vj * idpp;
                    wv[q] = nw; dv[q] = nd;
                    zv[q] = vj * rs;
                    if (est_next) sa[k] = score_estimate<Q>(nw, nd, q_next, gsc, gisc, gze, gmq, gr);
                    if (has_nm) {
                        if ((pq[q] >> nm_lg) == (op >> nm_lg)) cntw[g] += 1u << (8 * q);
                        if ((int)((cntw[g] >> (8 * q)) & 0xFFu) >= nm_prune) sa[k] = CUDART_NAN_F;
                    }
                    if (has_wfull) wfull[pq[q]] = (float)nw;
                }
                wq[0] = make_double2(wv[0], wv[1]); wq[1] = make_double2(wv[2], wv[3]);
                dq[0] = make_double2(dv[0], dv[1]); dq[1] = make_double2(dv[2], dv[3]);
                *reinterpret_cast<float4*>(zb + jb) = make_float4(zv[0], zv[1], zv[2], zv[3]);
                if (BC == 4 && ((alive >> (4 * g)) & 0xFu) == 0xFu) {
                    // Lemma 1 on the group's own 4 x 4 diagonal block (off-diagonal part; dg holds the diagonal)
                    double* o = boff + (jb >> 2) * 6;
                    const double v0 = (double)(c[4 * g] - corr[4 * g]), v1 = (double)(c[4 * g + 1] - corr[4 * g + 1]);
                    const double v2 = (double)(c[4 * g + 2] - corr[4 * g + 2]), v3 = (double)(c[4 * g + 3] - corr[4 * g + 3]);
                    o[0] -= v0 * v1 * idpp; o[1] -= v0 * v2 * idpp; o[2] -= v0 * v3 * idpp;
                    o[3] -= v1 * v2 * idpp; o[4] -= v1 * v3 * idpp; o[5] -= v2 * v3 * idpp;
                }
            }
            if (BC == 8) {
                // Lemma 1 on the 8 x 8 diagonal block of every other whole block: its two halves belong to
                // neighbouring lanes, which exchange their four column entries; the lane of the first half takes
                // the pairs whose smaller index is 0 or 1, the other lane the rest
#pragma unroll
                for (int g = 0; g < KMAX / 4; ++g) {
                    const int jb = own_slot<NT>(4 * g);
                    float mine[4], other[4];
#pragma unroll
                    for (int q = 0; q < 4; ++q) mine[q] = c[4 * g + q] - corr[4 * g + q];
#pragma unroll
                    for (int q = 0; q < 4; ++q) other[q] = __shfl_xor_sync(0xffffffffu, mine[q], 1);
                    if (jb < m0 && ((alive >> (4 * g)) & 0xFu) == 0xFu && (jb & ~7) != (p & ~7)) {
                        const bool first = (jb & 7) == 0;
                        double v[8];
#pragma unroll
                        for (int q = 0; q < 4; ++q) {
                            v[q] = (double)(first ? mine[q] : other[q]);
                            v[4 + q] = (double)(first ? other[q] : mine[q]);
                        }
                        double* o = boff + (jb >> 3) * 28;
#pragma unroll
                        for (int i = 0; i < 7; ++i)
#pragma unroll
                            for (int j = i + 1; j < 8; ++j)
                                if ((i < 2) == first) o[block8_index(i, j)] -= v[i] * v[j] * idpp;
                    }
                }
            }
            sa_valid = est_next;
            if (owner) {
                perm[p] = -1;
                if (has_nm) blkcnt[op >> nm_lg] += 1;              // read again only behind a barrier
            }
            if (tid == NT - 32) {                          // (of the warp with the fewest slots)
                pv[nb] = p;
                if (has_wfull) wfull[op] = (float)qp;
                if (a.W_out) a.W_out[(size_t)r * a.ldwo + op] = (float)qp;
                if (a.mask) a.mask[(size_t)r * d + op] = 0;
                if (!forced) {
                    const int t = s - n_forced;
                    if (a.order) a.order[(size_t)r * d + t] = op;
                    if (a.loss) a.loss[(size_t)r * d + t] = BC ? ((t % BCD) ? 0.f : (float)blk_score) : (float)(e * f);
                }
                if (q_now && a.codes) a.codes[(size_t)r * d + op] = (int)code;
            }
            ++nb;
            if (a.w_trace && s < a.trace_steps) {
                __syncthreads();
                for (int j = tid; j < d; j += NT)
                    a.w_trace[((size_t)r * (a.trace_steps + 1) + s + 1) * d + j] = wfull[j];
                // wfull is next written in the update phase of the following step, i.e. behind that step's
                // barrier, which every thread reaches only after these reads
            }
        }
        // ======================= the end of a row on chip ==========================================================
        // At most ms <= NT slots: one per thread, its weight, diagonal and score estimate in registers (the state arrays are kept
        // current for the pivot's readers).  A step is the pick's barrier, one entry of the pivot's column, its corrections by the
        // deferred updates (all TAIL_B of them, zero where there are none yet) and the state; every TAIL_B steps the triangle is
        // updated, and compacted when 32 slots or a quarter of them are gone.  What bounds it is the latency of that chain: about
        // 1500 cycles a step, where KMAX slots per thread, four barriers and a pass over the triangle in every step took 8000.
        if (s < total && m0 <= ms && !failed && !timed_out) {
            __syncthreads();                                   // (pending vectors' space changes hands)
            for (int i = warp; i < m0; i += NW)
                for (int j = lane; j <= i; j += 32)
                    S[tail_at(i, j)] = d > ms ? ld_tri<TC>(HP + tri_at<WIDE>(ldp, i, j)) : a.Hinv[(size_t)i * a.ldhi + j];
            const int j = tid;
            double w = 0.0, g = 0.0;
            int o = -1, cnt = 0;
            float est = CUDART_NAN_F;
            auto take_slot = [&](int from) {                   // this thread's slot holds what slot `from` held
                w = wd[from]; g = dg[from]; o = perm[from];
                if (has_nm && o >= 0) cnt = blkcnt[o >> nm_lg];
            };
            auto clear_updates = [&]() {
                if (j < ms) {
                    float4* z = reinterpret_cast<float4*>(vt + j * TAIL_LD);
                    float4* u = reinterpret_cast<float4*>(ut + j * TAIL_LD);
                    z[0] = z[1] = u[0] = u[1] = make_float4(0.f, 0.f, 0.f, 0.f);
                }
            };
            if (j < m0) take_slot(j);
            clear_updates();
            bool est_valid = false;
            int left = m0;                                     // live slots among the m0
            nb = 0;
            __syncthreads();
            for (; s < total; ++s) {
                const bool forced = s < n_forced;
                const bool q_now = Q && quant && !forced;
                if (Q && a.mode == MODE_REPLAY_QUANT && s == n_forced) {
                    survivors_grid(o >= 0 ? fminf(0.f, (float)w) : 0.f, o >= 0 ? fmaxf(0.f, (float)w) : 0.f);
                    est_valid = false;
                }
                const Records rec = rec_view(scratch, s & 1);
                Pick pk;
                if (forced) {
                    const int f = a.forced_order[(size_t)r * d + s];
                    pk = known_pick<NT>(o >= 0 && o == f ? j : -1, f, rec);      // (o = -1: a dead slot, or none)
                } else {
                    if (!est_valid) {
                        est = CUDART_NAN_F;
                        if (o >= 0 && !(has_nm && cnt >= nm_prune)) est = score_estimate<Q>(w, g, q_now, gsc, gisc, gze, gmq, gr);
                    }
                    bool sure = false;
                    if (!(Q && outliers)) pk = fast_pick<NT>(est, CUDART_INF_F, est == est ? j : -1, o, rec, &sure);
                    if (!sure) {                               // FP64 scores of all slots; the outlier rule as in thread_best
                        unsigned key = KEY_NONE;
                        double cs = CUDART_INF;
                        if (est == est) {
                            const double err = q_now ? grid_error(w, gsc, gisc, gze, gmq) : -w;
                            cs = err * err / g;
                            if (Q && outliers && fabs(err) > 0.5 * gsc) cs = -fabs(err);
                            if (cs == cs) key = float_key(__double2float_rn(cs));
                        }
                        pk = block_pick<NT>(key, cs, key != KEY_NONE ? j : -1, o, rec);
                    }
                }
                const int p = pk.slot, op = pk.orig;
                const double dpp = p < 0 ? 0.0 : dg[p], wp = p < 0 ? 0.0 : wd[p];      // (a pivot's state is not written again)
                if (p < 0 || !(dpp > 0.0) || !isfinite(dpp) || !isfinite(wp)) { failed = true; break; }
                double qp = 0.0, code = -1.0;
                if (Q && q_now) qp = grid_q_fast(wp, gsc, gisc, gze, gmq, &code);
                const double e = wp - qp, idpp = 1.0 / dpp, f = e * idpp;
                if (j == p) {
                    if (has_nm) blkcnt[op >> nm_lg] += 1;      // read again only behind a barrier
                    perm[p] = -1; o = -1;
                    est = CUDART_NAN_F;
                }
                const bool est_next = s + 1 >= n_forced && !outliers;
                if (o >= 0) {
                    float* vj = vt + j * TAIL_LD;
                    float* uj = ut + j * TAIL_LD;
                    const float4* up = reinterpret_cast<const float4*>(ut + p * TAIL_LD);
                    const float4 a0 = *reinterpret_cast<const float4*>(vj), a1 = *reinterpret_cast<const float4*>(vj + 4), b0 = up[0], b1 = up[1];
                    float x = a0.x * b0.x;
                    x = fmaf(a0.y, b0.y, x); x = fmaf(a0.z, b0.z, x); x = fmaf(a0.w, b0.w, x);
                    x = fmaf(a1.x, b1.x, x); x = fmaf(a1.y, b1.y, x); x = fmaf(a1.z, b1.z, x); x = fmaf(a1.w, b1.w, x);
                    const float v = S[j > p ? tail_at(j, p) : tail_at(p, j)] - x;
                    const double vd = (double)v, ud = vd * idpp;
                    w -= f * vd;
                    g -= vd * ud;
                    vj[nb] = v; uj[nb] = (float)ud;
                    wd[j] = w; dg[j] = g;
                    if (has_wfull) wfull[o] = (float)w;
                    if (has_nm && (o >> nm_lg) == (op >> nm_lg)) ++cnt;
                    if (est_next) {
                        est = score_estimate<Q>(w, g, Q && quant, gsc, gisc, gze, gmq, gr);
                        if (has_nm && cnt >= nm_prune) est = CUDART_NAN_F;
                    }
                }
                est_valid = est_next;
                if (tid == NT - 32) {
                    if (has_wfull) wfull[op] = (float)qp;
                    if (a.W_out) a.W_out[(size_t)r * a.ldwo + op] = (float)qp;
                    if (a.mask) a.mask[(size_t)r * d + op] = 0;
                    if (!forced) {
                        const int t = s - n_forced;
                        if (a.order) a.order[(size_t)r * d + t] = op;
                        if (a.loss) a.loss[(size_t)r * d + t] = (float)(e * f);
                    }
                    if (q_now && a.codes) a.codes[(size_t)r * d + op] = (int)code;
                }
                --left;
                if (a.w_trace && s < a.trace_steps) {
                    __syncthreads();
                    for (int i = tid; i < d; i += NT)
                        a.w_trace[((size_t)r * (a.trace_steps + 1) + s + 1) * d + i] = wfull[i];
                }
                if (++nb == TAIL_B && s + 1 < total) {
                    __syncthreads();
                    tail_flush<NT>(S, m0, vt, ut, perm);
                    const bool compact = m0 - left >= min(32, m0 >> 2);      // (at most 39 slots are gone: hl and mv hold 64)
                    if (compact && warp == NW - 1) {           // holes and, as many, live slots above the new size
                        int nh = 0, nm = 0;
                        for (int i0 = 0; i0 < m0; i0 += 32) {
                            const int i = i0 + lane;
                            const bool lv = i < m0 && perm[i] >= 0;
                            const unsigned hm = __ballot_sync(0xffffffffu, i < left && !lv), lm = __ballot_sync(0xffffffffu, i >= left && lv);
                            const unsigned below = (1u << lane) - 1u;
                            if (i < left && !lv) hl[nh + __popc(hm & below)] = i;
                            if (i >= left && lv) mv[nm + __popc(lm & below)] = i;
                            nh += __popc(hm); nm += __popc(lm);
                        }
                        if (lane == 0) bc->nh = nh;
                        __syncwarp();
                        for (int q = lane; q < nh; q += 32) srcm[hl[q]] = (unsigned short)mv[q];
                    }
                    __syncthreads();
                    clear_updates();
                    nb = 0;
                    if (compact) {
                        const int nh = bc->nh;
                        for (int q = warp; q < nh; q += NW) {  // read from rows >= left, which nothing here writes
                            const int h = hl[q], from = mv[q];
                            for (int i = lane; i < left; i += 32) {
                                const int si = srcm[i];
                                S[tail_at(max(h, i), min(h, i))] = S[tail_at(max(from, si), min(from, si))];
                            }
                        }
                        const int from = j < left ? (int)srcm[j] : j;
                        __syncthreads();
                        if (j >= left) o = -1;
                        else if (from != j) { take_slot(from); wd[j] = w; dg[j] = g; perm[j] = o; srcm[j] = (unsigned short)j; }
                        m0 = left;
                        est_valid = false;
                    }
                    __syncthreads();
                }
            }
        }
        // ---- row epilogue ---------------------------------------------------------------------------------
        __syncthreads();
        failed = failed || timed_out;
        if (SH && sched[0] == ITEM_HEAD) {
            // (shares of rows) leave the row to the next block: state at the flush boundary, then the flag
            const bool handed = !failed && s < total;
            if (handed)
                blk_state_copy(true, a.split_state + (size_t)blockIdx.x * a.split_stride, cap, d, m0, NT, wd, dg, perm, srcm,
                               has_wfull ? wfull : nullptr);
            else
                __threadfence();
            __syncthreads();
            if (tid == 0)
                blk_publish(a.split_state + (size_t)blockIdx.x * a.split_stride, a.split_flags + blockIdx.x, s, m0, handed ? 0 : 1);
            if (handed) { __syncthreads(); continue; }
        }
        if (failed) {           // stopped early: report the step, mark what was not produced
            if (tid == 0) a.row_status[r] = timed_out ? -(int)OBC_ERR_TIMEOUT : 1 + s;
            const int t0 = (s < n_forced) ? 0 : s - n_forced;
            for (int t = t0 + tid; t < n_free; t += NT) {
                if (a.order) a.order[(size_t)r * d + t] = -1;
                if (a.loss) a.loss[(size_t)r * d + t] = CUDART_INF_F;
            }
        }
        if (a.W_out)            // eliminated entries were written at their step; the live ones follow here
            for (int j = tid; j < m0; j += NT)
                if (perm[j] >= 0) a.W_out[(size_t)r * a.ldwo + perm[j]] = (float)wd[j];
        __syncthreads();
    }
    if (TC && d > ms) ft_free(fb);
}

#undef HP
#undef GVEC
#undef ZSTAGE

// ---- launch -------------------------------------------------------------------------------------------------------
template <int NT, int KMAX, bool Q, int BC, bool FG, bool GPV, bool NM>
inline obc_status blk_launch_g(const FlushMaps& zmaps, EngineArgs a, int blocks, size_t smem, int sm_count, cudaStream_t stream) {
    BlkMaps<NT, BC> maps;
    if constexpr (blk_tc<NT, BC>) maps = zmaps;
    auto kernel = blocked_engine_kernel<NT, KMAX, Q, BC, FG, GPV, false, NM>;
    auto kernel_sh = blocked_engine_kernel<NT, KMAX, Q, BC, FG, GPV, (BC == 0 && !NM), NM>;     // (block and N:M pruning take no shares)
    if (a.split) {
        // A block may wait (bounded) for the row its neighbour started, so all blocks must be resident at once: checked
        // here, and guaranteed by a cooperative launch.  If the grid does not fit, rows run in whole waves instead.
        OBC_CUDA_TRY(cudaFuncSetAttribute(kernel_sh, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        int per_sm = 0;
        OBC_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel_sh, NT, smem));
        int coop = 0, dev = 0;
        OBC_CUDA_TRY(cudaGetDevice(&dev));
        OBC_CUDA_TRY(cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev));
        if (BC != 0 || NM || !coop || (long long)per_sm * sm_count < blocks) a.split = 0;
    }
    if (a.split) {
        OBC_CUDA_TRY(cudaMemsetAsync(a.split_flags, 0, (size_t)blocks * sizeof(int), stream));
        void* params[2] = {(void*)&maps, (void*)&a};
        OBC_CUDA_TRY(cudaLaunchCooperativeKernel((const void*)kernel_sh, dim3(blocks), dim3(NT), params, smem, stream));
    } else {
        OBC_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        kernel<<<blocks, NT, smem, stream>>>(maps, a);
    }
    count_launch();
    OBC_CUDA_TRY(cudaGetLastError());
    return OBC_OK;
}

template <int NT, int KMAX, bool Q, int BC, bool FG, bool NM = false>
inline obc_status blk_launch_q(const FlushMaps& zmaps, const EngineArgs& a, int blocks, size_t smem, int sm_count, cudaStream_t stream) {
    if (NT >= 512 && a.Gpan != nullptr) return blk_launch_g<NT, KMAX, Q, BC, FG, (NT >= 512), NM>(zmaps, a, blocks, smem, sm_count, stream);
    return blk_launch_g<NT, KMAX, Q, BC, FG, false, NM>(zmaps, a, blocks, smem, sm_count, stream);
}

template <int NT, int KMAX>
inline obc_status blk_launch(const FlushMaps& zmaps, const EngineArgs& a, int blocks, size_t smem, int sm_count, cudaStream_t stream) {
    if (a.block_c == 4) return blk_launch_q<NT, KMAX, false, 4, false>(zmaps, a, blocks, smem, sm_count, stream);
    if (a.block_c == 8) return blk_launch_q<NT, KMAX, false, 8, false>(zmaps, a, blocks, smem, sm_count, stream);
    if (a.nm_prune > 0) return blk_launch_q<NT, KMAX, false, 0, false, true>(zmaps, a, blocks, smem, sm_count, stream);
    switch (a.mode) {                       // the replay modes are the ones with forced eliminations
        case MODE_QUANT:        return blk_launch_q<NT, KMAX, true, 0, false>(zmaps, a, blocks, smem, sm_count, stream);
        // (with 512 threads the OBQ kernel has no registers to spare for the four columns: single steps there)
        case MODE_REPLAY_QUANT: return blk_launch_q<NT, KMAX, true, 0, (NT <= 256)>(zmaps, a, blocks, smem, sm_count, stream);
        case MODE_REPLAY:       return blk_launch_q<NT, KMAX, false, 0, true>(zmaps, a, blocks, smem, sm_count, stream);
        default:                return blk_launch_q<NT, KMAX, false, 0, false>(zmaps, a, blocks, smem, sm_count, stream);
    }
}

}  // namespace obc
