// Global mask selection (Algorithm 2 of "Optimal Brain Compression", appendix "ExactOBS Global Step").
//
// The sequential procedure pops, k times, the row whose NEXT recorded loss is smallest (ties: lowest row).
// A row's losses need not be monotone, so a cheap entry hidden behind an expensive one is only reached
// after the expensive one was popped.  Equivalent parallel form: give entry (r,t) the key
// max_{t'<=t} L[r][t'] (prefix maximum); the procedure then pops exactly the k smallest entries in the
// lexicographic order (key, r, t).  Within a row keys are non-decreasing, so the popped entries of a row
// are a prefix and counts[r] = #{key < T} + (share of the entries with key == T, handed out by row).
//
// One cooperative launch does all of it (a barrier over the grid per 9 + 11 + 11 bits of the key would be two launches and
// their gaps otherwise: twelve kernels took 96 us a call, nearly all of it launch latency).  A block owns consecutive rows and keeps
// their keys in shared memory.  Keys of a row do not decrease, so a digit histogram needs only the places where the
// digit changes: key t with another digit than key t + 1 adds t + 1 to its own bin and takes t + 1 from the next one; and
// once a digit is decided, a binary search per row narrows the row to the keys that share it, so only the first digit
// (few bits: few changes) scans whole rows.
// Keys are non-negative floats compared as unsigned integers.
#include "common.cuh"
#include "grid_barrier.cuh"
#include <mutex>

namespace obc {

constexpr int SEL_THREADS = 1024;
constexpr int SEL_WARPS = SEL_THREADS / 32;
constexpr int SEL_MAX_BLOCKS = 512;
constexpr int SEL_MAX_UNITS = 128;                // row segments of a block, when rows are cut into segments
constexpr int SEL_BINS = 2048;
constexpr int64_t SEL_WIDE = 1ll << 32;           // from this many keys on, counts and bins have 64 bits
constexpr size_t SEL_WIDE_BYTES = 3 * SEL_BINS * 8;
constexpr int SEL_SMEM = 200 * 1024;              // keys of a block's rows, if they fit

struct SelectState {            // in the workspace, zero before the launch
    unsigned int hist[3][SEL_BINS];               // (from 2^32 keys on: 64-bit bins behind the other arrays)
    unsigned int arrived;       // blocks at the grid barriers
    unsigned int pad[63];
    unsigned long long ties[SEL_MAX_BLOCKS];      // keys equal to the k-th one, per block
};

__device__ __forceinline__ unsigned int loss_key(float x) {
    // losses are >= 0; NaN and negative values are mapped to the ends so that the order stays total
    if (x != x) return 0x7f800000u;          // NaN -> +inf
    if (x <= 0.f) return 0u;                 // -0, negatives
    return __float_as_uint(x);
}

template <typename Count> struct SelectShared {
    Count hist[SEL_BINS];
    unsigned int segmax[SEL_MAX_UNITS];
    Count scan[SEL_WARPS];
    Count rem, before;
    unsigned int digit;
    Count digit_count;
};

// Inclusive scan over the block of one value per thread; sh.scan[w] = total of warps 0 .. w afterwards.
template <typename Count>
__device__ __forceinline__ Count block_scan(Count v, SelectShared<Count>& sh) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const Count o = __shfl_up_sync(0xffffffffu, v, off);
        if (lane >= off) v += o;
    }
    __syncthreads();                                      // the previous scan's totals have been read
    if (lane == 31) sh.scan[warp] = v;
    __syncthreads();
    Count w = sh.scan[lane];                              // (every warp scans the 32 totals for itself)
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {
        const Count o = __shfl_up_sync(0xffffffffu, w, off);
        if (lane >= off) w += o;
    }
    const Count below = __shfl_sync(0xffffffffu, w, warp > 0 ? warp - 1 : 0);
    return warp > 0 ? v + below : v;
}

// Thread t owns bins 2t, 2t + 1 (counts a, b): the bin that holds rank sh.rem becomes sh.digit, sh.rem the rank inside it.
template <typename Count>
__device__ __forceinline__ void pick_digit(Count a, Count b, SelectShared<Count>& sh) {
    const Count incl = block_scan((Count)(a + b), sh);
    const Count rem = sh.rem, before = incl - a - b;
    __syncthreads();
    if (before < rem && rem <= incl) {
        const bool second = rem > before + a;
        sh.digit = 2 * threadIdx.x + (second ? 1 : 0);
        sh.digit_count = second ? b : a;
        sh.rem = rem - before - (second ? a : 0);
    }
    __syncthreads();
}

// keys: the block's rows in shared memory (IN_SMEM) or this call's rows in the workspace.  A block takes rows
// [rpb * blockIdx.x, + rpb), cut into `segs` segments each for the scans (one warp per segment).
template <bool IN_SMEM, typename Count>
__global__ void __launch_bounds__(SEL_THREADS, 1) select_kernel(const float* __restrict__ loss, const int32_t* __restrict__ order, int rows, int d,
                                                             unsigned long long k, int rpb, int segs, unsigned int* __restrict__ gkeys,
                                                             int* __restrict__ glt, int* __restrict__ gle, SelectState* __restrict__ st, Count* __restrict__ ghist,
                                                             int* __restrict__ counts, uint8_t* __restrict__ mask, int wait_limit) {
    extern __shared__ __align__(16) unsigned int skeys[];
    __shared__ SelectShared<Count> sh;
    __shared__ int slt[SEL_THREADS], sle[SEL_THREADS];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int r0 = blockIdx.x * rpb, nr = min(rpb, rows - r0);           // >= 1
    const unsigned int G = gridDim.x;
    const int ldk = IN_SMEM ? (d + 3) & ~3 : d;          // stride of the keys
    const int seg_len = ((d + segs - 1) / segs + 3) & ~3;
    const int units = nr * segs;
    unsigned int* keys = IN_SMEM ? skeys : gkeys + (size_t)r0 * ldk;
    const float* L = loss + (size_t)r0 * d;
    int* row_lt = rpb <= SEL_THREADS ? slt : glt + r0;
    int* row_le = rpb <= SEL_THREADS ? sle : gle + r0;
    unsigned int barrier_no = 0;

    for (int b = tid; b < SEL_BINS; b += SEL_THREADS) sh.hist[b] = 0;
    if (tid == 0) sh.rem = (Count)k;
    // keys [row_lt, row_le) of a row share the digits decided so far (in the end: are equal to the k-th key)
    for (int r = tid; r < nr; r += SEL_THREADS) { row_lt[r] = 0; row_le[r] = k > 0 ? d : 0; }
    // ---- prefix maxima within segments
    for (int u = warp; u < units; u += SEL_WARPS) {
        const int r = u / segs, g = u - r * segs;
        const int b = g * seg_len, e = min(d, b + seg_len);
        const float* Lr = L + (size_t)r * d;
        unsigned int carry = 0u;
        float nx[8];                                      // the next 256 losses are on their way while these are scanned
#pragma unroll
        for (int q = 0; q < 8; ++q) nx[q] = b + 32 * q + lane < e ? __ldg(Lr + b + 32 * q + lane) : 0.f;
        for (int t0 = b; t0 < e; t0 += 256) {
            unsigned int v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = loss_key(nx[q]);
#pragma unroll
            for (int q = 0; q < 8; ++q) nx[q] = t0 + 256 + 32 * q + lane < e ? __ldg(Lr + t0 + 256 + 32 * q + lane) : 0.f;
#pragma unroll
            for (int off = 1; off < 32; off <<= 1)
#pragma unroll
                for (int q = 0; q < 8; ++q) {             // eight independent scans
                    const unsigned int o = __shfl_up_sync(0xffffffffu, v[q], off);
                    if (lane >= off) v[q] = max(v[q], o);
                }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const unsigned int top = __shfl_sync(0xffffffffu, v[q], 31);
                if (t0 + 32 * q + lane < e) keys[(size_t)r * ldk + t0 + 32 * q + lane] = max(v[q], carry);
                carry = max(carry, top);
            }
        }
        if (segs > 1 && lane == 0) sh.segmax[u] = carry;
    }
    __syncthreads();
    // ---- the key of rank k, 9 + 11 + 11 bits
    unsigned int prefix = 0u;
    if (k > 0) {
#pragma unroll 1
        for (int pass = 0; pass < 3; ++pass) {
            const int shift = pass == 0 ? 22 : (pass == 1 ? 11 : 0);
            constexpr unsigned int dmask = 2047u;
            if (pass == 0) {
                // whole rows; segments also receive the maximum of what is before them
                for (int u = warp; u < units; u += SEL_WARPS) {
                    const int r = u / segs, g = u - r * segs;
                    unsigned int* K = keys + (size_t)r * ldk;
                    unsigned int carry = 0u;
                    for (int q = 0; q < g; ++q) carry = max(carry, sh.segmax[r * segs + q]);
                    const int e = min(d, (g + 1) * seg_len);
                    auto change = [&](unsigned int key, unsigned int next, int t) {      // t < d
                        const unsigned int f = key >> 22, fn = next >> 22;
                        if (t + 1 == d) atomicAdd(&sh.hist[f], (Count)d);
                        else if (f != fn) {
                            atomicAdd(&sh.hist[f], (Count)(t + 1));
                            atomicAdd(&sh.hist[fn], (Count)0 - (Count)(t + 1));
                        }
                    };
                    if (IN_SMEM) {
                        for (int t = g * seg_len + 4 * lane; t < e; t += 128) {
                            uint4 x = *reinterpret_cast<uint4*>(K + t);
                            unsigned int y = t + 4 < d ? K[t + 4] : 0u;
                            if (g > 0) {
                                x.x = max(x.x, carry); x.y = max(x.y, carry); x.z = max(x.z, carry); x.w = max(x.w, carry);
                                *reinterpret_cast<uint4*>(K + t) = x;
                            }
                            const int left = min(4, d - t);
                            // (y may be another segment's: at least this segment's last key)
                            y = max(y, left == 4 ? x.w : 0u);
                            if ((left == 4 && t + 4 < d) && ((x.x ^ y) >> 22) == 0u) continue;      // no change: the usual case
                            change(x.x, x.y, t);
                            if (left > 1) change(x.y, x.z, t + 1);
                            if (left > 2) change(x.z, x.w, t + 2);
                            if (left > 3) change(x.w, y, t + 3);
                        }
                    } else {
                        for (int t = g * seg_len + lane; t < e; t += 32) {
                            const unsigned int x = max(K[t], carry);
                            const unsigned int y = t + 1 < d ? max(K[t + 1], x) : 0u;
                            if (g > 0) K[t] = x;
                            change(x, y, t);
                        }
                    }
                }
            } else if (!IN_SMEM) {
                // What is left of a row may be long here (rows of equal or almost equal losses).  Its keys do not decrease, so between two
                // keys of the same digit nothing is read: first 1024 keys at a time, then 32.
                for (int u = warp; u < units; u += SEL_WARPS) {
                    const int r = segs == 1 ? u : u / segs, g = u - r * segs;
                    const unsigned int* K = keys + (size_t)r * ldk;
                    const int b = row_lt[r], e = row_le[r];
                    auto digit = [&](int t) { return t < e ? (int)((K[t] >> shift) & dmask) : -1; };
                    auto change = [&](int t, int f, int fn) {      // key t ends a run of digit f
                        if (f == fn) return;
                        atomicAdd(&sh.hist[f], (Count)(t + 1));
                        if (fn >= 0) atomicAdd(&sh.hist[fn], (Count)0 - (Count)(t + 1));
                    };
                    auto scan = [&](int from, int to) {
                        for (int t = from + lane; t < to; t += 32) change(t, digit(t), digit(t + 1));
                    };
                    if (g == 0 && b > 0 && b < e && lane == 0) atomicAdd(&sh.hist[digit(b)], (Count)0 - (Count)b);
                    if (e - b <= 256) {
                        if (g == 0) scan(b, e);
                        continue;
                    }
                    for (int64_t p0 = (int64_t)b + (int64_t)g * 1024; p0 < e; p0 += (int64_t)segs * 1024) {
                        const int from = (int)p0, to = (int)min(p0 + 1024, (int64_t)e);
                        const int whole = digit(to - 1);
                        if (digit(from) == whole) {
                            if (lane == 0) change(to - 1, whole, digit(to));
                            continue;
                        }
                        const int x = min(from + 32 * lane, to), y = min(x + 32, to);      // this lane's piece
                        const int last = x < to ? digit(y - 1) : -1;
                        const bool same = x == to || digit(x) == last;
                        if (same && x < to) change(y - 1, last, digit(y));
                        unsigned int todo = __ballot_sync(0xffffffffu, !same);
                        if (__popc(todo) > 8) {                    // (pieces one after the other would cost more than reading all)
                            for (int t = from + lane; t < to; t += 32)
                                if (todo >> ((t - from) >> 5) & 1u) change(t, digit(t), digit(t + 1));
                        } else {
                            for (; todo; todo &= todo - 1) {
                                const int at = from + 32 * (__ffs(todo) - 1);
                                scan(at, min(at + 32, to));
                            }
                        }
                    }
                }
            } else {
                for (int u = warp; u < nr; u += SEL_WARPS) {      // what is left of a row is short: one warp per row
                    const unsigned int* K = keys + (size_t)u * ldk;
                    const int b = row_lt[u], e = row_le[u];
                    for (int t = b + lane; t < e; t += 32) {
                        const int f = (int)((K[t] >> shift) & dmask);
                        const int fn = t + 1 < e ? (int)((K[t + 1] >> shift) & dmask) : -1;
                        if (t == b && b > 0) atomicAdd(&sh.hist[f], (Count)0 - (Count)b);
                        if (f != fn) {
                            atomicAdd(&sh.hist[f], (Count)(t + 1));
                            if (fn >= 0) atomicAdd(&sh.hist[fn], (Count)0 - (Count)(t + 1));
                        }
                    }
                }
            }
            __syncthreads();
            Count a = sh.hist[2 * tid], b = sh.hist[2 * tid + 1];
            if (G > 1) {
                Count* bins = ghist + pass * SEL_BINS + 2 * tid;
                if (a) atomicAdd(bins, a);
                if (b) atomicAdd(bins + 1, b);
                if (!grid_barrier(&st->arrived, G * ++barrier_no, wait_limit)) {      // (all blocks of a cooperative launch are resident)
                    for (int r = tid; r < nr; r += SEL_THREADS) counts[r0 + r] = COUNT_TIMED_OUT;
                    return;
                }
                if constexpr (sizeof(Count) == 4) {
                    const uint2 v = __ldcg(reinterpret_cast<const uint2*>(bins));
                    a = v.x; b = v.y;
                } else {
                    a = __ldcg(bins); b = __ldcg(bins + 1);
                }
            }
            sh.hist[2 * tid] = 0; sh.hist[2 * tid + 1] = 0;
            pick_digit(a, b, sh);
            prefix |= sh.digit << shift;
            // narrow every row to the keys that share the prefix: one thread per row, both ends in one loop
            for (int r = tid; r < nr; r += SEL_THREADS) {
                const unsigned int* K = keys + (size_t)r * ldk;
                const unsigned int want = prefix >> shift;
                int lo0 = row_lt[r], hi0 = row_le[r], lo1 = lo0, hi1 = hi0;
                while (lo0 < hi0 || lo1 < hi1) {
                    if (lo0 < hi0) { const int m = (lo0 + hi0) >> 1; if ((K[m] >> shift) < want) lo0 = m + 1; else hi0 = m; }
                    if (lo1 < hi1) { const int m = (lo1 + hi1) >> 1; if ((K[m] >> shift) <= want) lo1 = m + 1; else hi1 = m; }
                }
                row_lt[r] = lo0; row_le[r] = lo1;
            }
            __syncthreads();
        }
    }
    const Count rem = sh.rem;                             // of the keys equal to the k-th, this many are taken, in row order
    const bool all_ties = k == 0 || rem == (Count)sh.digit_count;
    // ---- counts; ties are handed out by row (only when not all of them are taken)
    if (tid == 0) sh.before = 0;
    if (!all_ties && G > 1) {
        Count mine = 0;
        for (int r = tid; r < nr; r += SEL_THREADS) mine += (Count)(row_le[r] - row_lt[r]);
        const Count total = block_scan(mine, sh);
        if (tid == SEL_THREADS - 1) st->ties[blockIdx.x] = total;
        if (!grid_barrier(&st->arrived, G * ++barrier_no, wait_limit)) {
            for (int r = tid; r < nr; r += SEL_THREADS) counts[r0 + r] = COUNT_TIMED_OUT;
            return;
        }
        Count b = 0;
        for (int q = tid; q < (int)blockIdx.x; q += SEL_THREADS) b += (Count)__ldcg(st->ties + q);
        const Count lower = block_scan(b, sh);
        if (tid == SEL_THREADS - 1) sh.before = lower;
    }
    __syncthreads();
    for (int q = 0; q < nr; q += SEL_THREADS) {
        const int r = q + tid;
        int take = r < nr ? row_le[r] - row_lt[r] : 0;
        if (!all_ties) {
            const Count incl = block_scan((Count)take, sh), before = sh.before;
            const Count first = before + incl - (Count)take;      // equal keys in rows before this one
            const Count left = rem > first ? rem - first : 0;
            if (left < (Count)take) take = (int)left;
            __syncthreads();
            if (tid == SEL_THREADS - 1) sh.before = before + incl;
            __syncthreads();
        }
        if (r < nr) {
            const int n = row_lt[r] + take;
            row_lt[r] = n;
            counts[r0 + r] = n;
        }
    }
    __syncthreads();
    // ---- mask: 1, then 0 at the first counts[r] entries of the row's order
    const size_t bytes = (size_t)nr * d;
    uint8_t* M = mask + (size_t)r0 * d;
    if (IN_SMEM) {                                        // built where the keys were, written out in 16-byte pieces
        const int skew = (int)(reinterpret_cast<uintptr_t>(M) & 15u);
        uint8_t* S = reinterpret_cast<uint8_t*>(skeys) + skew;
        uint4* S4 = reinterpret_cast<uint4*>(skeys);
        const int n16 = (int)((bytes + skew + 15) >> 4);
        for (int q = tid; q < n16; q += SEL_THREADS) S4[q] = make_uint4(0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u);
        __syncthreads();
        for (int u = warp; u < units; u += SEL_WARPS) {
            const int r = u / segs, g = u - r * segs;
            const int e = min(row_lt[r], (g + 1) * seg_len);
            const int32_t* P = order + (size_t)(r0 + r) * d;
            for (int t = g * seg_len + lane; t < e; t += 256) {      // eight loads in flight per lane
                int j[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) j[q] = t + 32 * q < e ? __ldg(P + t + 32 * q) : -1;
#pragma unroll
                for (int q = 0; q < 8; ++q) if (j[q] >= 0 && j[q] < d) S[(size_t)r * d + j[q]] = 0;
            }
        }
        __syncthreads();
        uint8_t* base = M - skew;
        for (int q = tid; q < n16; q += SEL_THREADS) {
            const int lo = 16 * q, hi = lo + 16;
            if (lo >= skew && (size_t)hi <= bytes + skew) *reinterpret_cast<uint4*>(base + lo) = S4[q];
            else
                for (int x = max(lo, skew); x < hi && (size_t)x < bytes + skew; ++x) base[x] = reinterpret_cast<uint8_t*>(skeys)[x];
        }
    } else {
        const size_t head = min((size_t)((0 - reinterpret_cast<uintptr_t>(M)) & 15u), bytes), n16 = (bytes - head) >> 4;
        for (size_t x = tid; x < n16; x += SEL_THREADS)
            reinterpret_cast<uint4*>(M + head)[x] = make_uint4(0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u);
        if (tid < head) M[tid] = 1;
        for (size_t x = head + 16 * n16 + tid; x < bytes; x += SEL_THREADS) M[x] = 1;
        __syncthreads();
        for (int u = warp; u < units; u += SEL_WARPS) {
            const int r = u / segs, g = u - r * segs;
            const int e = min(row_lt[r], (g + 1) * seg_len);
            for (int t = g * seg_len + lane; t < e; t += 32) {
                const int j = order[(size_t)(r0 + r) * d + t];
                if (j >= 0 && j < d) M[(size_t)r * d + j] = 0;
            }
        }
    }
}

size_t select_workspace_bytes(int rows, int d) {
    return round_up((size_t)rows * d * 4, 256) + round_up(sizeof(SelectState), 256) + 2 * round_up((size_t)rows * 4, 256) +
           ((int64_t)rows * d < SEL_WIDE ? 0 : SEL_WIDE_BYTES);
}

obc_status select_launch(const float* loss, const int32_t* order, int rows, int d, int64_t k, int32_t* counts,
                         uint8_t* mask, void* ws, cudaStream_t stream, int wait_limit) {
    DeviceInfo di;
    const obc_status ds = device_info(&di);
    if (ds != OBC_OK) return ds;
    char* p = reinterpret_cast<char*>(ws);
    unsigned int* gkeys = reinterpret_cast<unsigned int*>(p); p += round_up((size_t)rows * d * 4, 256);
    SelectState* st = reinterpret_cast<SelectState*>(p); p += round_up(sizeof(SelectState), 256);
    int* glt = reinterpret_cast<int*>(p); p += round_up((size_t)rows * 4, 256);
    int* gle = reinterpret_cast<int*>(p); p += round_up((size_t)rows * 4, 256);
    // Blocks: one SM each, at least SEL_BLOCK_KEYS keys a block -- below that the barriers of a further block cost more than
    // its share of the scans saves -- and a single block (no barriers at all) up to SEL_ONE_BLOCK_KEYS.
    constexpr int64_t SEL_BLOCK_KEYS = 4096, SEL_ONE_BLOCK_KEYS = 12288;
    const int64_t n = (int64_t)rows * d;
    int64_t blocks = n <= SEL_ONE_BLOCK_KEYS ? 1 : (n + SEL_BLOCK_KEYS - 1) / SEL_BLOCK_KEYS;
    const int most = di.sm_count < SEL_MAX_BLOCKS ? di.sm_count : SEL_MAX_BLOCKS;
    if (blocks > most) blocks = most;
    if (blocks > rows) blocks = rows;
    int rpb = (int)((rows + blocks - 1) / blocks);
    const int grid = (rows + rpb - 1) / rpb;
    int segs = rpb >= 2 * SEL_WARPS ? 1 : 2 * SEL_WARPS / rpb;       // about two segments per warp, of 256 keys or more
    while (segs > 1 && d / segs < 256) --segs;
    const size_t key_bytes = (size_t)rpb * ((d + 3) & ~3) * 4 + 32;        // (the mask is built in the same space, shifted by up to 15 bytes)
    const bool wide = n >= SEL_WIDE, in_smem = key_bytes <= (size_t)SEL_SMEM && !wide;
    void* ghist = wide ? (void*)p : (void*)st->hist;
    unsigned long long kk = (unsigned long long)k;
    int limit = wait_limit == 0 ? GRID_BARRIER_LIMIT : (wait_limit < 0 ? 0 : wait_limit);
    if (grid > 1) OBC_CUDA_TRY(cudaMemsetAsync(st, 0, sizeof(SelectState), stream));
    if (wide && grid > 1) OBC_CUDA_TRY(cudaMemsetAsync(ghist, 0, SEL_WIDE_BYTES, stream));
    void* args[] = {&loss, &order, &rows, &d, &kk, &rpb, &segs, &gkeys, &glt, &gle, &st, &ghist, &counts, &mask, &limit};
    const void* kernel = in_smem ? (const void*)select_kernel<true, unsigned int>
                                 : (!wide ? (const void*)select_kernel<false, unsigned int> : (const void*)select_kernel<false, unsigned long long>);
    const size_t smem = in_smem ? key_bytes : 0;
    if (in_smem) OBC_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, SEL_SMEM));
    if (grid > 1) OBC_CUDA_TRY(cudaLaunchCooperativeKernel(kernel, dim3(grid), dim3(SEL_THREADS), args, smem, stream));
    else OBC_CUDA_TRY(cudaLaunchKernel(kernel, dim3(1), dim3(SEL_THREADS), args, smem, stream));
    count_launch();
    return OBC_OK;
}
// ---- allocation-free variant ----------------------------------------------------------------------------------
// Scratch for obc_select_global_mask_static: a fixed array in device memory that every GPU loading this library
// holds until the process exits.  Sized for OBC_SELECT_STATIC_MAX_KEYS loss entries and
// OBC_SELECT_STATIC_MAX_ROWS rows (16 MiB of keys + 128 KiB of per-row counters + the selection state).
constexpr size_t SELECT_STATIC_BYTES =
    ((size_t)OBC_SELECT_STATIC_MAX_KEYS * 4 + 255) / 256 * 256 + (sizeof(SelectState) + 255) / 256 * 256 +
    2 * (((size_t)OBC_SELECT_STATIC_MAX_ROWS * 4 + 255) / 256 * 256);
static __device__ __align__(256) unsigned char g_select_scratch[SELECT_STATIC_BYTES];

// Device address of the array on the CURRENT device.  In host code the array's name is only a stand-in, so
// the address is looked up once per device (with that device current) and cached.
static obc_status select_static_scratch(void** out) {
    static std::mutex mu;
    static void* ptrs[64] = {};
    int dev = 0;
    OBC_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= 64) return OBC_ERR_CUDA;
    std::lock_guard<std::mutex> lock(mu);
    if (!ptrs[dev]) {
        void* p = nullptr;
        OBC_CUDA_TRY(cudaGetSymbolAddress(&p, g_select_scratch));
        if (!p) return OBC_ERR_CUDA;
        ptrs[dev] = p;
    }
    *out = ptrs[dev];
    return OBC_OK;
}

}  // namespace obc

extern "C" obc_status obc_select_global_mask_static(const float* loss, const int32_t* order, int d_row, int d_col,
                                                    int64_t k, int32_t* counts, uint8_t* mask, obc_stream stream) {
    using namespace obc;
    if (d_row <= 0 || d_col <= 0 || !loss || !order || !counts || !mask) return OBC_ERR_INVALID_ARG;
    if (k < 0 || k > (int64_t)d_row * d_col) return OBC_ERR_INVALID_ARG;
    if (d_row > OBC_SELECT_STATIC_MAX_ROWS || (int64_t)d_row * d_col > (int64_t)OBC_SELECT_STATIC_MAX_KEYS)
        return OBC_ERR_STATIC_SCRATCH;
    void* scratch = nullptr;
    const obc_status st = select_static_scratch(&scratch);
    if (st != OBC_OK) return st;
    // every launch sequence re-initialises the selection state and overwrites the keys / counters it reads
    return select_launch(loss, order, d_row, d_col, k, counts, mask, scratch, (cudaStream_t)stream);
}
