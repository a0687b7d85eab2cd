// Host side of the blocked row engine (row_engine_blocked.cuh): how a launch is laid out over the SMs, workspace, launch.
#include "row_engine_blocked.cuh"

namespace obc {

// ---- host side ---------------------------------------------------------------------------------------------
struct BlkPlan {
    int nt;            // threads per block
    int per_sm;        // blocks per SM the shared-memory split is made for
    size_t smem;       // dynamic shared memory per block
    int panel_floats;
    int ms;
    int g_vectors;     // overflow pending vectors per block in global memory (0 = none)
    int g_ld;          // their stride in floats
    int max_pending;   // limit on deferred updates
};

obc_status blk_launch_128_8(const FlushMaps& zmaps, const EngineArgs& a, int blocks, size_t smem, int sm_count, cudaStream_t stream);
obc_status blk_launch_256_8(const FlushMaps& zmaps, const EngineArgs& a, int blocks, size_t smem, int sm_count, cudaStream_t stream);
obc_status blk_launch_512_4(const FlushMaps& zmaps, const EngineArgs& a, int blocks, size_t smem, int sm_count, cudaStream_t stream);
obc_status blk_launch_512_8(const FlushMaps& zmaps, const EngineArgs& a, int blocks, size_t smem, int sm_count, cudaStream_t stream);
obc_status blk_launch_512_12(const FlushMaps& zmaps, const EngineArgs& a, int blocks, size_t smem, int sm_count, cudaStream_t stream);

// All blocks' overflow vectors together: the size of L2, which they share with the planes and the streamed triangles.  (Only the
// longest rows reach the limit; when it was chosen, 48 / 64 / 80 / 110 MB at 128 rows x 4608 took 249 / 220 / 202 / 181 ms; the case
// takes 141 ms now.)
constexpr size_t BLK_L2_PANEL_BUDGET = (size_t)110 << 20;

// One slot per thread on chip, at most 256 of them: 512 threads could hold 309, which measured the same (256 / 309 slots, pruning, OBQ:
// 64 x 1152 4.71 / 4.70, 5.15 / 5.10 ms, 148 x 2304 23.0 / 23.2, 24.5 / 24.8, 64 x 3072 36.1 / 36.0, 38.9 / 39.0), and so rows from 257
// columns on have passes with every thread count.
static int blk_pick_ms(int d, size_t panel_bytes, int nt) {
    const int most = nt < 256 ? nt : 256;
    int ms = d < most ? d : most;
    if (ms < 2) ms = 2;
    while (ms > 2 && blk_tail_bytes(ms) > panel_bytes) --ms;
    return ms;
}

// Threads per block and blocks per SM by row length: short rows are bound by the latency of a step, so
// several of them share an SM; long rows need the shared memory for pending vectors.
// row_count = rows of the launch (0 = many).
static bool blk_plan(int d, bool wfull, const DeviceInfo& di, BlkPlan* out, bool nm = false, int bc = 0,
                     int row_count = 0, int threads = 0, int mode = MODE_PRUNE) {
    const int cap = (d + 3) & ~3;
    int nt = threads;
    if (nt != 128 && nt != 256 && nt != 512) {
        // measured on 1184 rows (ms with 128 / 256 / 512 threads): pruning 560 6.72 / 7.45 / 12.1, 640 9.65 / 9.61 / 14.7, 704 12.4 / 11.5 /
        // 17.2, 1152 - / 38.5 / 43.3, 1280 - / 53.8 / 52.8; OBQ 640 11.0 / 11.2, 1280 57.1 / 57.1; replay before OBQ 560 7.25 / 7.24
        nt = d <= 624 ? 128 : (d <= 1216 ? 256 : 512);
        // few rows (one per SM pair at most): nothing to share an SM with, the larger block is faster per row (260 rows, 128 / 256
        // threads: 320 0.75 / 0.73, 576 2.42 / 1.98)
        if (nt == 128 && row_count > 0 && row_count <= 2 * di.sm_count) nt = 256;
        // at most one row per SM, which then has all its shared memory: 512 threads (passes on tcgen05) win from d_col ~ 1050 on (64
        // rows, 256 / 512: pruning 960 3.46 / 3.55, 1152 5.08 / 4.85, OBQ 960 3.88 / 3.95, 1152 5.65 / 5.33, replay before OBQ 960 3.49 /
        // 3.63, 1152 5.16 / 4.96), blocks of 4 at 736, blocks of 8 at 896, a replay alone, which is all passes, from 450 on (64
        // rows: 320 0.36 / 0.35, 480 0.59 / 0.52, 704 1.04 / 0.85)
        const int whole_sm = mode == MODE_REPLAY ? 448 : (bc == 4 ? 736 : bc == 8 ? 896 : 1056);
        if (nt == 256 && row_count > 0 && row_count <= di.sm_count && d > whole_sm) nt = 512;
    }
    if (nt == 128 && cap > 1024) nt = 256;
    if (nt == 256 && cap > 2048) nt = 512;
    BlkPlan p;
    p.nt = nt;
    p.per_sm = 512 / nt;
    // at most one row per SM: all of its shared memory (more updates per pass, more slots on chip: 64 x 576 layer 2283 -> 2180 us).  Two such
    // calls on two streams then share no SM.  Half of it from 75 rows on would let them (two calls / one call of 100 rows, all -> half, ms: 576
    // 2.83 -> 2.07 / 1.41 -> 1.52, 704 3.93 -> 2.97 / 1.97 -> 2.17, 960 7.02 -> 5.86 / 3.58 -> 4.26): layers are solved one call after
    // another, so the single call decides.
    if (row_count > 0 && row_count <= di.sm_count) p.per_sm = 1;
    // 1 KB per resident block is reserved by the hardware; keep every block's share 128-byte aligned
    const size_t sm_total = (size_t)di.smem_optin + 1024;
    size_t share = (sm_total / p.per_sm - 1024) & ~(size_t)127;
    if (share > (size_t)di.smem_optin) share = (size_t)di.smem_optin;
    const size_t fixed = BLK_FIXED + blk_state_bytes(cap, wfull, nm, bc);
    const size_t min_panel = (size_t)4 * blk_ldz(cap);
    const size_t min_vectors = bc > 4 ? (size_t)bc : 4;         // (block pruning flushes whole blocks of bc updates)
    while (p.per_sm > 1 && share < fixed + min_vectors * min_panel) {     // too little room: fewer, larger blocks
        p.per_sm >>= 1;
        share = (sm_total / p.per_sm - 1024) & ~(size_t)127;
        if (share > (size_t)di.smem_optin) share = (size_t)di.smem_optin;
    }
    if (share < fixed + min_panel || share < fixed + blk_tail_bytes(2)) return false;
    p.smem = share;
    p.panel_floats = (int)((share - fixed) / 4);
    p.ms = blk_pick_ms(d, share - fixed, nt);
    // A replay alone that does not fit on chip from its start, or takes more than 224 slots there: four known eliminations off chip take less time
    // than four steps on chip until few slots are left (30 % / 95 % of a row, ms, on chip as soon as it fits / by this rule: 64 x 320
    // 0.247 / 0.201 and 0.520 / 0.522, 64 x 256 0.195 / 0.163 and 0.377 / 0.384, 600 x 160 0.216 / 0.173 and 0.455 / 0.400; 64 x 224 the
    // other way round, 0.151 / 0.155 and 0.300 / 0.311).
    if (mode == MODE_REPLAY && (d > p.ms || d > 224) && p.ms > (nt == 128 ? 64 : 128)) p.ms = nt == 128 ? 64 : 128;
    // Rows of one 512-thread block per SM: shared memory holds fewer pending vectors than a pass can apply (19 at d_col = 2304, 12
    // at 3072, 6 at 4608); further ones go to a global buffer small enough to stay in L2 (the triangle itself is streamed past
    // it with evict-first hints).
    p.g_ld = (cap + 15) & ~15;
    p.g_vectors = 0;
    p.max_pending = BLK_MAXB;
    if (p.nt == 512) {
        const int in_smem = p.panel_floats / blk_ldz(cap);
        int g = (int)(BLK_L2_PANEL_BUDGET / ((size_t)di.sm_count * p.g_ld * 4));
        if (bc == 8) {
            // (passes by mma.sync: their overflow vectors come 8 at a time and need staging space)
            if (g > 24) g = 24;
            g &= ~7;
            const size_t stage = (size_t)(p.nt / 32) * g * 16 * 4;
            if (in_smem < 16 && g >= 8 && share - fixed >= stage + 4 * min_panel) {
                p.g_vectors = g;
                p.panel_floats = (int)((share - fixed - stage) / 4);
            }
        } else {
            // as many updates per pass as it has accumulators and operand space for
            int groups = FT_GMAX;
            // 64 for rows of middling length: shorter ones hold nearly all of 48 in shared memory, for longer ones the steps between two
            // passes, which read them all from L2, cost more than the rarer passes save (148 rows, pruning, 48 / 64 updates: 1280
            // 6.75 / 6.78, 1536 9.88 / 9.72, 2304 23.9 / 23.1, 3072 49.3 / 47.0, 3584 74.0 / 72.6, 4096 107 / 109, 4608 156 / 157)
            // A replay alone reads them for four columns at a time: 64 from 1921 on (64 rows, 48 / 64: 1536 5.00 / 5.20, 1800 7.61 / 7.96, 2048 10.26 /
            // 10.11, 2304 14.4 / 14.0, 3072 28.9 / 27.6).
            // Blocks of 4 have less shared memory for them (six FP64 off-diagonals a block): 64 from 2049 to 2752 (32 / 148 rows, 48 : 64: 1536 6.72 :
            // 6.90 / 7.85 : 8.07, 2304 17.8 : 17.6 / 21.0 : 20.3, 2700 25.4 : 25.6 / 31.2 : 31.0, 2900 30.1 : 32.2 / 37.8 : 39.2, 3584 49.7 : 53.9).
            if (d <= (bc ? 2048 : mode == MODE_REPLAY ? 1920 : 1408) || d > (bc ? 2752 : 3840)) groups = 3;
            while (groups > 1 && (size_t)ft_stage_bytes(groups, FlushBufs{1, 1, 2}) + 1024 > share - fixed + 16 * (size_t)cap) --groups;
            if (d > p.ms && (size_t)ft_stage_bytes(1, FlushBufs{1, 1, 1}) + 1024 > share - fixed + 16 * (size_t)cap) return false;
            p.max_pending = 16 * groups;
            g &= ~7;                                               // (whole multiples of 8, as the plan reports them)
            const int want = (p.max_pending - in_smem + 7) & ~7;
            if (g > want) g = want;
            if (g >= 8) p.g_vectors = g;
        }
    }
    *out = p;
    return true;
}

// The largest grid any thread-count choice uses at this row length (threads per row are bounded below by the row
// length, see blk_plan).
static int blk_max_blocks(int d, const DeviceInfo& di) {
    const int cap = (d + 3) & ~3;
    return di.sm_count * (cap > 2048 ? 1 : (cap > 1024 ? 2 : 4));
}

// FP16 planes of the pending vectors of every 512-thread block (64 hi, 64 lo rows), the parked FP64 state of its row, and the
// slots' powers of two
static int blk_zld(int cap) { return (cap + 127) & ~127; }
size_t blk_plane_bytes(int blocks, int cap) {
    return round_up((size_t)blocks * 128 * blk_zld(cap) * sizeof(__half), 256) + round_up((size_t)blocks * cap * sizeof(double2), 256) + round_up((size_t)blocks * cap, 256);
}

size_t blocked_engine_workspace_bytes(int row_count, int d, const DeviceInfo& di) {
    // valid for every per-call choice: a row needs its private triangle whenever d exceeds the on-chip threshold,
    // and that threshold depends on the threads per row and on the per-row state the call keeps
    bool off_chip = false;
    const int nts[4] = {0, 128, 256, 512};
    for (int k = 0; k < 4; ++k)
        for (int nm = 0; nm < 2; ++nm) {
            BlkPlan p;
            if (!blk_plan(d, true, di, &p, nm != 0, false, row_count, nts[k])) continue;
            if (d > p.ms) off_chip = true;
        }
    if (!off_chip) return 256;
    const int cap = (d + 3) & ~3;
    int blocks = blk_max_blocks(d, di);
    // more rows than blocks: every block may also hold the row it starts for its neighbour (a second triangle),
    // plus the saved state and the flags of the hand-over
    const bool may_split = row_count == 0 || row_count > di.sm_count;
    if (row_count > 0 && row_count < blocks) blocks = row_count;
    const int gblocks = blocks < di.sm_count ? blocks : di.sm_count;     // overflow vectors: one block per SM only
    return round_up((size_t)blocks * (may_split ? 2 : 1) * tri_floats(cap) * sizeof(float), 256) +
           round_up((size_t)gblocks * BLK_MAXB * ((cap + 15) & ~15) * sizeof(float), 256) + blk_plane_bytes(gblocks, cap) +
           (may_split ? round_up((size_t)blocks * blk_split_stride(cap), 256) + round_up((size_t)blocks * sizeof(int), 256) : 0);
}

obc_status blocked_engine_plan(int d, int with_trace, int row_count, const EngineOpts& eo, int32_t* plan) {
    DeviceInfo di;
    obc_status st = device_info(&di);
    if (st != OBC_OK) return st;
    BlkPlan p;
    if (d > OBC_MAX_DCOL || !blk_plan(d, with_trace != 0, di, &p, false, false, row_count, eo.threads)) return OBC_ERR_UNSUPPORTED;
    const int mp = eo.max_pending;
    plan[0] = OBC_ENGINE_BLOCKED; plan[1] = p.nt; plan[2] = p.per_sm; plan[3] = p.ms; plan[4] = p.panel_floats;
    plan[5] = (mp >= 1 && mp < p.max_pending) ? mp : p.max_pending; plan[6] = di.sm_count; plan[7] = p.g_vectors;
    return OBC_OK;
}

obc_status blocked_engine_launch(EngineArgs a, void* ws, size_t ws_bytes, cudaStream_t stream) {
    DeviceInfo di;
    obc_status st = device_info(&di);
    if (st != OBC_OK) return st;
    a.cap = (a.d + 3) & ~3;
    if (a.d > OBC_MAX_DCOL) return OBC_ERR_UNSUPPORTED;
    BlkPlan p;
    const int bc = (a.block_c == 4 || a.block_c == 8) ? a.block_c : 0;      // block pruning: the block size
    if (!blk_plan(a.d, a.w_trace != nullptr, di, &p, a.nm_prune > 0, bc, a.row_count, a.opts.threads, a.mode))
        return OBC_ERR_UNSUPPORTED;
    a.ms = p.ms;
    a.panel_floats = p.panel_floats;
    const int mp = a.opts.max_pending;
    a.max_pending = (mp >= 1 && mp < p.max_pending) ? mp : p.max_pending;
    if (bc) {
        // the slots of a block must stay together: no on-chip tail (it compacts slot by slot), whole blocks per flush
        a.ms = 0;
        if (a.max_pending < bc) a.max_pending = bc;
        if (p.panel_floats / blk_ldz(a.cap) + p.g_vectors < bc) return OBC_ERR_UNSUPPORTED;
    }
    int blocks = di.sm_count * p.per_sm;
    if (a.row_count < blocks) blocks = a.row_count;
    a.Hws = nullptr;
    a.Gpan = nullptr;
    a.g_vectors = 0;
    a.g_ld = p.g_ld;
    a.ldp = a.cap;
    a.split = 0;
    a.split_state = nullptr; a.split_flags = nullptr; a.split_stride = 0;
    a.stop_tile = a.opts.stop_tile;
    a.Zws = nullptr; a.park = nullptr; a.zexp = nullptr; a.zld = blk_zld(a.cap);
    FlushMaps zmaps = {};
    if (a.d > a.ms) {
        // Shares of rows (equal work per block instead of whole waves): when there are more rows than blocks and they
        // do not divide evenly; not with the N:M pattern or block pruning, whose extra per-row state is not handed over.
        // With one row per SM (long rows) at any number of waves: measured 5.2 waves of 3072-column rows 428 -> 385 ms,
        // 10.1 waves 794 -> 757 ms, 5.2 waves of 2304-column rows 219 -> 194 ms, of 1536-column rows 75.8 -> 68.7 ms.
        // With several rows per SM only up to three waves: the pieces are smaller and the kernels with this code slower,
        // above all the forced-order ones (10.4 waves of 768-column rows: trace 50.5 -> 51.0 ms, replay + quantisation
        // 51.1 -> 55.3 ms; 5.1 waves of 704-column rows 39.5 -> 40.5 and 42.5 -> 48.9 ms; 3.4 waves of 1408-column rows
        // gain, 79.9 -> 70.9 ms, 5.7 waves of 1152-column rows do not).
        const bool want_split = a.row_count > blocks && a.row_count % blocks != 0 && (p.per_sm == 1 || a.row_count < 3 * blocks) &&
                                a.nm_prune == 0 && !bc && !(a.opts.flags & OBC_ENGINE_WHOLE_WAVES);
        const size_t tri = round_up((size_t)blocks * (want_split ? 2 : 1) * tri_floats(a.cap) * sizeof(float), 256);
        const size_t gpan = p.g_vectors ? round_up((size_t)blocks * p.g_vectors * p.g_ld * sizeof(float), 256) : 0;
        const size_t sst = want_split ? round_up((size_t)blocks * blk_split_stride(a.cap), 256) : 0;
        const size_t sfl = want_split ? round_up((size_t)blocks * sizeof(int), 256) : 0;
        const size_t planes = p.nt == 512 ? blk_plane_bytes(blocks, a.cap) : 0;
        if (!ws || !aligned256(ws) || ws_bytes < tri + gpan + planes + sst + sfl) return OBC_ERR_WORKSPACE;
        a.Hws = reinterpret_cast<float*>(ws);
        if (planes) {
            a.Zws = reinterpret_cast<__half*>(reinterpret_cast<char*>(ws) + tri + gpan);
            a.park = reinterpret_cast<double2*>(reinterpret_cast<char*>(a.Zws) + round_up((size_t)blocks * 128 * a.zld * sizeof(__half), 256));
            a.zexp = reinterpret_cast<signed char*>(a.park) + round_up((size_t)blocks * a.cap * sizeof(double2), 256);
            const int64_t groups = (int64_t)blocks * (want_split ? 2 : 1) * (((a.cap + 63) & ~63) >> 5);      // of 32 columns
            for (int k = 0; k < FT_GMAX; ++k)
                if (!make_tensor_map_3d(&zmaps.z[k], CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, a.Zws, a.zld, 64, 2 * (int64_t)blocks, 64, 16 * (k + 1), 2))
                    return OBC_ERR_CUDA;
            if (!make_tensor_map_3d(&zmaps.h128, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.Hws, 32, a.ldp, groups, 32, FT_M, 2) ||
                !make_tensor_map_3d(&zmaps.h32, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, a.Hws, 32, a.ldp, groups, 32, 32, 1))
                return OBC_ERR_CUDA;
        }
        if (p.g_vectors) {
            a.Gpan = reinterpret_cast<float*>(reinterpret_cast<char*>(ws) + tri);
            a.g_vectors = p.g_vectors;
        }
        if (want_split) {
            a.split = 1;
            a.split_state = reinterpret_cast<char*>(ws) + tri + gpan + planes;
            a.split_stride = blk_split_stride(a.cap);
            a.split_flags = reinterpret_cast<int*>(reinterpret_cast<char*>(ws) + tri + gpan + planes + sst);
        }
    }
    // Slots per thread of the 512-thread kernels: every one costs instructions in every step (4 against 12: 960 columns, one row per
    // SM, 7.7 -> 5.3 ms; 8 against 12: 256 x 2304 54 -> 48 ms).  (4 instead of 8 with 128 or 256 threads measured no faster.)
    auto launch = p.nt == 128 ? blk_launch_128_8 : p.nt == 256 ? blk_launch_256_8
                : (a.cap <= 2048 ? blk_launch_512_4 : (a.cap <= 4096 ? blk_launch_512_8 : blk_launch_512_12));
    return launch(zmaps, a, blocks, p.smem, di.sm_count, stream);
}

}  // namespace obc
