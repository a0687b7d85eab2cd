// The blocked row engine with 512 threads per row of up to 6144 columns (a file per variant: they compile in parallel).
#include "row_engine_blocked.cuh"

namespace obc {

obc_status blk_launch_512_12(const FlushMaps& zmaps, const EngineArgs& a, int blocks, size_t smem, int sm_count, cudaStream_t stream) {
    return blk_launch<512, 12>(zmaps, a, blocks, smem, sm_count, stream);
}

}  // namespace obc
