// Entry points for tests that make bounded device-side waits run out: the library's launchers with arguments that the C ABI does
// not offer.  Compiled by the tests against libobc.so.
#include "common.cuh"

extern "C" int shim_prune_trace(const float* W, int ldw, int rows, int d, const float* Hinv, int ldhi, int32_t* order, float* loss,
                                int32_t* row_status, void* ws, size_t ws_bytes, int threads, int stop_tile, void* stream) {
    obc::EngineOpts eo = {OBC_ENGINE_BLOCKED, threads, 0, 0};
    eo.stop_tile = stop_tile;
    return obc::engine_prune_trace(W, ldw, rows, d, 0, rows, Hinv, ldhi, d, order, loss, nullptr, row_status, ws, ws_bytes, eo, (cudaStream_t)stream);
}

extern "C" int shim_select(const float* loss, const int32_t* order, int rows, int d, long long k, int32_t* counts, uint8_t* mask, void* ws,
                           int wait_limit, void* stream) {
    return obc::select_launch(loss, order, rows, d, k, counts, mask, ws, (cudaStream_t)stream, wait_limit);
}
