// Warp-specialised TMA sweep, tile shape 6 (two y-adjacent points per thread, two planes at a time; see WsShape
// in tdks_tma.cuh), compiled on its own so that the shapes build in parallel.
#include "tdks_tma.cuh"

namespace tdks {
template cudaError_t launch_ws_shape<6>(int, int, int, int, const SweepMaps &, const SweepParams &, int,
                                          cudaStream_t);
template cudaError_t launch_ws_batch_shape<6>(int, int, int, const BatchSweepArgs &, cudaStream_t);
}  // namespace tdks
