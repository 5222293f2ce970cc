// Warp-specialised TMA sweep, tile shape 7 (2 x 2 points per thread, complex64; see WsShape in
// tdks_tma.cuh), compiled on its own so that the shapes build in parallel.
#include "tdks_tma.cuh"

namespace tdks {
template cudaError_t launch_ws_shape<7>(int, int, int, int, const SweepMaps &, const SweepParams &, int,
                                          cudaStream_t);
template cudaError_t launch_ws_batch_shape<7>(int, int, int, const BatchSweepArgs &, cudaStream_t);
}  // namespace tdks
