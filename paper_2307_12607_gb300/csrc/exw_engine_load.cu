// exw_engine_load.cu -- the engine kernel with loader warps (launches with a stream that TMA cannot stage).
#include "exw_engine_kernel.cuh"

namespace exw {

cudaError_t launch_engine_load(const EngineParams &ep, bool fill, int shape, int grid, cudaStream_t s) {
    return launch_engine_as<true>(ep, fill, shape, grid, s);
}

}  // namespace exw
