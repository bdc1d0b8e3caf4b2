// exw_engine.cu -- the engine kernel of launches whose windows TMA stages (or no one: tiles from global memory).
#include "exw_engine_kernel.cuh"

namespace exw {

cudaError_t launch_engine(const EngineParams &ep, bool fill, int shape, int grid, cudaStream_t s) {
    return launch_engine_as<false>(ep, fill, shape, grid, s);
}

}  // namespace exw
