// exw_engine_load.cu -- the engine kernel with loader warps (launches with a stream that TMA cannot stage): 896 threads.
#define EXW_LAUNCH_ENGINE launch_engine_load
#define EXW_ENGINE_LOAD true
#include "exw_engine.cu"
