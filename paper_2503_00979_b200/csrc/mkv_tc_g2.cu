#include "mkv_tc_kernel.cuh"

namespace mkv {
template cudaError_t tc_launch_group<2>(TcPlan *, const DecodeArgs &, cudaStream_t);
}
