#include "mkv_tc_kernel.cuh"

namespace mkv {
template cudaError_t tc_launch_group<8>(TcPlan *, const DecodeArgs &, cudaStream_t);
}
