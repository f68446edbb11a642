// Flooding slot decoder, thread slots end to end in a warp: instances for FP32 messages.
#include "flood_packed_kernel.cuh"

namespace ldpc {
template cudaError_t flood_packed_launch<float, false>(const FloodPlan &, cudaStream_t);
}  // namespace ldpc
