// Flooding slot decoder: instances for FP32 messages.
#include "flood_slots_kernel.cuh"

namespace ldpc {
template cudaError_t flood_slots_launch<float, false>(const FloodPlan &, cudaStream_t);
}  // namespace ldpc
