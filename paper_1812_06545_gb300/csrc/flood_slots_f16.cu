// Flooding slot decoder: instances for FP16 messages.
#include "flood_slots_kernel.cuh"

namespace ldpc {
template cudaError_t flood_slots_launch<__half, false>(const FloodPlan &, cudaStream_t);
}  // namespace ldpc
