// Flooding slot decoder: instances for FP16 messages, upper clamp of |Q| at phi(X) applied.
#include "flood_slots_kernel.cuh"

namespace ldpc {
template cudaError_t flood_slots_launch<__half, true>(const FloodPlan &, cudaStream_t);
}  // namespace ldpc
