// Flooding slot decoder, thread slots end to end in a warp: instances for FP16 messages, upper clamp of |Q| at phi(X) applied.
#include "flood_packed_kernel.cuh"

namespace ldpc {
template cudaError_t flood_packed_launch<__half, true>(const FloodPlan &, cudaStream_t);
}  // namespace ldpc
