// Flooding slot decoder: instances for FP16 messages.
#include "flood_slots_kernel.cuh"

namespace ldpc {
template cudaError_t flood_slots_launch<__half, false>(int, int, const FloodArgs &, size_t, int, int, cudaStream_t);
}  // namespace ldpc
