// FP32 (FLAME_FP32_MIXED) launchers of the passes on the public grid: steps
// that record the surface area.
#include "flame_ops.cuh"

namespace flame {
template cudaError_t Ops<float>::passA_full(const FlameDesc &, cudaStream_t, const CUtensorMap *);
template cudaError_t Ops<float>::passB_area(const FlameDesc &, cudaStream_t);
template cudaError_t Ops<float>::passC_full(const FlameDesc &, cudaStream_t);
}  // namespace flame
