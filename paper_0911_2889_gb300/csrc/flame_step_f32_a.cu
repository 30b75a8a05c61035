// FP32 (FLAME_FP32_MIXED) launchers of the step's pass A and twiddle tables.
#include "flame_step_ops.cuh"

namespace flame {
template cudaError_t Ops<float>::init_twiddles3(float2 *, int, cudaStream_t);
template cudaError_t Ops<float>::passA(const FlameDesc &, cudaStream_t, int, const CUtensorMap *);
template cudaError_t Ops<float>::passA_batch(const FlameDesc *, int, const StepArgs &, cudaStream_t, int);
template void Ops<float>::tiles(const StepArgs &, int, int *, int *);
}  // namespace flame
