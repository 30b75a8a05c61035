// FP32 (FLAME_FP32_MIXED) launchers of the step's pass C.
#include "flame_step_ops.cuh"

namespace flame {
template cudaError_t Ops<float>::passC(const FlameDesc &, cudaStream_t);
template cudaError_t Ops<float>::passC_batch(const FlameDesc *, int, const StepArgs &, cudaStream_t, bool, bool);
}  // namespace flame
