// FP64 launchers of the step's pass B.
#include "flame_step_ops.cuh"

namespace flame {
template cudaError_t Ops<double>::passB(const FlameDesc &, cudaStream_t, int, const CUtensorMap *);
template cudaError_t Ops<double>::passB_batch(const FlameDesc *, int, const StepArgs &, cudaStream_t, int);
}  // namespace flame
