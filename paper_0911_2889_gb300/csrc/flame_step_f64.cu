// FP64 launchers of the step's passes A and C and twiddle tables.
#include "flame_step_ops.cuh"

namespace flame {
template cudaError_t Ops<double>::init_kappa(double *, const StepArgs &, cudaStream_t);
template cudaError_t Ops<double>::init_twiddles3(double2 *, int, cudaStream_t);
template cudaError_t Ops<double>::passA(const FlameDesc &, cudaStream_t, int, const CUtensorMap *);
template cudaError_t Ops<double>::passA_batch(const FlameDesc *, int, const StepArgs &, cudaStream_t, int);
template cudaError_t Ops<double>::passC(const FlameDesc &, cudaStream_t);
template cudaError_t Ops<double>::passC_batch(const FlameDesc *, int, const StepArgs &, cudaStream_t, bool, bool);
template cudaError_t Ops<double>::passCA(const FlameDesc &, cudaStream_t, const CUtensorMap *);
template void Ops<double>::tiles(const StepArgs &, int, int *, int *);
}  // namespace flame
