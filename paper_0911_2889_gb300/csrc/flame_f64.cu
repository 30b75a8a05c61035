// FP64 instantiation of the public grid's kernels and launchers (FLAME_FP64).
#include "flame_ops.cuh"

namespace flame {
extern template cudaError_t Ops<double>::passA(const FlameDesc &, cudaStream_t, int, const CUtensorMap *);
template cudaError_t Ops<double>::init_twiddles(double2 *, int, cudaStream_t);
template cudaError_t Ops<double>::rows_r2c(const double *, double2 *, int, int, const double2 *, const double2 *, cudaStream_t, int *);
template cudaError_t Ops<double>::rows_c2r(const double2 *, double *, int, int, const double2 *, const double2 *, cudaStream_t, int *);
template cudaError_t Ops<double>::cols(const double2 *, double2 *, int, int, int, int, int, const double2 *, cudaStream_t, int *);
template cudaError_t Ops<double>::box_from_spec(const double2 *, double2 *, double *, int, int, int, int, cudaStream_t, int *);
template cudaError_t Ops<double>::passA_full(const FlameDesc &, cudaStream_t, const CUtensorMap *);
template cudaError_t Ops<double>::passB_area(const FlameDesc &, cudaStream_t);
template cudaError_t Ops<double>::passC_full(const FlameDesc &, cudaStream_t);
template cudaError_t Ops<double>::area(const AdjDesc &, cudaStream_t);
template cudaError_t Ops<double>::adj_step(const AdjDesc &, cudaStream_t);
}  // namespace flame
