// FP32 (FLAME_FP32_MIXED) launcher of pass C fused with the next pass A.
#include "flame_step_ops.cuh"

namespace flame {
template cudaError_t Ops<float>::passCA(const FlameDesc &, cudaStream_t, const CUtensorMap *);
}  // namespace flame
