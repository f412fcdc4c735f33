// fused_bf16.cu -- the fused Arnoldi cycle (fused.cuh) with a BF16 basis.
#include "fused.cuh"

namespace gg {

cudaError_t launch_arnoldi_bf16(const CycleArgs& a, int jmax, bool defl, cudaStream_t st) {
  return Arn<__nv_bfloat16, float>::launch(a, jmax, defl, st);
}

}  // namespace gg
