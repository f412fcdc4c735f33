// fused_fp32.cu -- the fused Arnoldi cycle (fused.cuh) with an FP32 basis.
#include "fused.cuh"

namespace gg {

cudaError_t launch_arnoldi_fp32(const CycleArgs& a, int jmax, bool defl, cudaStream_t st) {
  return Arn<float, float>::launch(a, jmax, defl, st);
}

}  // namespace gg
