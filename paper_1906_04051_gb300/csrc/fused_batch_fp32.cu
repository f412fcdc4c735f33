// fused_batch_fp32.cu -- the fused Arnoldi cycles of a batch (fused.cuh), a cluster per system.
#include "fused.cuh"

namespace gg {

size_t arnoldi_args_fp32(const CycleArgs& a, bool defl, void* dst) {
  using K = Arn<float, float>;
  if (dst) *static_cast<K::Args*>(dst) = K::fill(a, a.m, defl);
  return sizeof(K::Args);
}

cudaError_t launch_arnoldi_batch_fp32(const FusedBatch& f, int clusters, int lo, int hi, int G,
                                    cudaStream_t st) {
  return Arn<float, float>::batch(f, clusters, lo, hi, G, st);
}

}  // namespace gg
