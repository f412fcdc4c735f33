// fused_fp64.cu -- the fused Arnoldi cycle (fused.cuh) with an FP64 basis, and the rule that says
// which solves it takes.
#include "fused.cuh"

namespace gg {

cudaError_t launch_arnoldi_fp32(const CycleArgs& a, int jmax, bool defl, cudaStream_t st);
cudaError_t launch_arnoldi_bf16(const CycleArgs& a, int jmax, bool defl, cudaStream_t st);

// CGS2 or the one-reduction MGS, EBP deflation by aggregates or none (no projector, no dense
// deflation space); BF16 bases with CGS2.  Against one kernel per phase (CGS2, FP64, 9-point
// stencils): 51 to 35 us a step at 4,225 unknowns, 152 to 98 us at 262k; thread-per-row CSR, 238k
// unknowns: 112 to 75 us; long rows (3-D hexahedra, 275k unknowns): 196 to 190 us; BF16 basis,
// 362k unknowns: 92 to 85 us.
bool arnoldi_fusable(const CycleArgs& a) {
  if (a.proj || a.op.defl.qd != 0 || a.ldv % kArnUnit != 0 || a.m + 1 > kMaxK) return false;
  if (a.ortho != GMRES_ORTHO_CGS2 && !(a.ortho == GMRES_ORTHO_MGS_LOWSYNC && a.prec != P_BF16))
    return false;
  const int r = a.op.defl.r;
  // with deflation: the pieces split at this kernel's block rows (built at setup for a
  // grid of min(units, SMs) blocks)
  if (r > 0 && (!a.op.defl.blk_piece_start ||
                a.op.defl.blk_grid != (int)std::min<long long>(a.ldv / kArnUnit, a.sms)))
    return false;
  // the FP32 coarse solve of the FP32 one-reduction step
  if (r > 0 && a.prec == P_FP32 && !a.op.defl.tinv32) return false;
  const long long rs = a.prec == P_FP64 ? arn_super_rows(r, sizeof(double))
                                        : arn_super_rows(r, sizeof(float));
  // c (r doubles) lives where w and u_j do
  const size_t esz = a.prec == P_FP64 ? sizeof(double) : sizeof(float);
  return rs >= kArnUnit && (size_t)r * sizeof(double) <= 2 * (size_t)rs * esz;
}

bool arnoldi_fixed(const CycleArgs& a) {
  return a.prec == P_FP64 && !(a.ortho == GMRES_ORTHO_MGS_LOWSYNC &&
                               a.dot_arith == GMRES_DOT_DF32 && a.op.dia.nd > 0);
}

cudaError_t launch_arnoldi(const CycleArgs& a, int jmax, bool defl, cudaStream_t st) {
  switch (a.prec) {
    case P_FP64: return Arn<double, double>::launch(a, jmax, defl, st);
    case P_FP32: return launch_arnoldi_fp32(a, jmax, defl, st);
    default: return launch_arnoldi_bf16(a, jmax, defl, st);
  }
}

}  // namespace gg
