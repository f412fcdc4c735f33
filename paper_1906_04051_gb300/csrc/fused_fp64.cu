// fused_fp64.cu -- the fused Arnoldi cycle (fused.cuh) with an FP64 basis, and the rule that says
// which solves it takes.
#include <climits>

#include "fused.cuh"

namespace gg {

cudaError_t launch_arnoldi_fp32(const CycleArgs& a, int jmax, bool defl, cudaStream_t st);
cudaError_t launch_arnoldi_bf16(const CycleArgs& a, int jmax, bool defl, cudaStream_t st);

// Most rows (padded) up to which the fused cycle is the faster one; us a step against one kernel
// per phase, 40 to 50 columns:
//   FP64 diagonals, CGS2     4,225 rows 35 / 51, 262k 98 / 152, 4M 652 / 900
//   FP64 CSR, CGS2           238k 77 / 133, 2.25M 508 / 595, 4M 871 / 913
//   FP64 CSR, one reduction  238k 61 / 115, 2.25M 395 / 472, 4M 635 / 700
//   FP32 diagonals, CGS2     1.44M 121 / 148, 2.9M 240 / 243, 3.2M 280 / 266
//   FP32 CSR, CGS2           90k 38 / 51, 1M 111 / 119, 2.6M 271 / 229
//   FP32 CSR, one reduction  90k 29 / 44, 2.6M 192 / 195, 4M 304 / 277
//   BF16 diagonals, CGS2     1M 95 / 107, 1.44M 124 / 137, 1.96M 171 / 167, 4M 361 / 289
//   long rows (hexahedra)    36k 48 / 66, 275k 173 / 185 (BF16 122 / 119), 531k 300 / 283,
//                            1.77M 907 / 782
// Past these sizes the phases stream: the per-phase kernels have more loads in flight than one
// block of 16 warps per multiprocessor, and with long rows the SpMV outweighs the rest of the
// step.  FP64 dots and updates stay ahead, being fixed point here and FP64 multiply-adds there.
long long fused_rows(const CycleArgs& a) {
  const bool csr = a.op.dia.nd == 0, cgs2 = a.ortho == GMRES_ORTHO_CGS2;
  if (a.op.vec) return a.prec == P_BF16 ? 200000 : 350000;
  if (a.prec == P_FP64) return csr ? 4500000 : LLONG_MAX;
  if (csr) return cgs2 ? 1200000 : 2600000;
  if (!cgs2) return LLONG_MAX;
  return a.prec == P_BF16 ? 1700000 : 2600000;
}

// CGS2 or the one-reduction MGS, EBP deflation by aggregates or none (no projector, no dense
// deflation space); BF16 bases with CGS2.
bool arnoldi_fusable(const CycleArgs& a) {
  if (a.ldv > fused_rows(a)) return false;
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
