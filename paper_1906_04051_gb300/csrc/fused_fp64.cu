// fused_fp64.cu -- the fused Arnoldi cycle (fused.cuh) with an FP64 basis, and the rule that says
// which solves it takes.
#include <climits>

#include "fused.cuh"

namespace gg {

cudaError_t launch_arnoldi_fp32(const CycleArgs& a, int jmax, bool defl, cudaStream_t st);
cudaError_t launch_arnoldi_bf16(const CycleArgs& a, int jmax, bool defl, cudaStream_t st);

// Most rows (padded) up to which the fused cycle is the faster one; us a step against one kernel
// per phase, 45 columns, no deflation (nd: diagonals):
//   FP64, nd 5 to 27, CGS2   33k 45 / 63 (27), 1M 204 / 309 (9), 276 / 362 (27),
//                            4.1M 1006 / 1209 (27), 16M 2792 / 3855 (9)
//   FP32, CGS2               nd 9: 2.9M 252 / 267, 4M 356 / 355; nd 7: 2.1M 183 / 199, 3M 286 / 282;
//                            nd 19: 0.78M 84 / 105, 1.4M 157 / 155; nd 27: 0.88M 110 / 125,
//                            1M 136 / 133
//   FP32, one reduction      nd 9: 1M 64 / 101, 16M 856 / 959; nd 27: 2.7M 261 / 261
//   BF16, CGS2               nd 9: 2M 163 / 179, 2.6M 210 / 214; nd 7: 2.1M 176 / 179, 3M 285 / 234;
//                            nd 19: 0.78M 92 / 99, 1.4M 186 / 151; nd 27: 0.7M 100 / 104,
//                            0.88M 124 / 118
// CSR, 9 entries a row, numbered tile by tile, and at random (columns scattered):
//   FP64, CGS2               4.5M 1032 / 1128       1.5M 444 / 447, 2M 578 / 575
//   FP64, one reduction      4.5M 729 / 855         1.5M 351 / 352, 2M 460 / 450
//   FP32, CGS2               1.2M 142 / 144         0.49M 90 / 94, 0.72M 129 / 119
//   FP32, one reduction      2.6M 199 / 210         0.72M 102 / 104, 1M 140 / 129
//   BF16, CGS2               1M 107 / 113           0.36M 74 / 76, 0.49M 89 / 87
// long rows (27 entries by tiles or at random; the hexahedra's up to 125, lexicographic):
//   FP64                     0.44M 174 / 188        0.2M 118 / 120, 0.22M 130 / 125
//                            (hexahedra 275k 173 / 185, 531k 300 / 283)
//   FP32                     0.44M 86 / 97          0.2M 77 / 82, 0.22M 85 / 84
//   BF16                     0.34M 68 / 84          0.2M 79 / 83, 0.22M 87 / 85
//                            (hexahedra 275k 122 / 119)
// Past these sizes the phases stream: the per-phase kernels have more loads in flight than one
// block of 16 warps per multiprocessor, for the SpMV above all (so the limits fall with its
// share: many diagonals, long rows, gathers all over the vector).  FP64 dots and updates stay
// ahead, being fixed point here and FP64 multiply-adds there.
long long fused_rows(const CycleArgs& a) {
  const bool cgs2 = a.ortho == GMRES_ORTHO_CGS2;
  if (const int nd = a.op.dia.nd) {
    if (a.prec == P_FP64 || !cgs2) return LLONG_MAX;
    return a.prec == P_BF16 ? std::min(2100000, 20000000 / nd) : std::min(2600000, 25000000 / nd);
  }
  if (a.op.vec) return a.op.scattered ? 190000 : a.prec == P_BF16 ? 200000 : 350000;
  if (a.prec == P_FP64) return a.op.scattered ? 1500000 : 4500000;
  if (!cgs2) return a.op.scattered ? 750000 : 2600000;
  if (a.prec == P_BF16) return a.op.scattered ? 400000 : 1050000;
  return a.op.scattered ? 500000 : 1200000;
}

// CGS2 or the one-reduction MGS, EBP deflation by aggregates or none (no projector, no dense
// deflation space); BF16 bases with CGS2.
bool arnoldi_fusable(const CycleArgs& a) {
  if (a.ldv > fused_rows(a)) return false;
  // GMRES(1) in FP64: the exponent of u_0 costs a grid barrier and a pass over it in every cycle (10
  // cycles, us, fused / phases: 10,000 rows CGS2 883 / 849, CSR 879 / 814; GMRES(2) 652 / 665)
  const bool dia = a.op.dia.nd > 0, cgs2 = a.ortho == GMRES_ORTHO_CGS2;
  if (a.m < 2 && a.prec == P_FP64 && (cgs2 || !dia)) return false;
  if (a.proj || a.op.defl.qd != 0 || a.ldv % kArnUnit != 0 || a.m + 1 > kMaxK) return false;
  if (!cgs2 && !(a.ortho == GMRES_ORTHO_MGS_LOWSYNC && a.prec != P_BF16))
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
