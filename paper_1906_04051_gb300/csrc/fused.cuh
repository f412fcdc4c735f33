// fused.cuh -- the Arnoldi steps of a restart cycle of deflated GMRES(m) in one persistent
// kernel: per step the SpMV w = A M^-1 v_j (Eq. 10 with Eqs. 16-17), the orthogonalisation
// (Eq. 13), ||w||, the plane rotations with the stopping tests (Eqs. 12, 14) and the coarse
// solve of the next step's preconditioner (Eq. 17: s' = U (|mu| T^-1 - I) U^T v_{j+1}).  The
// orthogonalisation is the paper's modified Gram-Schmidt projections in their one-reduction
// form or CGS2; the operator is in diagonal storage or CSR; the basis is FP64, FP32 or (CGS2)
// BF16.  Each precision is instantiated in a file of its own (fused_*.cu).
//
// One block of 16 warps per multiprocessor, launched cooperatively (every block resident).
// Block b owns a contiguous range of rows (a multiple of 128) for the whole cycle, taken in
// super-tiles of at most RS rows whose slices of w and u_j stay in shared memory.  A step:
//   1. SpMV of the super-tile's rows (diagonal storage; the coarse correction through the
//      A W rows, s' staged in shared memory): w into shared memory (and global memory when
//      the update reads it there), u_j next to it.  Step 0's diagonal part runs before the
//      programmatic-launch wait, overlapping the coarse-solve kernel that produces its s'.
//   2. Multi-dot g = V^T w and the new row of L (u_j . u_c), streamed from HBM against the
//      shared-memory slices, by row chunks over column groups (FP64: fixed point on the
//      integer pipe, fixed.cuh; double-FP32 on request).
//   3. Grid barrier 1; every block adds the G partial sums in the same order (identical
//      totals in every block) and solves (I + L) h = g itself.
//   4. Update of its rows, u_{j+1} = w - V (sigma o h), in the reverse order of step 2 (the
//      columns read last are the likeliest to be in L2; FP64 in fixed point); partial sums of
//      ||u_{j+1}||^2 and of u_{j+1} over the block's pieces of aggregates (U^T u_{j+1}).
//   5. Grid barrier 2; block 0 adds the norm partials and applies the rotations and the
//      stopping tests; the other blocks form c = U^T u_{j+1} from the piece sums and share
//      the rows of y = T^-1 c, giving s' for step j + 1.
//   6. A split barrier: each block arrives once its share of step 5 is published, forms the
//      diagonal part of the next step's SpMV (it needs only u_{j+1}), then waits for all
//      arrivals and reads the same stopping decision and sigma_{j+1}.
// CGS2 forms only g = V^T w in step 2, takes h = g in step 3 and inserts between 3 and 4 the
// first update w -= V h with the second multi-dot h' = V^T w (a pass over each super-tile's
// rows, w' in shared memory in between), one more grid barrier, and coefficients h + h'.
// Every reduction is formed in a fixed order: runs are bitwise reproducible.  The per-phase
// register budgets (loads in flight) are set so that no loop needs local memory: with 220 KB
// of shared memory per block, spilled registers would live in L2 (the FP64 one-reduction step with a
// run-time number of diagonals keeps 4 bytes there, 16 in clusters; the others none).
//
// The batched form (k_arnoldi_batch) runs the same cycle for one system per thread-block
// cluster, whose hardware barrier takes the place of the grid barriers.
//
// The basis is streamed with plain vectorised loads rather than bulk asynchronous copies:
// measured on GB300, a multiprocessor fed by bulk copies reached about 10 bytes per clock,
// against the 22 that the HBM copy bandwidth asks of each of the 152.
#pragma once

#include <algorithm>
#include <type_traits>
#include <utility>

#include "fixed.cuh"
#include "internal.h"
#include "kernels.cuh"

namespace gg {

namespace {

constexpr int kArnWarps = 16;
constexpr int kArnThreads = kArnWarps * 32;
constexpr int kArnUnit = kPartUnit;              // rows per unit of the row partition
constexpr size_t kArnSmem = 220 * 1024;          // dynamic shared memory
// reductions: per set of dots, warp and column an int4 (fixed point) or a pair of floats; the
// updates' coefficients and shared partial sums (arn_sk)
constexpr size_t kArnScratch = 2 * kMaxK * 33 * sizeof(double);
static_assert(kArnScratch >= 2 * kArnWarps * kMaxK * sizeof(int4), "two sets of slots");
constexpr long long kArnSpins = 1LL << 21;       // polls of the barrier word: about a second
constexpr int kArnNormCol = 2 * kMaxK;           // column of ctl.part holding the norm partials
constexpr int kArnMaxCol = kArnNormCol + 1;      // and the blocks' largest |u_{j+1}| (high words)
constexpr int kArnAwRows64 = 6;  // rows per thread of an A W gather batch: FP64 (CSR rows)
constexpr int kArnAwRows32 = 7;  // FP32 (row-indexed planes)
// columns per pass of the fixed-point multi-dot with two dots and with one, passes in flight
// (q1-n1024, create + 300 steps: 58.7 ms; 4 and 6 columns, one pass: 60.6; 2 columns, 3 passes:
// 60.9; reads alone run at 4.7, 5.6 and 5.8 TB/s with 4, 6 and 8 16-byte loads per lane)
constexpr int kArnFxGroup = 3;
constexpr int kArnFxGroup1 = 4;
constexpr int kArnFxDepth = 2;

// orthogonalisation of an instantiation, and its operator (ND): 9 diagonals unrolled, a run-time
// number of diagonals, CSR
enum { kArnLowsync = 0, kArnLowsyncDf = 1, kArnCgs2 = 2 };
constexpr int kArnCsr = -1;

template <typename TV, typename TACC>
struct ArnArgs {
  int N;          // rows of A
  int units;      // ldv / kArnUnit
  int fine;       // ranges of units that the aggregate pieces are cut at (ArnRows)
  int jmax, m;    // steps of this cycle (<= m), restart length
  int pre;        // the predecessor is the coarse solve of step 0: the diagonal part of
                  // its SpMV may run before the wait
  int defl;       // add the coarse correction A W s'
  int r;          // aggregates (entries of s')
  int RS;         // rows per super-tile (a multiple of kArnUnit)
  long long ldv, ldd;
  const TV* V;    // basis, column-major (ldv)
  TACC* w;        // working vector
  DiaOffsets dia;
  const TACC* dval;
  const int* rowptr;  // CSR (no diagonal storage)
  const int* col;
  const TACC* val;
  int vec;            // CSR: long rows, 8 lanes each (arn_csr)
  const int* aurp;
  const int* aucol;
  const TACC* auval;
  const int* aup_col;   // the rows' first two A W entries, two planes of N
  const TACC* aup_val;
  const TACC* sdefl;  // s' in the step's precision (step 0: from the coarse-solve kernel)
  // the coarse solve of the next step, in the kernel: pieces of aggregates (nodes perm
  // [piece_start[p], piece_start[p + 1]), each inside one block's rows), block b's pieces
  // blk_piece[blk_piece_start[b] ...], T^-1 (r x r, row-major)
  const int* perm;
  const int* piece_start;
  const int* agg_piece;
  const int* blk_piece_start;
  const int* blk_piece;
  const double* uscale;
  const double* tinv;
  const float* tinv32;  // FP32 copy of T^-1 (FP32 basis)
  Ctl ctl;
  unsigned* gbar;  // [0] arrivals, [1] generation
};

// Block `bid` of the G that share a system: its rows [R0, R1), whole fine ranges f0 .. f1 - 1 (fine
// range f: the units [f U / F, (f + 1) U / F) of the U); one fine range per block where a grid of
// F blocks runs the system, several where a cluster of fewer blocks does
struct ArnRows {
  int G, bid, f0, f1;
  long long R0, R1;
};
template <typename A>
__device__ __forceinline__ ArnRows arn_rows(const A& a, int G, int bid) {
  ArnRows o;
  o.G = G;
  o.bid = bid;
  o.f0 = (int)((long long)bid * a.fine / G);
  o.f1 = (int)((long long)(bid + 1) * a.fine / G);
  o.R0 = (long long)o.f0 * a.units / a.fine * kArnUnit;
  o.R1 = (long long)o.f1 * a.units / a.fine * kArnUnit;
  return o;
}

// rows VN elements at a time (16-byte loads of the basis type, 8-byte for BF16: a warp's chunk is
// then at most kArnUnit rows)
template <typename TV> struct ArnVec { static constexpr int n = sizeof(TV) == 8 ? 2 : 4; };

// Grid barrier (cooperative launch: every block resident).  Thread 0 arrives on bar[0];
// the last arrival resets it and advances the generation bar[1]; the others poll the
// generation with a bound and report false when it never moves.
// CL: the blocks are one thread-block cluster, whose hardware barrier (all its threads) takes
// the place of the words in global memory.
__device__ __forceinline__ void arn_cluster_arrive() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
}
__device__ __forceinline__ void arn_cluster_wait() {
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

template <bool CL>
__device__ __forceinline__ bool arn_grid_sync(unsigned* bar, unsigned gen) {
  if constexpr (CL) {
    __syncwarp();
    arn_cluster_arrive();
    arn_cluster_wait();
    return true;
  }
  __shared__ int s_ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    int ok = 1;
    __threadfence();
    const unsigned arrived = atomicAdd(&bar[0], 1u);
    if (arrived == gridDim.x - 1) {
      atomicExch(&bar[0], 0u);
      __threadfence();
      atomicExch(&bar[1], gen + 1u);
    } else {
      long long spins = 0;
      while (*(volatile unsigned*)&bar[1] == gen) {
        if (++spins > kArnSpins) {
          ok = 0;
          break;
        }
      }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// Split grid barrier on a counter that only grows (bar[2]): a block arrives once its share
// of a phase is published, carries on with work that does not need the other blocks'
// shares, and waits later until the counter reaches the target (G arrivals per phase,
// counted from the value read at the kernel's start; compared modulo 2^32).
template <bool CL>
__device__ __forceinline__ void arn_arrive(unsigned* cnt) {
  __syncthreads();
  if constexpr (CL) {
    arn_cluster_arrive();
    return;
  }
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(cnt, 1u);
  }
}

template <bool CL>
__device__ __forceinline__ bool arn_wait(const unsigned* cnt, unsigned target) {
  if constexpr (CL) {
    __syncwarp();
    arn_cluster_wait();
    return true;
  }
  __shared__ int s_ok;
  if (threadIdx.x == 0) {
    int ok = 1;
    long long spins = 0;
    while ((int)(*(volatile const unsigned*)cnt - target) < 0) {
      if (++spins > kArnSpins) {
        ok = 0;
        break;
      }
    }
    __threadfence();
    s_ok = ok;
  }
  __syncthreads();
  return s_ok != 0;
}

// dst[c] = sum_{r < nrows} src[r * ldp + c] for c < ncols, in a fixed order: the Q threads
// of a column (consecutive lanes) take rows q, q + Q, ..., each issuing up to 8 loads at
// once before adding them, then combine by shuffles; ends with a block barrier.  (FP64 adds
// issue at a quarter-warp per clock on GB300: the trees are kept short.)
__device__ __forceinline__ void arn_reduce_cols(const double* src, int nrows, int ncols, int ldp,
                                                double* dst) {
  constexpr int L = 8;
  int Q = 1;
  while (Q * 2 <= 32 && Q * 2 * ncols <= (int)blockDim.x) Q *= 2;
  const int rounds = (ncols * Q + blockDim.x - 1) / blockDim.x;
  for (int rd = 0; rd < rounds; ++rd) {
    const int idx = rd * blockDim.x + threadIdx.x;
    const int c = idx / Q, q = idx % Q;
    double sum = 0.0;
    if (c < ncols) {
      for (int r0 = q; r0 < nrows; r0 += L * Q) {
        double v[L];
#pragma unroll
        for (int u = 0; u < L; ++u) {
          const int r = r0 + u * Q;
          v[u] = r < nrows ? __ldcg(src + (size_t)r * ldp + c) : 0.0;
        }
#pragma unroll
        for (int h = L / 2; h > 0; h >>= 1)
#pragma unroll
          for (int u = 0; u < h; ++u) v[u] += v[u + h];
        sum += v[0];
      }
    }
    for (int o = 1; o < Q; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (c < ncols && q == 0) dst[c] = sum;
  }
  __syncthreads();
}

// 16-byte vector load of VN basis elements from global memory, streamed past L1 (the basis is read
// once per pass; L1 is mostly carved out for shared memory here).  Not the read-only path: the
// launch that reads a column has stored it.
template <typename TV, typename TACC, int VN>
__device__ __forceinline__ void arn_ldg(const TV* p, TACC (&o)[VN]) {
  if constexpr (std::is_same<TV, double>::value) {
    double x, y;
    asm volatile("ld.global.L1::no_allocate.v2.f64 {%0, %1}, [%2];"
                 : "=d"(x), "=d"(y)
                 : "l"(p));
    o[0] = (TACC)x;
    o[1] = (TACC)y;
  } else if constexpr (std::is_same<TV, float>::value) {
    float x, y, z, w;
    asm volatile("ld.global.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(x), "=f"(y), "=f"(z), "=f"(w)
                 : "l"(p));
    o[0] = x; o[1] = y; o[2] = z; o[3] = w;
  } else {
    unsigned x, y;
    asm volatile("ld.global.L1::no_allocate.v2.b32 {%0, %1}, [%2];"
                 : "=r"(x), "=r"(y)
                 : "l"(p));
    // a BF16 value is the upper half of its FP32 form
    o[0] = __uint_as_float(x << 16);
    o[1] = __uint_as_float(x & 0xffff0000u);
    o[2] = __uint_as_float(y << 16);
    o[3] = __uint_as_float(y & 0xffff0000u);
  }
}

// An entry of u_j, which other blocks stored earlier in the launch (nor is this the read-only path),
// kept in L1 for the neighbouring rows of the SpMV
template <typename TACC>
__device__ __forceinline__ TACC arn_ldx(const double* p) {
  double v;
  asm volatile("ld.global.ca.f64 %0, [%1];" : "=d"(v) : "l"(p));
  return (TACC)v;
}
template <typename TACC>
__device__ __forceinline__ TACC arn_ldx(const float* p) {
  float v;
  asm volatile("ld.global.ca.f32 %0, [%1];" : "=f"(v) : "l"(p));
  return (TACC)v;
}
template <typename TACC>
__device__ __forceinline__ TACC arn_ldx(const __nv_bfloat16* p) {
  unsigned v;
  asm volatile("ld.global.ca.u16 %0, [%1];" : "=r"(v) : "l"(p));
  return (TACC)__uint_as_float(v << 16);
}

// An FP64 operator value read with the L2 evict-first priority: the diagonals (76 MB at
// 1M rows) then give way to the basis columns, which the update re-reads right after the
// multi-dot (measured on q1-n1024: FP64 step 236.4 to 228.0 us at the fixed 100-step
// protocol; the FP32 step, whose 38 MB of diagonals stay useful in L2 across steps, went
// from 76.9 to 80.0 us with the same hint and keeps plain loads)
__device__ __forceinline__ double arn_ld_evict_first(const double* p) {
  unsigned long long pol;
  asm("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  double v;
  asm volatile("ld.global.nc.L2::cache_hint.f64 %0, [%1], %2;" : "=d"(v) : "l"(p), "l"(pol));
  return v;
}

template <typename TV, typename TACC, int VN>
__device__ __forceinline__ void arn_stv(TV* p, const TACC (&v)[VN]) {
  if constexpr (std::is_same<TV, double>::value) {
    *reinterpret_cast<double2*>(p) = make_double2(v[0], v[1]);
  } else if constexpr (std::is_same<TV, float>::value) {
    *reinterpret_cast<float4*>(p) = make_float4(v[0], v[1], v[2], v[3]);
  } else {
    uint2 o;
    __nv_bfloat162* h = reinterpret_cast<__nv_bfloat162*>(&o);
#pragma unroll
    for (int e = 0; e < 2; ++e) h[e] = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
    *reinterpret_cast<uint2*>(p) = o;
  }
}

// a grid barrier that never completed: the solve stops with GMRES_ERR_TIMEOUT
__device__ __forceinline__ void arn_timeout(Ctl& ctl) {
  if (threadIdx.x == 0) {
    ctl.flags[F_STATUS] = GMRES_ERR_TIMEOUT;
    ctl.flags[F_STOP] = 1;
    ctl.flags[F_CYCLE_DONE] = 1;
  }
}

// a basis entry written earlier in this launch, read through L2 as FP64
__device__ __forceinline__ double arn_ldcg_d(const double* p) { return __ldcg(p); }
__device__ __forceinline__ double arn_ldcg_d(const float* p) { return (double)__ldcg(p); }
__device__ __forceinline__ double arn_ldcg_d(const __nv_bfloat16* p) {
  return (double)__bfloat162float(__ldcg(p));
}

// ---- double-FP32 arithmetic for the FP64 multi-dot (GMRES_DOT_DF32) ---------------------
// In the double-FP32 form of the multi-dot each FP64 operand is split into two floats, x ~ hi + lo, with integer operations only (hi = x with
// its significand cut to 24 bits, lo = the remaining 29 bits rounded to 24: 47 significant
// bits in all); a product takes the exact product of the high parts by an FMA (Dekker's
// two-product), the two cross terms in FP32 (lo * lo, below 2^-46 of the product, is
// dropped), and the running sum is a pair (s, c) advanced by Knuth's TwoSum, every rounding
// error gathered in c.  Magnitudes between 2^-126 and 2^127 split exactly as stated; smaller
// ones become 0 (an absolute error below 2^-126), larger ones infinity.
__device__ __forceinline__ void arn_df_split(double v, float& hi, float& lo) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned h32 = (unsigned)(b >> 32), l32 = (unsigned)b;
  const unsigned sgn = h32 & 0x80000000u;
  const unsigned ah = h32 & 0x7fffffffu;
  const int E = (int)(ah >> 20);  // biased FP64 exponent
  // exponent and top 23 significand bits, rebiased from 1023 to 127 (mod 2^32)
  unsigned hb = ((ah << 3) | (l32 >> 29)) - (896u << 23);
  const unsigned m29 = l32 & 0x1fffffffu;  // the significand bits below hi's
  const unsigned fb = __float_as_uint(__uint2float_rn(m29));
  const unsigned lb = fb + ((unsigned)(E - 1075) << 23);  // m29 * 2^(E - 1075)
  const bool okh = E >= 897;
  const bool okl = okh && m29 != 0u && (int)(fb >> 23) + E - 1075 >= 1;
  hb = E > 1150 ? 0x7f800000u : hb;
  hi = __uint_as_float(okh ? (hb | sgn) : sgn);
  lo = __uint_as_float(okl ? (lb | sgn) : 0u);
}

// (s, c) += (ah + al) (bh + bl); the _rn intrinsics keep the compiler from contracting the
// error-free steps into FMAs
__device__ __forceinline__ void arn_df_fma(float& s, float& c, float ah, float al, float bh,
                                           float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = __fmaf_rn(ah, bh, -p);  // exact: p + e = ah bh
  e = __fmaf_rn(ah, bl, e);
  e = __fmaf_rn(al, bh, e);
  const float t = __fadd_rn(s, p);  // TwoSum: t + err = s + p exactly
  const float bp = __fsub_rn(t, s);
  const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(p, bp));
  s = t;
  c = __fadd_rn(c, __fadd_rn(err, e));
}

// (s, c) += (s2, c2)
__device__ __forceinline__ void arn_df_add(float& s, float& c, float s2, float c2) {
  const float t = __fadd_rn(s, s2);
  const float bp = __fsub_rn(t, s);
  const float err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, bp)), __fsub_rn(s2, bp));
  s = t;
  c = __fadd_rn(__fadd_rn(c, c2), err);
}

// The same over partials stored as double-FP32 pairs (two floats per slot): TwoSum on the
// FP32 pipe in a fixed order, L loads in flight per thread, rounded to FP64 once per column.
template <int L>
__device__ __forceinline__ void arn_reduce_cols_df(const double* src, int nrows, int ncols,
                                                   int ldp, double* dst) {
  int Q = 1;
  while (Q * 2 <= 32 && Q * 2 * ncols <= (int)blockDim.x) Q *= 2;
  const int rounds = (ncols * Q + blockDim.x - 1) / blockDim.x;
  for (int rd = 0; rd < rounds; ++rd) {
    const int idx = rd * blockDim.x + threadIdx.x;
    const int c = idx / Q, q = idx % Q;
    float hs = 0.f, hc = 0.f;
    if (c < ncols) {
      for (int r0 = q; r0 < nrows; r0 += L * Q) {
        float2 v[L];
#pragma unroll
        for (int u = 0; u < L; ++u) {
          const int r = r0 + u * Q;
          v[u] = r < nrows ? __ldcg(reinterpret_cast<const float2*>(src + (size_t)r * ldp + c))
                           : make_float2(0.f, 0.f);
        }
#pragma unroll
        for (int u = 0; u < L; ++u) arn_df_add(hs, hc, v[u].x, v[u].y);
      }
    }
    for (int o = 1; o < Q; o <<= 1) {
      const float a2 = __shfl_xor_sync(0xffffffffu, hs, o);
      const float b2 = __shfl_xor_sync(0xffffffffu, hc, o);
      arn_df_add(hs, hc, a2, b2);
    }
    if (c < ncols && q == 0) dst[c] = (double)hs + (double)hc;
  }
  __syncthreads();
}

// How the 16 warps share nch 64-row chunks: from 16 chunks on a warp takes the chunks warp, warp +
// 16, ... with all columns; with fewer, S = 16 / nch warps share a chunk's columns (integer sums:
// the result does not depend on the split).
struct ArnSplit {
  int S, q0, p, rows;  // warps per chunk, the warp's first chunk, its share, chunks taken at once
  bool live;
};
__device__ __forceinline__ ArnSplit arn_split(int nch) {
  const int warp = threadIdx.x >> 5;
  if (nch >= kArnWarps || nch == 0) return ArnSplit{1, warp, 0, kArnWarps, nch > 0};
  const int S = kArnWarps / nch;
  return ArnSplit{S, warp % nch, warp / nch, nch, warp / nch < S};
}

// The shifts of the rows (fixed.cuh), 16 bits each, in the last of the m + 1 columns: the cycle needs
// u_m's norm only, so that column is never stored
template <typename TV, typename TACC>
__device__ __forceinline__ short* arn_shifts(const ArnArgs<TV, TACC>& a) {
  return reinterpret_cast<short*>(const_cast<TV*>(a.V) + (size_t)a.m * a.ldv);
}

// Two rows of a basis column held as fixed-point integers, past L1 (a column is converted in
// place within the launch, after its FP64 form was read through L1)
__device__ __forceinline__ void arn_ldfx(const long long* p, uint4& o) {
  asm volatile("ld.global.cg.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(o.x), "=r"(o.y), "=r"(o.z), "=r"(o.w)
               : "l"(p));
}

// Multi-dot of an FP64 basis in fixed point (fixed.cuh): NSET dots per column, with w (Wf)
// and u_j (Uf), both already operands (limbs of two rows per int4).  The first kf columns are
// fixed-point integers, a last column kf (k = kf + 1), not converted yet, FP64 (largest exponent
// ej; its dot with w only).  Row order: per pass a warp takes a group of G columns at the same
// 64 rows (one 16-byte load per column and lane), D such units in flight; each value's register
// is reloaded for a later unit as soon as it is used.  At the end of a group the lanes' integer totals meet by warp
// reductions and lane 0 stores them in slot[set][first chunk][c] (once per super-tile).
// Bound by the loads; per element 6 IMAD.WIDE and a few simple integer operations, where 2 FP64
// multiply-adds hold their pipe for 64 issue slots each (q1-n1024, GMRES(50), a step of the whole
// kernel: 228 us with FP64 multiply-adds in dots and update, 152 us in fixed point; 4M rows without
// deflation, 45 columns: 743 us as FP64 phases, 453 us).
template <int NSET, int G, int D>
__device__ __forceinline__ void arn_dots_fx(int4* slot, const double* V, long long ldv, int kf,
                                            int k, int ej, long long s0, int nch, const int4* Wf,
                                            const int4* Uf, const short* Sg, int lane) {
  const ArnSplit sp = arn_split(nch);
  if (!sp.live) return;
  const int nqw = (nch - 1 - sp.q0) / kArnWarps + 1;  // chunks of this warp
  const long long at = s0 + (long long)sp.q0 * 64 + lane * 2;
  const long long* const base = reinterpret_cast<const long long*>(V) + at;
  // a unit: a group's columns at one chunk.  D units are in flight (b), reloaded as they are used
  int ln = 0, gn = sp.p * G;  // chunk and first column of the next unit to load
  const long long* pn = base + (size_t)gn * ldv;
  auto advance = [&] {
    pn += kArnWarps * 64;
    if (++ln == nqw) {  // on to the next group's first chunk
      ln = 0;
      gn += G * sp.S;
      pn = base + (size_t)gn * ldv;
    }
  };
  uint4 b[D][G];
#pragma unroll
  for (int d = 0; d < D; ++d) {
#pragma unroll
    for (int u = 0; u < G; ++u) {
      b[d][u] = make_uint4(0, 0, 0, 0);
      if (gn + u < kf) arn_ldfx(pn + (size_t)u * ldv, b[d][u]);
    }
    advance();
  }
  auto store = [&](int set, int c, const FxDot& a) {
    const FxSum t = fx_warp_sum(a);
    if (lane == 0)
      slot[(size_t)(set * kArnWarps + sp.q0) * kMaxK + c] =
          make_int4((int)t.s, (int)(t.s >> 32), (int)t.f, (int)(t.f >> 32));
  };
  FxDot acc[NSET][G];
#pragma unroll
  for (int u = 0; u < G; ++u)
#pragma unroll
    for (int s = 0; s < NSET; ++s) acc[s][u] = FxDot{0, 0, 0, 0};
  int g0 = sp.p * G, qi = 0;  // first column and chunk of the unit in use
  const int at0 = sp.q0 * 32 + lane;
#pragma unroll 1
  while (g0 < kf) {
#pragma unroll
    for (int d = 0; d < D; ++d) {
      if (D > 1 && g0 >= kf) break;
      const int4 w = Wf[at0 + qi * (kArnWarps * 32)];
      int4 uu = make_int4(0, 0, 0, 0);
      if (NSET == 2) uu = Uf[at0 + qi * (kArnWarps * 32)];
#pragma unroll
      for (int u = 0; u < G; ++u) {  // (an absent column's stale values meet its sums only)
        const Fx v0 = fx_limbs(b[d][u].x, b[d][u].y), v1 = fx_limbs(b[d][u].z, b[d][u].w);
        if (gn + u < kf) arn_ldfx(pn + (size_t)u * ldv, b[d][u]);
        fx_dot(acc[0][u], v0, make_int2(w.x, w.y));
        fx_dot(acc[0][u], v1, make_int2(w.z, w.w));
        if (NSET == 2) {
          fx_dot(acc[NSET - 1][u], v0, make_int2(uu.x, uu.y));
          fx_dot(acc[NSET - 1][u], v1, make_int2(uu.z, uu.w));
        }
      }
      advance();
      if (++qi == nqw) {  // the group's last chunk in this warp
#pragma unroll
        for (int u = 0; u < G; ++u)
#pragma unroll
          for (int s = 0; s < NSET; ++s) {
            if (g0 + u < kf) store(s, g0 + u, acc[s][u]);
            acc[s][u] = FxDot{0, 0, 0, 0};
          }
        qi = 0;
        g0 += G * sp.S;
      }
    }
  }
  if (kf < k && sp.p == sp.S - 1) {  // the FP64 column
    FxDot a{0, 0, 0, 0};
    for (int qi = 0; qi < nqw; ++qi) {
      const long long r = at + (long long)qi * (kArnWarps * 64);
      const double2 v = __ldcg(reinterpret_cast<const double2*>(V + (size_t)kf * ldv + r));
      const short2 sh = __ldcg(reinterpret_cast<const short2*>(Sg + r));
      const int4 w = Wf[(size_t)(sp.q0 + qi * kArnWarps) * 32 + lane];
      fx_dot(a, fx_limbs(fx_basis(v.x, ej - sh.x)), make_int2(w.x, w.y));
      fx_dot(a, fx_limbs(fx_basis(v.y, ej - sh.y)), make_int2(w.z, w.w));
    }
    store(0, kf, a);
    if (NSET == 2) store(1, kf, FxDot{0, 0, 0, 0});
  }
}

// Multi-dot of an FP64 basis in double-FP32 (row order): warp w takes the chunks w, w + 16,
// ... of 64 rows of the super-tile and, per pass, G columns at the same rows (one 16-byte
// load per column and lane, all issued before the products); w and u_j come split from
// shared memory (float2 hi, lo per row).  At the end of a pass the lanes' pairs of each
// column meet by a shuffle tree of TwoSums and lane 0 adds them into dfp[warp][c][set]:
// no FP64 instruction in the loop.
constexpr int kArnDfGroup = 6;

__device__ __forceinline__ void arn_dots_df(float* dfp, const double* V, long long ldv, int k,
                                            long long s0, int nch, const float2* Ws,
                                            const float2* Us, int warp, int lane) {
  constexpr int G = kArnDfGroup;
  for (int g0 = 0; g0 < k; g0 += G) {
    const int gc = k - g0 < G ? k - g0 : G;
    float s1[G], c1[G], s2[G], c2[G];
#pragma unroll
    for (int q = 0; q < G; ++q) s1[q] = c1[q] = s2[q] = c2[q] = 0.f;
    const double* col = V + (size_t)g0 * ldv + s0 + (size_t)lane * 2;
    for (int ch = warp; ch < nch; ch += kArnWarps) {
      const int r = ch * 64 + lane * 2;
      double v[G][2];
#pragma unroll
      for (int q = 0; q < G; ++q)
        if (q < gc) arn_ldg<double, double, 2>(col + (size_t)q * ldv + (size_t)ch * 64, v[q]);
      const float4 wv = *reinterpret_cast<const float4*>(Ws + r);
      const float4 uv = *reinterpret_cast<const float4*>(Us + r);
#pragma unroll
      for (int q = 0; q < G; ++q)
        if (q < gc) {
          float h0, l0, h1, l1;
          arn_df_split(v[q][0], h0, l0);
          arn_df_split(v[q][1], h1, l1);
          arn_df_fma(s1[q], c1[q], h0, l0, wv.x, wv.y);
          arn_df_fma(s1[q], c1[q], h1, l1, wv.z, wv.w);
          arn_df_fma(s2[q], c2[q], h0, l0, uv.x, uv.y);
          arn_df_fma(s2[q], c2[q], h1, l1, uv.z, uv.w);
        }
    }
#pragma unroll
    for (int q = 0; q < G; ++q)
      if (q < gc) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const float a = __shfl_xor_sync(0xffffffffu, s1[q], o);
          const float b = __shfl_xor_sync(0xffffffffu, c1[q], o);
          const float d = __shfl_xor_sync(0xffffffffu, s2[q], o);
          const float e = __shfl_xor_sync(0xffffffffu, c2[q], o);
          arn_df_add(s1[q], c1[q], a, b);
          arn_df_add(s2[q], c2[q], d, e);
        }
        if (lane == 0) {
          float* p = dfp + ((size_t)warp * kMaxK + g0 + q) * 4;
          float a = p[0], b = p[1];
          arn_df_add(a, b, s1[q], c1[q]);
          p[0] = a;
          p[1] = b;
          a = p[2];
          b = p[3];
          arn_df_add(a, b, s2[q], c2[q]);
          p[2] = a;
          p[3] = b;
        }
      }
  }
}

// Diagonal part of the SpMV for B rows (row0 + b * stride) at once: all loads of the B
// rows are issued before their products (ND > 0: ND diagonals, unrolled; ND = 0: nd at
// run time, four at a time).  x indexes are clamped to a valid row, where the stored
// value is 0.
template <int B, int ND, typename TV, typename TACC>
__device__ __forceinline__ void arn_dia_rows(TACC (&acc)[B], long long row0, long long stride,
                                             long long Nn, int nd, const int* off,
                                             long long ldd, const TACC* __restrict__ dval,
                                             const TV* __restrict__ x) {
  constexpr int NQ = ND > 0 ? ND : 4;
#pragma unroll
  for (int b = 0; b < B; ++b) acc[b] = 0;
  for (int q0 = 0; q0 < (ND > 0 ? ND : nd); q0 += NQ) {
    TACC av[B][NQ], xv[B][NQ];
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const long long row = row0 + b * stride;
      const long long rr = row < Nn ? row : Nn - 1;
#pragma unroll
      for (int u = 0; u < NQ; ++u) {
        const int q = q0 + u;
        const bool live = ND > 0 || q < nd;
        const long long c = min(max(rr + off[live ? q : 0], 0LL), Nn - 1);
        if constexpr (sizeof(TACC) == 8)
          av[b][u] = live ? arn_ld_evict_first(dval + (size_t)q * ldd + rr) : (TACC)0;
        else
          av[b][u] = live ? __ldg(dval + (size_t)q * ldd + rr) : (TACC)0;
        xv[b][u] = live ? arn_ldx<TACC>(x + c) : (TACC)0;
      }
    }
#pragma unroll
    for (int b = 0; b < B; ++b)
#pragma unroll
      for (int u = 0; u < NQ; ++u) acc[b] += av[b][u] * xv[b][u];
  }
}

// warps that share a chunk in every block of the system: 16 / the most chunks of a block
template <typename TV, typename TACC>
__device__ __forceinline__ int arn_share(const ArnArgs<TV, TACC>& a, int G) {
  constexpr int per = kArnUnit / (32 * ArnVec<TV>::n);  // chunks per unit
  const int most = ((a.fine + G - 1) / G) * ((a.units + a.fine - 1) / a.fine) * per;
  return most < kArnWarps ? kArnWarps / most : 1;
}

// Multi-dot in row-chunk order (FP32 or BF16 basis): per unit, a warp takes a group of up to G
// columns at one chunk: one 16-byte (BF16: 8-byte) load per column and lane for the same rows, so
// the loads in flight of a warp fall in one row window of many columns (on GB300 this streams
// about twice as fast as a warp reading one column through many consecutive chunks).  Units run
// group by group, the warp's chunks in order, two units in flight, each value's register reloaded
// as it is used.  S warps share a chunk's groups where the blocks have few chunks (arn_split32).
// At a group's last chunk the lanes' partial sums meet as double-FP32 pairs (arn_warp_pairs) and are
// accumulated into wsum[set][first chunk][c].
template <int ND> constexpr int arn_group() { return ND == 9 ? 6 : 5; }

// Sums over the warp's lanes of up to 8 values, as double-FP32 pairs (FP32 adds would round in the
// last bits of the largest partial sum, FP64 adds hold their pipe 64 issue slots each).  Lanes halve
// the columns they keep in the first three exchanges: 9 pair additions for 8 columns, where a tree
// per column takes 5 each.  The total of column arn_pairs_col(lane), in every lane.
__device__ __forceinline__ int arn_pairs_col(int lane) {
  return (lane >> 2 & 4) | (lane >> 2 & 2) | (lane >> 2 & 1);
}
template <int G>
__device__ __forceinline__ float2 arn_warp_pairs(const float (&v)[G], int lane) {
  static_assert(G <= 8, "eight columns at a time");
  float s[4], c[4];
  const bool h4 = lane & 16, h2 = lane & 8, h1 = lane & 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float lo = i < G ? v[i < G ? i : 0] : 0.f, hi = i + 4 < G ? v[i + 4 < G ? i + 4 : 0] : 0.f;
    s[i] = h4 ? hi : lo;
    c[i] = 0.f;
    arn_df_add(s[i], c[i], __shfl_xor_sync(0xffffffffu, h4 ? lo : hi, 16), 0.f);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float so = __shfl_xor_sync(0xffffffffu, h2 ? s[i] : s[i + 2], 8);
    const float co = __shfl_xor_sync(0xffffffffu, h2 ? c[i] : c[i + 2], 8);
    s[i] = h2 ? s[i + 2] : s[i];
    c[i] = h2 ? c[i + 2] : c[i];
    arn_df_add(s[i], c[i], so, co);
  }
  const float so = __shfl_xor_sync(0xffffffffu, h1 ? s[0] : s[1], 4);
  const float co = __shfl_xor_sync(0xffffffffu, h1 ? c[0] : c[1], 4);
  float rs = h1 ? s[1] : s[0], rc = h1 ? c[1] : c[0];
  arn_df_add(rs, rc, so, co);
#pragma unroll
  for (int o = 2; o > 0; o >>= 1) {
    const float s2 = __shfl_xor_sync(0xffffffffu, rs, o);
    const float c2 = __shfl_xor_sync(0xffffffffu, rc, o);
    arn_df_add(rs, rc, s2, c2);
  }
  return make_float2(rs, rc);
}

// S: warps per chunk, the same in every block of the system (so that equal rows are summed in the
// same order everywhere): 16 / the most chunks a block holds, at least 1
__device__ __forceinline__ ArnSplit arn_split32(int S, int nch) {
  const int warp = threadIdx.x >> 5;
  if (S <= 1) return ArnSplit{1, warp, 0, kArnWarps, warp < nch};
  const int w = kArnWarps / S;  // chunk places
  return ArnSplit{S, warp % w, warp / w, w, warp / w < S && warp % w < nch};
}

template <typename TV, typename TACC, int NSET, int G>
__device__ __forceinline__ void arn_dots_rows(double* wsum, const TV* V, long long ldv, int k,
                                              long long s0, int nch, int S, const TACC* Ws,
                                              const TACC* Us, int lane) {
  constexpr int VN = ArnVec<TV>::n, D = 2;
  const ArnSplit sp = arn_split32(S, nch);
  if (!sp.live) return;
  const int nqw = S > 1 ? 1 : (nch - 1 - sp.q0) / kArnWarps + 1;  // chunks of this warp
  const long long step = (long long)kArnWarps * 32 * VN;
  const TV* const base = V + s0 + (size_t)sp.q0 * 32 * VN + (size_t)lane * VN;
  int ln = 0, gn = sp.p * G;
  const TV* pn = base + (size_t)gn * ldv;
  auto advance = [&] {
    pn += step;
    if (++ln == nqw) {
      ln = 0;
      gn += G * sp.S;
      pn = base + (size_t)gn * ldv;
    }
  };
  TACC b[D][G][VN];
#pragma unroll
  for (int d = 0; d < D; ++d) {
#pragma unroll
    for (int u = 0; u < G; ++u) {
#pragma unroll
      for (int e = 0; e < VN; ++e) b[d][u][e] = 0;
      if (gn + u < k) arn_ldg<TV, TACC, VN>(pn + (size_t)u * ldv, b[d][u]);
    }
    advance();
  }
  TACC acc[NSET][G];
#pragma unroll
  for (int u = 0; u < G; ++u)
#pragma unroll
    for (int t = 0; t < NSET; ++t) acc[t][u] = 0;
  int g0 = sp.p * G, qi = 0;
  const int at = (sp.q0 * 32 + lane) * VN;
#pragma unroll 1
  while (g0 < k) {
#pragma unroll
    for (int d = 0; d < D; ++d) {
      if (g0 >= k) break;
      TACC wv[VN], uv[VN];
      ld_acc<VN>(Ws + at + qi * step, wv);
      if (NSET == 2) ld_acc<VN>(Us + at + qi * step, uv);
#pragma unroll
      for (int u = 0; u < G; ++u) {
        if (g0 + u < k)
#pragma unroll
          for (int e = 0; e < VN; ++e) {
            acc[0][u] += b[d][u][e] * wv[e];
            if (NSET == 2) acc[NSET - 1][u] += b[d][u][e] * uv[e];
          }
        if (gn + u < k) arn_ldg<TV, TACC, VN>(pn + (size_t)u * ldv, b[d][u]);
      }
      advance();
      if (++qi == nqw) {  // the group's last chunk in this warp
#pragma unroll
        for (int t = 0; t < NSET; ++t) {
          const float2 v = arn_warp_pairs<G>(acc[t], lane);
          const int u = arn_pairs_col(lane);
          if ((lane & 3) == 0 && u < G && g0 + u < k) {
            float2* pw = reinterpret_cast<float2*>(wsum) +
                         (size_t)(t * kArnWarps + sp.q0) * kMaxK + g0 + u;
            float2 o = *pw;
            arn_df_add(o.x, o.y, v.x, v.y);
            *pw = o;
          }
#pragma unroll
          for (int q = 0; q < G; ++q) acc[t][q] = 0;
        }
        qi = 0;
        g0 += G * sp.S;
      }
    }
  }
}

// The same rows of a CSR operator: a thread per row (ten entries' loads, then their gathers, in
// flight at once), or 8 lanes per row for long rows (two rows of up to 64 entries in flight per
// lane group; 4 lanes: 24.8 against 22.2 ms on the 274,625-unknown Bratu matrix, 100 steps).  With
// one block of 16 warps per multiprocessor the loads in flight per thread stand in for the
// occupancy of a kernel of its own.  Sharing the long rows out by entries instead of the basis'
// row ranges, through w in global memory, did not pay (19.9 against 19.7 ms).
template <typename TV, typename TACC>
__device__ __forceinline__ void arn_csr(const ArnArgs<TV, TACC>& a, const TV* xj, long long s0,
                                        long long s1, TACC* Ws, TACC* Us, int tid, int nthr) {
  const long long N = a.N;
  if (!a.vec) {
    constexpr int U = 10;
    for (long long row = s0 + tid; row < s1; row += nthr) {
      TACC acc = 0, x = 0;
      if (row < N) {
        const int rs = __ldg(a.rowptr + row), re = __ldg(a.rowptr + row + 1);
        x = arn_ldx<TACC>(xj + row);
        for (int q = rs; q < re; q += U) {
          int c[U];
          TACC v[U], xv[U];
#pragma unroll
          for (int u = 0; u < U; ++u) {
            c[u] = q + u < re ? __ldg(a.col + q + u) : 0;
            v[u] = q + u < re ? __ldg(a.val + q + u) : (TACC)0;
          }
#pragma unroll
          for (int u = 0; u < U; ++u)  // (16-bit gathers under a predicate wait for one another: a row
                                       // of 100,000 BF16 entries 8.3 ms, 6.2 without; column 0 then)
            xv[u] = sizeof(TV) == 2 || q + u < re ? arn_ldx<TACC>(xj + c[u]) : (TACC)0;
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (q + u < re) acc += v[u] * xv[u];
        }
      }
      Ws[row - s0] = acc;
      Us[row - s0] = x;
    }
    return;
  }
  constexpr int L = 8, U = 8;  // lanes per row, entries per lane and trip
  const int sub = tid & (L - 1);
  // (a warp's lane groups take 8 consecutive rows: the loop is uniform in a warp)
  for (long long r0 = s0 + 2 * (tid / L); r0 < s1; r0 += 2 * (nthr / L)) {
    TACC acc[2] = {0, 0};
    int q[2], re[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      q[h] = r0 + h < N ? __ldg(a.rowptr + r0 + h) + sub : 0;
      re[h] = r0 + h < N ? __ldg(a.rowptr + r0 + h + 1) : 0;
    }
    while (q[0] < re[0] || q[1] < re[1]) {
      int c[2][U];
      TACC v[2][U];
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int e = q[h] + L * u;
          c[h][u] = e < re[h] ? __ldg(a.col + e) : -1;
          v[h][u] = e < re[h] ? __ldg(a.val + e) : (TACC)0;
        }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        TACC xv[U];
#pragma unroll
        for (int u = 0; u < U; ++u) xv[u] = c[h][u] >= 0 ? arn_ldx<TACC>(xj + c[h][u]) : (TACC)0;
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (c[h][u] >= 0) acc[h] += v[h][u] * xv[u];
        q[h] += L * U;
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int o = L / 2; o > 0; o >>= 1) acc[h] += __shfl_xor_sync(0xffffffffu, acc[h], o);
    if (sub < 2) {
      Ws[r0 + sub - s0] = sub ? acc[1] : acc[0];
      Us[r0 + sub - s0] = r0 + sub < N ? arn_ldx<TACC>(xj + r0 + sub) : (TACC)0;
    }
  }
}

// Diagonal part of step j's SpMV for the rows [s0, s1) of a super-tile: (A v_j) into Ws and
// u_j into Us (shared memory, from row s0; zeros past N)
template <int ND, typename TV, typename TACC>
__device__ __forceinline__ void arn_diag(const ArnArgs<TV, TACC>& a, int j, long long s0,
                                         long long s1, TACC* Ws, TACC* Us, int tid, int nthr) {
  // SpMV rows per thread and batch (4 in FP32 and BF16 spill 12 to 72 bytes: 361k rows BF16 76.0 ms
  // against 71.4, 1M rows FP32 93.9 against 93.3)
  constexpr int B = sizeof(TACC) == 8 ? 2 : 3;
  const long long N = a.N;
  const TV* xj = a.V + (size_t)j * a.ldv;
  if constexpr (ND == kArnCsr) {
    arn_csr<TV, TACC>(a, xj, s0, s1, Ws, Us, tid, nthr);
    return;
  }
  const int nd = ND > 0 ? ND : a.dia.nd;
  for (long long i0 = s0 + tid; i0 < s1; i0 += (long long)B * nthr) {
    TACC v[B];
    arn_dia_rows<B, (ND > 0 ? ND : 0), TV, TACC>(v, i0, nthr, N, nd, a.dia.off, a.ldd, a.dval, xj);
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const long long row = i0 + (long long)b * nthr;
      if (row < s1) {
        Ws[row - s0] = row < N ? v[b] : (TACC)0;
        Us[row - s0] = row < N ? arn_ldx<TACC>(xj + row) : (TACC)0;
      }
    }
  }
}

// The block's column sums of a fixed-point multi-dot over nch chunks: the warps' integer totals, then FP64 once
// per super-tile (added to the earlier super-tiles' unless first)
template <int NSET>
__device__ __forceinline__ void arn_slot_sums(const int4* slot, int nch, int k, const int* sE,
                                              int ew, int eu, bool first, double* sred) {
  const int rows = nch < kArnWarps ? nch : kArnWarps;
  for (int q = threadIdx.x; q < NSET * k; q += kArnThreads) {
    const int set = q / k, c = q % k;
    long long sum = 0, f = 0;
#pragma unroll 4
    for (int w = 0; w < rows; ++w) {
      const int4 v = slot[(size_t)(set * kArnWarps + w) * kMaxK + c];
      sum += ((long long)v.y << 32) | (unsigned)v.x;
      f += ((long long)v.w << 32) | (unsigned)v.z;
    }
    const double d = fx_value(sum, f, sE[c], set ? eu : ew);
    sred[q] = first ? d : sred[q] + d;
  }
}

// The shift of a row with entry u of column j (largest exponent E), kept at p: chosen at the first
// column, reduced where u does not fit
__device__ __forceinline__ int arn_shift_of(short* p, int j, double u, int E, bool row) {
  const int ex = fx_mag(u) >> 20;  // (subnormal entries count as zeros)
  int s = j > 0 ? __ldcg(p) : (row ? kFxUnset : 0);
  if (ex > 0 && (s == kFxUnset || ex > E - s)) s = fx_shift(ex, E);
  else if (j > 0) return s;
  __stcg(p, (short)s);
  return s;
}

// Rows that column j outgrew (bit b of grow: row q0 + b kArnThreads; any: of the warp's lanes): their
// new shifts, their earlier entries in the new unit, their operands
// again.  Rare; the warp shares a row's columns, one round of loads per 32 of them.
template <int NSET>
__device__ __forceinline__ void arn_grow(double* V, long long ldv, const double* w, short* Sg, int j,
                                         int q0, unsigned any, unsigned grow, int ew, int eu, int2* Wf,
                                         int2* Uf) {
  const int lane = threadIdx.x & 31;
#pragma unroll 1
  for (; any; any &= any - 1) {
    const int b = __ffs(any) - 1, q = q0 + b * kArnThreads;
    const bool mine = grow >> b & 1u;
    int so = 0, sn = 0;
    if (mine) {
      const double u = __ldcg(V + (size_t)j * ldv + q);
      so = __ldcg(Sg + q);
      sn = arn_shift_of(Sg + q, j, u, eu, true);
      Wf[q] = fx_operand(__ldcg(w + q), ew + sn);
      if (NSET == 2) Uf[q] = fx_operand(u, eu + sn);
    }
    unsigned lanes = __ballot_sync(0xffffffffu, mine && so != kFxUnset);
#pragma unroll 1
    for (; lanes; lanes &= lanes - 1) {
      const int l = __ffs(lanes) - 1;
      const int d = __shfl_sync(0xffffffffu, so - sn, l);
      long long* col = reinterpret_cast<long long*>(V) + (q - lane + l) + (size_t)lane * ldv;
      for (int c = lane; c < j; c += 32, col += 32 * ldv)
        __stcg(col, fx_less_shift(__ldcg(col), d));
    }
  }
}

// w and u_j (for two dots) of n rows, at Ws and Us, as operands of the fixed-point dots in place: ew,
// eu the largest exponents of w in the super-tile and of u_j.  V, w and Sg point at the first row;
// the first `live` rows exist.  (A call of its own: inlined it would spill registers around the dots.)
template <int NSET>
__device__ __noinline__ void arn_operands(double* V, long long ldv, const double* w, short* Sg, int j,
                                          int n, int live, int ew, int eu, double* Ws, double* Us) {
  constexpr int B = 4;  // rows per thread whose shifts are loaded at once
  int2* const Wf = reinterpret_cast<int2*>(Ws);
  int2* const Uf = reinterpret_cast<int2*>(Us);
  for (int q0 = threadIdx.x; q0 < n; q0 += B * kArnThreads) {
    int sh[B];
    if (j > 0) {
#pragma unroll
      for (int b = 0; b < B; ++b)
        sh[b] = q0 + b * kArnThreads < n ? __ldcg(Sg + q0 + b * kArnThreads) : 0;
    } else {
#pragma unroll
      for (int b = 0; b < B; ++b) {
        const int q = q0 + b * kArnThreads;
        sh[b] = q < n ? arn_shift_of(Sg + q, 0, Us[q], eu, q < live) : 0;
      }
    }
    unsigned grow = 0;  // rows whose shift is too large for u_j
#pragma unroll
    for (int b = 0; b < B; ++b) {
      const int q = q0 + b * kArnThreads;
      if (q < n) {
        const double u = Us[q];
        grow |= (fx_mag(u) >> 20 > max(eu - sh[b], 0) ? 1u : 0u) << b;
        Wf[q] = fx_operand(Ws[q], ew + sh[b]);
        if (NSET == 2) Uf[q] = fx_operand(u, eu + sh[b]);
      }
    }
    const unsigned any = __reduce_or_sync(0xffffffffu, grow);
    if (any) arn_grow<NSET>(V, ldv, w, Sg, j, q0, any, grow, ew, eu, Wf, Uf);
  }
}

// SpMV, coarse correction and multi-dot of step j over the block's super-tiles (a function
// of its own, so that the cycle loop's state stays out of these loops' registers)
template <typename TV, typename TACC, int ND, int MODE>
__device__ __forceinline__ void arn_front(const ArnArgs<TV, TACC>& a, const ArnRows& g, int j, TACC sig, bool waited,
                                       bool first_diag_done, TACC* Ws, TACC* Us, TACC* Ss,
                                       double* sbuf, const int* sE, int* semax, double* sred) {
  constexpr int VN = ArnVec<TV>::n;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = threadIdx.x;
  const long long R0 = g.R0, R1 = g.R1;
  const long long N = a.N;
  const int k = j + 1;
  const bool multi = R1 - R0 > a.RS;  // w goes through global memory to the update
  int tile = 0;
  for (long long s0 = R0; s0 < R1; s0 += a.RS, ++tile) {
    const long long s1 = s0 + a.RS < R1 ? s0 + a.RS : R1;
    // ---- 1. SpMV of the super-tile's rows: w and u_j into shared memory (the first
    // super-tile's may have been formed during the previous step's coarse solve) ---------
    if (!(first_diag_done && s0 == R0)) arn_diag<ND, TV, TACC>(a, j, s0, s1, Ws, Us, t, kArnThreads);
    // + A W s' (the row's A W entries, s' from shared memory), the scale sigma_j; w also to
    // global memory when the update reads it there.
    if constexpr (sizeof(TACC) == 8) {
      // FP64 (every FP64 instruction costs the scarce FP64 pipe): the CSR rows, kArnAwRows64
      // rows per thread at once, each level of the gather (row pointers, then the first entry
      // of every row) issued for all of them; s' is staged pre-scaled by sigma_j, so that
      // w = sigma_j Ws + sum a_iq (sigma_j s'_q) takes one multiply-add per entry and row
      if (!waited) {  // s' (the coarse solve's output) is read from here on
        pdl_wait();
        pdl_trigger();
        waited = true;
      }
      if (a.defl && s0 == R0)
        for (int q = t; q < a.r; q += kArnThreads) Ss[q] = sig * __ldcg(a.sdefl + q);
      if (t == 0) semax[0] = 0;
      __syncthreads();
      int mw = 0;  // high word of the largest |w| of the super-tile
      constexpr int AWR = kArnAwRows64;
      for (long long i0 = s0 + t; i0 < s1; i0 += (long long)AWR * kArnThreads) {
        int e0[AWR], e1[AWR];
#pragma unroll
        for (int b = 0; b < AWR; ++b) {
          const long long row = i0 + (long long)b * kArnThreads;
          const bool live = a.defl && row < N && row < s1;
          e0[b] = live ? __ldg(a.aurp + row) : 0;
          e1[b] = live ? __ldg(a.aurp + row + 1) : 0;
        }
        TACC av[AWR];
        int ac[AWR];
#pragma unroll
        for (int b = 0; b < AWR; ++b) {
          const bool has = e0[b] < e1[b];
          av[b] = has ? __ldg(a.auval + e0[b]) : (TACC)0;
          ac[b] = has ? __ldg(a.aucol + e0[b]) : 0;
        }
#pragma unroll
        for (int b = 0; b < AWR; ++b) {
          const long long row = i0 + (long long)b * kArnThreads;
          if (row < s1) {
            TACC wv = 0;
            if (row < N) {
              TACC aw = a.defl ? av[b] * Ss[ac[b]] : (TACC)0;
              for (int e = e0[b] + 1; e < e1[b]; ++e) aw += __ldg(a.auval + e) * Ss[__ldg(a.aucol + e)];
              wv = fma(sig, Ws[row - s0], aw);
              a.w[row] = wv;  // the update reads w there
            }
            Ws[row - s0] = wv;
            mw = max(mw, fx_mag(wv));
          }
        }
      }
      mw = __reduce_max_sync(0xffffffffu, mw);
      if (lane == 0) atomicMax(&semax[0], mw);
    } else {
      // FP32: a row's first two A W entries from the row-indexed planes (one level of loads,
      // kArnAwRows32 rows per thread at once); the first batch's loads are issued before s'
      // is read, since they do not depend on it
      constexpr int AWR = kArnAwRows32;
      TACC av0[AWR], av1[AWR];
      int ac0[AWR], ac1[AWR];
      auto aw_load = [&](long long i0) {
#pragma unroll
        for (int b = 0; b < AWR; ++b) {
          const long long row = i0 + (long long)b * kArnThreads;
          const bool live = a.defl && row < N && row < s1;
          ac0[b] = live ? __ldg(a.aup_col + row) : -1;
          ac1[b] = live ? __ldg(a.aup_col + N + row) : -1;
          av0[b] = live ? __ldg(a.aup_val + row) : (TACC)0;
          av1[b] = live ? __ldg(a.aup_val + N + row) : (TACC)0;
        }
      };
      auto aw_apply = [&](long long i0) {
#pragma unroll
        for (int b = 0; b < AWR; ++b) {
          const long long row = i0 + (long long)b * kArnThreads;
          if (row < s1) {
            // absent entries carry the value 0 (and read s'_0, which is finite)
            TACC aw = 0;
            if (a.defl) {
              aw = av0[b] * Ss[ac0[b] >= 0 ? ac0[b] : 0];
              aw += av1[b] * Ss[ac1[b] >= 0 ? ac1[b] : (ac1[b] == -1 ? 0 : -ac1[b] - 2)];
              if (ac1[b] < -1) {  // the row's third and later entries (rare)
                const int e1 = __ldg(a.aurp + row + 1);
#pragma unroll 1
                for (int e = __ldg(a.aurp + row) + 2; e < e1; ++e)
                  aw += __ldg(a.auval + e) * Ss[__ldg(a.aucol + e)];
              }
            }
            const TACC wv = row < N ? sig * (Ws[row - s0] + aw) : (TACC)0;
            Ws[row - s0] = wv;
            if (multi && row < N) a.w[row] = wv;
          }
        }
      };
      aw_load(s0 + t);
      if (!waited) {  // s' (the coarse solve's output) is read from here on
        pdl_wait();
        pdl_trigger();
        waited = true;
      }
      if (a.defl && s0 == R0)
        for (int q = t; q < a.r; q += kArnThreads) Ss[q] = __ldcg(a.sdefl + q);
      __syncthreads();
      for (long long i0 = s0 + t; i0 < s1; i0 += (long long)AWR * kArnThreads) {
        if (i0 != s0 + t) aw_load(i0);
        aw_apply(i0);
      }
    }
    __syncthreads();
    const int nch = (int)((s1 - s0) / (32 * VN));
    constexpr int NSET = MODE == kArnCgs2 ? 1 : 2;  // w alone, or w and u_j
    if constexpr (sizeof(TV) == 8) {
      // w and u_j to fixed point in place (relative to the largest exponent of w in the
      // super-tile, of u_j as a whole), then the dots with every column
      const int ew = semax[0] >> 20, eu = sE[j], n = (int)(s1 - s0);
      short* const Sg = arn_shifts(a) + s0;
      if constexpr (MODE == kArnLowsyncDf) {
        // w and u_j split in place (float2 hi, lo in the 8 bytes of each double)
        for (int q = t; q < n; q += kArnThreads) {
          arn_shift_of(Sg + q, j, Us[q], eu, s0 + q < N);
          float h1, l1, h2, l2;
          arn_df_split((double)Ws[q], h1, l1);
          arn_df_split((double)Us[q], h2, l2);
          reinterpret_cast<float2*>(Ws)[q] = make_float2(h1, l1);
          reinterpret_cast<float2*>(Us)[q] = make_float2(h2, l2);
        }
        __syncthreads();
        arn_dots_df(reinterpret_cast<float*>(sbuf), reinterpret_cast<const double*>(a.V), a.ldv,
                    k, s0, nch, reinterpret_cast<const float2*>(Ws),
                    reinterpret_cast<const float2*>(Us), warp, lane);
        __syncthreads();
        continue;
      }
      arn_operands<NSET>(reinterpret_cast<double*>(const_cast<TV*>(a.V)) + s0, a.ldv, a.w + s0, Sg, j, n,
                         (int)min(N - s0, (long long)n), ew, eu, Ws, Us);
      __syncthreads();
      int4* slot = reinterpret_cast<int4*>(sbuf);
      arn_dots_fx<NSET, (NSET == 2 ? kArnFxGroup : kArnFxGroup1), kArnFxDepth>(
          slot, reinterpret_cast<const double*>(a.V), a.ldv, j, k, eu, s0, nch,
          reinterpret_cast<const int4*>(Ws), reinterpret_cast<const int4*>(Us), arn_shifts(a), lane);
      __syncthreads();
      arn_slot_sums<NSET>(slot, nch, k, sE, ew, eu, tile == 0, sred);
    } else {
      arn_dots_rows<TV, TACC, NSET, arn_group<ND>()>(sbuf, a.V, a.ldv, k, s0, nch, arn_share(a, g.G),
                                                     Ws, Us, lane);
    }
    __syncthreads();  // the slices are rewritten by the next super-tile
  }
}

// The update's part of the reduction scratch: the coefficients at its end, past one dot set's slots
// (CGS2's second multi-dot) and the split update's partial sums
__device__ __forceinline__ int4* arn_sk(double* sbuf) {
  static_assert(kArnScratch >= (15 * 32 * 3 + kMaxK) * 16, "partial sums and coefficients");
  static_assert(kArnScratch >= (kArnWarps + 1) * kMaxK * 16, "slots and coefficients");
  return reinterpret_cast<int4*>(sbuf) + kArnScratch / 16 - kMaxK;
}

// w - V (sigma o h) of the rows [s0, s1) (an FP64 basis): a row's sum of M_c K_c (at most kMaxK
// terms) stays in integer accumulators, and FP64 enters once per row; put(r, value of row r, of
// row r + 1, their shifts) takes the results.  FIXED: the first kf columns are fixed-point integers, a last one
// (k = kf + 1) is FP64 and is converted in place on the way (no other block reads it any more:
// the SpMV is behind the last grid barrier); else all columns are FP64 and stay so.  Each loaded
// value's register is reloaded U columns on (past the last column: from the warp's next chunk)
// as soon as it is used.  With fewer than 16 chunks the warps of a chunk share its columns and
// add their integer sums through sP.  Bound by the basis loads; FP64 multiply-adds would cost 64
// issue slots per entry, this form about 7.  Called by all threads.
constexpr int kArnUpdLoads = 6;  // basis loads in flight per lane

template <bool FIXED, typename F>
__device__ __forceinline__ void arn_rows_update_fx(const double* V, long long ldv,
                                                   const short* Sg, const double* w, int N,
                                                   long long s0, long long s1,
                                                   int kf, int k, const int* sE, const int4* sK,
                                                   double nscale, longlong2* sP, F&& put) {
  constexpr int U = kArnUpdLoads;
  const int lane = threadIdx.x & 31;
  const int nch = (int)((s1 - s0) >> 6);
  const ArnSplit sp = arn_split(nch);
  const int c0 = sp.p * kf / sp.S, c1 = (sp.p + 1) * kf / sp.S;
  long long r = s0 + (long long)(nch - 1 - sp.q0) * 64 + lane * 2;
  const bool one = sp.S > 1;
  const long long* const Vi = reinterpret_cast<const long long*>(V);
  // the FP64 column's part of the rows at r, then the finished rows
  auto finish = [&](FxAcc& a0, FxAcc& a1) {
    const double2 wv = __ldcg(reinterpret_cast<const double2*>(w + r));
    const short2 sh = __ldcg(reinterpret_cast<const short2*>(Sg + r));
    if (FIXED && kf < k) {
      double* pj = const_cast<double*>(V) + (size_t)kf * ldv + r;
      const double2 v = __ldcg(reinterpret_cast<const double2*>(pj));
      const long long m0 = fx_basis(v.x, sE[kf] - sh.x), m1 = fx_basis(v.y, sE[kf] - sh.y);
      *reinterpret_cast<longlong2*>(pj) = make_longlong2(m0, m1);
      fx_axpy(a0, fx_limbs(m0), sK[kf]);
      fx_axpy(a1, fx_limbs(m1), sK[kf]);
    }
    double n0 = nscale, n1 = nscale;
    if (sh.x | sh.y) {
      n0 *= fx_pow2(sh.x);
      n1 *= fx_pow2(sh.y);
    }
    // rows past N: w and the basis are zeros there, and stay so when a coefficient is not finite
    put(r, r < N ? fx_axpy_add(a0, wv.x, n0) : 0.0, r + 1 < N ? fx_axpy_add(a1, wv.y, n1) : 0.0, sh);
  };
  FxAcc a0{0, 0, 0, 0}, a1{0, 0, 0, 0};
  if (sp.live && (!one || c0 < c1)) {
    int nb = c0;  // column and row of the next load
    long long nr = r;
    const long long* pn = Vi + (size_t)c0 * ldv + r;
    uint4 v[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      v[u] = make_uint4(0, 0, 0, 0);
      if (nb + u < c1) arn_ldfx(pn + (size_t)u * ldv, v[u]);
    }
    for (; r >= s0; r -= kArnWarps * 64) {
      if (!one) a0 = a1 = FxAcc{0, 0, 0, 0};
      short2 sr = make_short2(0, 0);
      if (!FIXED) sr = __ldcg(reinterpret_cast<const short2*>(Sg + r));
#pragma unroll 1
      for (int b = c0; b < c1; b += U) {
        nb += U;
        pn += (size_t)U * ldv;
        if (nb >= c1) {  // on to the next chunk
          nb = c0;
          nr -= kArnWarps * 64;
          pn = Vi + (size_t)c0 * ldv + nr;
        }
        const bool more = nr >= s0 && (!one || nb > c0);
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const bool on = b + u < c1;
          Fx f0, f1;
          if (FIXED) {
            f0 = fx_limbs(v[u].x, v[u].y);
            f1 = fx_limbs(v[u].z, v[u].w);
          } else {
            const int e = sE[on ? b + u : c0];
            f0 = fx_limbs(fx_basis(__hiloint2double((int)v[u].y, (int)v[u].x), e - sr.x));
            f1 = fx_limbs(fx_basis(__hiloint2double((int)v[u].w, (int)v[u].z), e - sr.y));
          }
          if (more && nb + u < c1) arn_ldfx(pn + (size_t)u * ldv, v[u]);
          if (on) {
            const int4 kc = sK[b + u];
            fx_axpy(a0, f0, kc);
            fx_axpy(a1, f1, kc);
          }
        }
      }
      if (one) break;
      finish(a0, a1);
    }
  }
  if (!one) return;
  // sP[part][chunk][lane][3]: hh, hl with the leading l kl, lh of both rows
  if (sp.live && sp.p > 0) {
    longlong2* q = sP + ((size_t)((sp.p - 1) * nch + sp.q0) * 32 + lane) * 3;
    q[0] = make_longlong2(a0.hh, a1.hh);
    q[1] = make_longlong2(a0.hl + 4ll * a0.ll, a1.hl + 4ll * a1.ll);
    q[2] = make_longlong2(a0.lh, a1.lh);
  }
  __syncthreads();
  if (sp.live && sp.p == 0) {
    for (int p = 1; p < sp.S; ++p) {
      const longlong2* q = sP + ((size_t)((p - 1) * nch + sp.q0) * 32 + lane) * 3;
      const longlong2 hh = q[0], hl = q[1], lh = q[2];
      a0.hh += hh.x; a0.hl += hl.x; a0.lh += lh.x;
      a1.hh += hh.y; a1.hl += hl.y; a1.lh += lh.y;
    }
    finish(a0, a1);
  }
}

// the coefficients (sK) and minus the unit of the sum (sscale), the same in every block; called by
// all threads, ends with a barrier
__device__ __forceinline__ void arn_fx_coefs(int k, const double* scoef, const int* sE, int4* sK,
                                             double* sscale) {
  if (threadIdx.x < 32) {
    const double s = fx_coefs(k, scoef, sE, sK);
    if (threadIdx.x == 0) *sscale = -s;
  }
  __syncthreads();
}

// u_{j+1} of the block's rows into vout unless null (and ush, indexed from R0); returns the warp's part of
// ||u_{j+1}||^2, and in mx the high word of the thread's largest |u_{j+1}|.  kf: the columns
// already in fixed point
template <bool FIXED>
__device__ __forceinline__ double arn_update_fx(const double* V, long long ldv, const short* Sg,
                                                double* vout, const double* w, int N,
                                                long long R0, long long R1,
                                                int kf, int k, const double* scoef,
                                                const int* sE, double* sbuf, double* sscale,
                                                double* ush, int& mx) {
  int4* sK = arn_sk(sbuf);
  double nrm = 0.0;
  int m = 0;
  arn_fx_coefs(k, scoef, sE, sK, sscale);
  arn_rows_update_fx<FIXED>(
      V, ldv, Sg, w, N, R0, R1, kf, k, sE, sK, *sscale, reinterpret_cast<longlong2*>(sbuf),
      [&](long long r, double u0, double u1, short2) {
        if (vout) *reinterpret_cast<double2*>(vout + r) = make_double2(u0, u1);
        if (ush) *reinterpret_cast<double2*>(ush + (r - R0)) = make_double2(u0, u1);
        nrm = fma(u0, u0, fma(u1, u1, nrm));
        m = max(m, max(fx_mag(u0), fx_mag(u1)));
      });
  mx = m;
  return warp_sum(nrm);
}

// CGS2, first update and second multi-dot of an FP64 basis: per super-tile (from the last) w -= V
// (sigma o h) into w and shared memory (the newest column becomes fixed-point on the way), its
// operand form, then V^T w into sred
__device__ __forceinline__ void arn_pass2_fx(const double* V, long long ldv, const short* Sg,
                                             double* w, int N, int RS, long long R0, long long R1,
                                             int k,
                                             const double* scoef, const int* sE, double* Ws,
                                             double* sbuf, int* semax, double* sscale,
                                             double* sred) {
  const int lane = threadIdx.x & 31;
  int4* slot = reinterpret_cast<int4*>(sbuf);
  int4* sK = arn_sk(sbuf);
  const int tiles = (int)((R1 - R0 + RS - 1) / RS);
  __syncthreads();  // scoef
  arn_fx_coefs(k, scoef, sE, sK, sscale);
  for (int tile = tiles - 1; tile >= 0; --tile) {
    const long long s0 = R0 + (long long)tile * RS;
    const long long s1 = s0 + RS < R1 ? s0 + RS : R1;
    if (threadIdx.x == 0) semax[0] = 0;
    __syncthreads();
    int mw = 0;
    arn_rows_update_fx<true>(
        V, ldv, Sg, w, N, s0, s1, k - 1, k, sE, sK, *sscale, reinterpret_cast<longlong2*>(sbuf),
        [&](long long r, double u0, double u1, short2 sh) {
          *reinterpret_cast<double2*>(w + r) = make_double2(u0, u1);
          if (sh.x | sh.y) {  // (the operand's shift, ahead of the conversion)
            u0 *= fx_pow2(sh.x);
            u1 *= fx_pow2(sh.y);
          }
          *reinterpret_cast<double2*>(Ws + (r - s0)) = make_double2(u0, u1);
          mw = max(mw, max(fx_mag(u0), fx_mag(u1)));
        });
    mw = __reduce_max_sync(0xffffffffu, mw);
    if (lane == 0) atomicMax(&semax[0], mw);
    __syncthreads();
    const int ew = semax[0] >> 20;
    for (int q = threadIdx.x; q < (int)(s1 - s0); q += kArnThreads)
      reinterpret_cast<int2*>(Ws)[q] = fx_operand(Ws[q], ew);
    __syncthreads();
    const int nch = (int)((s1 - s0) >> 6);
    arn_dots_fx<1, kArnFxGroup1, kArnFxDepth>(slot, V, ldv, k, k, 0, s0, nch,
                                 reinterpret_cast<const int4*>(Ws), nullptr, Sg, lane);
    __syncthreads();
    arn_slot_sums<1>(slot, nch, k, sE, ew, 0, tile == tiles - 1, sred);
  }
  __syncthreads();
}

// u_{j+1} = w - V (sigma o h) over the block's rows of an FP32 or BF16 basis (also into ush, indexed from
// the block's first row, when given); returns the warp's part of ||u_{j+1}||^2 (in every lane)
// (PASS2: only the rows [base, end), w back into Ws, indexed from base, and global memory)
template <typename TV, typename TACC, bool PASS2>
__device__ __forceinline__ double arn_update(const ArnArgs<TV, TACC>& a, const ArnRows& g, int k, TACC* Ws,
                                          const TACC* scoef, TACC* ush, long long base,
                                          long long end, float* sP) {
  constexpr int VN = ArnVec<TV>::n;
  constexpr int U = PASS2 ? 6 : 8;  // basis loads in flight per lane, reloaded as they are used
  constexpr int chunk = 32 * VN;
  const int lane = threadIdx.x & 31;
  const long long R0 = g.R0, R1 = g.R1;
  const long long N = a.N;
  TV* __restrict__ vout = const_cast<TV*>(a.V) + (size_t)k * a.ldv;
  float ns = 0.f, nc = 0.f;  // a double-FP32 pair (FP64 adds are dear)
  const int nch = (int)((end - base) / chunk);
  const bool wsm = R1 - R0 <= a.RS;  // the block's w is still in shared memory
  const ArnSplit sp = arn_split32(arn_share(a, g.G), nch);
  const bool one = sp.S > 1;
  const int c0 = sp.p * k / sp.S, c1 = (sp.p + 1) * k / sp.S;
  long long r = base + (long long)(nch - 1 - sp.q0) * chunk + (long long)lane * VN;
  TACC p[VN];
  auto finish = [&] {
    TACC wv[VN], un[VN];
    if (wsm) {
      ld_acc<VN>(Ws + (r - R0), wv);
    } else {
#pragma unroll
      for (int e = 0; e < VN; ++e) wv[e] = r + e < N ? __ldcg(a.w + r + e) : (TACC)0;
    }
#pragma unroll
    for (int e = 0; e < VN; ++e) un[e] = r + e < N ? wv[e] - p[e] : (TACC)0;  // (as in FP64)
    if constexpr (PASS2) {  // CGS2's first update: w stays where it came from
      if (wsm) {
        acc_store<VN>(Ws + (r - R0), un);
      } else {
        acc_store<VN>(a.w + r, un);
        acc_store<VN>(Ws + (r - base), un);
      }
    } else {
      arn_stv<TV, TACC, VN>(vout + r, un);
      if constexpr (sizeof(TV) == 2) {  // the stored (rounded) values count
#pragma unroll
        for (int e = 0; e < VN; ++e) un[e] = __bfloat162float(__float2bfloat16_rn(un[e]));
      }
      if (ush) acc_store<VN>(ush + (r - R0), un);  // for the piece sums
      TACC s = 0;
#pragma unroll
      for (int e = 0; e < VN; ++e) s += un[e] * un[e];
      arn_df_add(ns, nc, s, 0.f);
    }
  };
#pragma unroll
  for (int e = 0; e < VN; ++e) p[e] = 0;
  if (sp.live) {
    int nb = c0;  // column and row of the next load
    long long nr = r;
    TACC v[U][VN];
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int e = 0; e < VN; ++e) v[u][e] = 0;
      if (nb + u < c1) arn_ldg<TV, TACC, VN>(a.V + (size_t)(nb + u) * a.ldv + nr, v[u]);
    }
    for (; r >= base; r -= (long long)kArnWarps * chunk) {
#pragma unroll
      for (int e = 0; e < VN; ++e) p[e] = 0;
#pragma unroll 1
      for (int b = c0; b < c1; b += U) {
        nb += U;
        if (nb >= c1) {  // on to the warp's next chunk
          nb = c0;
          nr -= (long long)kArnWarps * chunk;
        }
        const bool more = nr >= base && (!one || nb > c0);
        const TV* pn = a.V + (size_t)nb * a.ldv + nr;
#pragma unroll
        for (int u = 0; u < U; ++u) {
          if (b + u < c1) {
            const TACC cf = scoef[b + u];
#pragma unroll
            for (int e = 0; e < VN; ++e) p[e] += v[u][e] * cf;
          }
          if (more && nb + u < c1) arn_ldg<TV, TACC, VN>(pn + (size_t)u * a.ldv, v[u]);
        }
      }
      if (one) break;
      finish();
    }
  }
  if (one) {  // the shares' partial sums, added in order
    if (sp.live && sp.p > 0) acc_store<VN>(sP + ((size_t)((sp.p - 1) * sp.rows + sp.q0) * 32 + lane) * VN, p);
    __syncthreads();
    if (sp.live && sp.p == 0) {
      for (int q = 1; q < sp.S; ++q) {
        TACC o[VN];
        ld_acc<VN>(sP + ((size_t)((q - 1) * sp.rows + sp.q0) * 32 + lane) * VN, o);
#pragma unroll
        for (int e = 0; e < VN; ++e) p[e] += o[e];
      }
      finish();
    }
  }
  if constexpr (PASS2) {
    return 0.0;
  } else {  // the warp's total in double-FP32, rounded once
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float a2 = __shfl_xor_sync(0xffffffffu, ns, o);
      const float b2 = __shfl_xor_sync(0xffffffffu, nc, o);
      arn_df_add(ns, nc, a2, b2);
    }
    return (double)ns + (double)nc;
  }
}

// CGS2, first update and second multi-dot of an FP32 or BF16 basis: per super-tile (from the last)
// w -= V (sigma o h), then V^T w into the per-warp pairs
template <typename TV, typename TACC, int ND>
__device__ __forceinline__ void arn_pass2_rows(const ArnArgs<TV, TACC>& a, const ArnRows& g, int k, TACC* Ws,
                                            const TACC* scoef, double* sbuf) {
  const int lane = threadIdx.x & 31;
  const long long R0 = g.R0, R1 = g.R1;
  const int tiles = (int)((R1 - R0 + a.RS - 1) / a.RS);
  for (int tile = tiles - 1; tile >= 0; --tile) {
    const long long s0 = R0 + (long long)tile * a.RS;
    const long long s1 = s0 + a.RS < R1 ? s0 + a.RS : R1;
    __syncthreads();
    arn_update<TV, TACC, true>(a, g, k, Ws, scoef, nullptr, s0, s1,
                               reinterpret_cast<float*>(sbuf));
    __syncthreads();
    if (tile == tiles - 1) {  // (the shares of a chunk, one super-tile only, used sbuf)
      for (int q = threadIdx.x; q < kMaxK * kArnWarps; q += kArnThreads) sbuf[q] = 0.0;
      __syncthreads();
    }
    arn_dots_rows<TV, TACC, 1, arn_group<ND>()>(sbuf, a.V, a.ldv, k, s0,
                                                (int)((s1 - s0) / (32 * ArnVec<TV>::n)),
                                                arn_share(a, g.G), Ws, nullptr, lane);
  }
  __syncthreads();
}

// Sums of u_{j+1} over this block's aggregate pieces (c of the next step's coarse solve, by
// pieces, a warp each).  The pieces' bounds are loaded up front (lane i < 8 holds the
// warp's i-th piece), then per piece the node indexes and the values: from the shared-memory
// copy of the block's rows when there is one (ush, from row R0), else through L2 (this
// block wrote them just before).  Fixed order throughout.
template <bool C32, typename TV, typename TACC>
__device__ __forceinline__ void arn_piece_sums(const ArnArgs<TV, TACC>& a, const TV* vout,
                                               const TACC* ush, const ArnRows& g) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const long long R0 = g.R0;
  const int p0 = __ldg(a.blk_piece_start + g.f0), p1 = __ldg(a.blk_piece_start + g.f1);
  for (int base = p0 + warp; base < p1; base += kArnWarps * 8) {
    const int pi = base + kArnWarps * lane;
    int mp = -1, ms = 0, me = 0;
    if (lane < 8 && pi < p1) {
      mp = __ldg(a.blk_piece + pi);
      ms = __ldg(a.piece_start + mp);
      me = __ldg(a.piece_start + mp + 1);
    }
    for (int i = 0; i < 8; ++i) {
      const int p = __shfl_sync(0xffffffffu, mp, i);
      const int s = __shfl_sync(0xffffffffu, ms, i), e = __shfl_sync(0xffffffffu, me, i);
      if (p < 0) break;
      double acc[2] = {0.0, 0.0};
      for (int o = s; o < e; o += 32 * 8) {
        int node[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int q = o + lane + 32 * u;
          node[u] = q < e ? __ldg(a.perm + q) : -1;
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          double v = 0.0;
          if (node[u] >= 0) v = ush ? (double)ush[node[u] - R0] : arn_ldcg_d(vout + node[u]);
          acc[u & 1] += v;
        }
      }
      const double sum = warp_sum(acc[0] + acc[1]);
      if (lane == 0) {
        if constexpr (!C32) {
          __stcg(a.ctl.cpart + p, sum);
        } else {  // the pair the FP32 coarse solve reads
          const float hs = (float)sum;
          __stcg(reinterpret_cast<float2*>(a.ctl.cpart + p), make_float2(hs, (float)(sum - (double)hs)));
        }
      }
    }
  }
}

// The same sums from the staged node list: a warp per piece, values from the shared-memory
// copy of u_{j+1}.  FP64 rows add in FP64; FP32 rows in double-FP32 (TwoSum on the FP32
// pipe, exact to about 2^-48 of the sum's magnitude), rounded to FP64 once per piece.
constexpr int kArnMaxBlkPieces = 256;

template <bool C32, typename TACC>
__device__ __forceinline__ void arn_piece_sums_staged(double* cpart, const TACC* ush,
                                                      const unsigned short* snode,
                                                      const int* spid, const int* spls, int np) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = warp; i < np; i += kArnWarps) {
    const int ls = spls[i], le = spls[i + 1];
    if constexpr (!C32) {
      double acc[2] = {0.0, 0.0};
      for (int q = ls + lane; q < le; q += 64) {
        acc[0] += (double)ush[snode[q]];
        if (q + 32 < le) acc[1] += (double)ush[snode[q + 32]];
      }
      const double sum = warp_sum(acc[0] + acc[1]);
      if (lane == 0) __stcg(cpart + spid[i], sum);
    } else {
      float hs = 0.f, hc = 0.f;
      for (int q = ls + lane; q < le; q += 32) arn_df_add(hs, hc, (float)ush[snode[q]], 0.f);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float a2 = __shfl_xor_sync(0xffffffffu, hs, o);
        const float b2 = __shfl_xor_sync(0xffffffffu, hc, o);
        arn_df_add(hs, hc, a2, b2);
      }
      // an FP32 basis keeps the pair (two floats in the slot) for the FP32 coarse solve
      if (lane == 0) __stcg(reinterpret_cast<float2*>(cpart + spid[i]), make_float2(hs, hc));
    }
  }
}

// The block's largest high word of |u| (the warp's lanes hold the candidates) into its slot of the
// partials, and after a grid barrier the largest exponent over all blocks (one warp each)
__device__ __forceinline__ void arn_put_max(Ctl& ctl, int bid, int m) {
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0)
    __stcg(&ctl.part[(size_t)bid * ctl.ldp + kArnMaxCol], __hiloint2double(0, m));
}
__device__ __forceinline__ int arn_get_max(const Ctl& ctl, int G) {
  int m = 0;
  for (int b = threadIdx.x & 31; b < G; b += 32)
    m = max(m, __double2loint(__ldcg(&ctl.part[(size_t)b * ctl.ldp + kArnMaxCol])));
  return __reduce_max_sync(0xffffffffu, m) >> 20;
}

// The 16 warps' pairs of ncols columns (sets of k) in warp order: double-FP32 multi-dots of an
// FP64 basis rounded to FP64 once, sums of an FP32 or BF16 basis kept as pairs.  A block without
// rows (none: some blocks of a small system's cluster) has passed no barrier since the pairs were
// cleared, so it does not read them.
template <typename TV, int MODE>
__device__ __forceinline__ void arn_block_sums(const double* sbuf, int ncols, int k, bool none,
                                               double* sred) {
  if (none) {
    for (int q = threadIdx.x; q < ncols; q += kArnThreads) sred[q] = 0.0;
  } else if constexpr (sizeof(TV) == 8 && MODE == kArnLowsyncDf) {
    for (int q = threadIdx.x; q < ncols; q += kArnThreads) {
      const int set = q / k, c = q % k;
      const float* dfp = reinterpret_cast<const float*>(sbuf);
      float s = 0.f, cc = 0.f;
      for (int w = 0; w < kArnWarps; ++w) {
        const float* p = dfp + ((size_t)w * kMaxK + c) * 4 + 2 * set;
        arn_df_add(s, cc, p[0], p[1]);
      }
      sred[q] = (double)s + (double)cc;
    }
  } else if constexpr (sizeof(TV) < 8) {
    for (int q = threadIdx.x; q < ncols; q += kArnThreads) {
      const int set = q / k, c = q % k;
      const float2* ws = reinterpret_cast<const float2*>(sbuf);
      float hs = 0.f, hc = 0.f;
      for (int w = 0; w < kArnWarps; ++w) {
        const float2 v = ws[(size_t)(set * kArnWarps + w) * kMaxK + c];
        arn_df_add(hs, hc, v.x, v.y);
      }
      reinterpret_cast<float2*>(sred)[q] = make_float2(hs, hc);
    }
  }
  __syncthreads();
}

// The cycle of one system by G blocks, this one bid; CL: the blocks are a cluster
template <typename TV, typename TACC, int ND, int MODE, bool CL>
__device__ __forceinline__ void arn_cycle(const ArnArgs<TV, TACC>& a, const int G, const int bid) {
  static_assert(MODE != kArnLowsyncDf || sizeof(TV) == 8, "the double-FP32 multi-dot takes an FP64 basis");
  static_assert(MODE == kArnCgs2 || sizeof(TV) == sizeof(TACC), "BF16 bases use CGS2");
  // the FP32 one-reduction step of a banded operator in a grid runs its coarse solve in FP32, every
  // other instantiation in FP64
  constexpr bool C32 = sizeof(TV) == 4 && MODE == kArnLowsync && ND != kArnCsr && !CL;
  constexpr int NSET = MODE == kArnCgs2 ? 1 : 2;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ double tot[2 * kMaxK + 1];
  __shared__ double sred[2 * kMaxK];
  __shared__ double sg[kMaxK];
  __shared__ TACC scoef[kMaxK];
  __shared__ double snrm[kArnWarps];
  __shared__ int smax[kArnWarps];
  __shared__ double ssig[kMaxK + 1];
  // FP64: the columns' largest exponents, of w in a super-tile, and the unit of an update
  __shared__ int sE[kMaxK + 1];
  __shared__ int semax[1];
  __shared__ double sscale;
  // the control block is read from the grid-constant parameter (no register copy)
  Ctl& ctl = const_cast<Ctl&>(a.ctl);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int t = threadIdx.x;
  const ArnRows g = arn_rows(a, G, bid);
  const long long R0 = g.R0, R1 = g.R1;
  // shared memory: w and u_j of a super-tile, s' (r), reduction scratch, the rows of L
  // (stride kMaxK)
  TACC* Ws = reinterpret_cast<TACC*>(smem);
  TACC* Us = Ws + a.RS;
  TACC* Ss = Us + a.RS;
  double* scratch = reinterpret_cast<double*>(
      smem + ((2 * (size_t)a.RS + (size_t)a.r) * sizeof(TACC) + 127) / 128 * 128);
  double* sL = scratch + kArnScratch / sizeof(double);
  double* sbuf = scratch;
  double* sc = reinterpret_cast<double*>(smem);  // c of the coarse solve (w, u_j are dead)

  if (!a.pre) {
    pdl_wait();
    pdl_trigger();
  }
  // the flag is final here (set by the previous cycle's last step, reset by the residual
  // kernel before this one started): the same value in every block
  if (__ldcg(&ctl.flags[F_CYCLE_DONE])) {
    if (a.pre) {
      pdl_wait();
      pdl_trigger();
    }
    return;
  }
  unsigned gen = CL ? 0u : *(volatile unsigned*)&a.gbar[1];  // advanced only once all arrive
  // the split barrier's counter: no block arrives before every block has passed the first
  // grid barrier, so all read the same base
  const unsigned cbase = CL ? 0u : *(volatile unsigned*)&a.gbar[2];
  for (int q = t; q < kMaxK * kMaxK; q += kArnThreads) sL[q] = 0.0;
  if (t == 0) ssig[0] = __ldcg(&ctl.sigma[0]);
  // the block's aggregate pieces for the whole cycle: their ids, local starts and nodes (as
  // offsets from R0, 16 bits) in shared memory, past the rows of u_j's slice, when the
  // block's rows fit one super-tile with room to spare (else the sums read perm from L2)
  __shared__ int spid[kArnMaxBlkPieces];
  __shared__ int spls[kArnMaxBlkPieces + 1];
  const long long nrows = R1 - R0;
  unsigned short* snode = reinterpret_cast<unsigned short*>(Us + nrows);
  const int bp0 = a.defl ? __ldg(a.blk_piece_start + g.f0) : 0;
  const int bp1 = a.defl ? __ldg(a.blk_piece_start + g.f1) : 0;
  const bool staged = a.defl && bp1 - bp0 <= kArnMaxBlkPieces && nrows <= 65536 &&
                      (size_t)nrows * sizeof(TACC) + (size_t)nrows * 2 <= (size_t)a.RS * sizeof(TACC);
  if (staged) {
    if (warp == 0) {  // ids and sizes 32 at a time, local starts by a warp scan
      int run = 0;
      for (int i0 = 0; i0 < bp1 - bp0; i0 += 32) {
        const int i = i0 + lane;
        int p = 0, n = 0;
        if (i < bp1 - bp0) {
          p = __ldg(a.blk_piece + bp0 + i);
          n = __ldg(a.piece_start + p + 1) - __ldg(a.piece_start + p);
        }
        int inc = n;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, inc, o);
          if (lane >= o) inc += v;
        }
        if (i < bp1 - bp0) {
          spid[i] = p;
          spls[i] = run + inc - n;
        }
        run += __shfl_sync(0xffffffffu, inc, 31);
      }
      if (lane == 0) spls[bp1 - bp0] = run;
    }
    __syncthreads();
    for (int i = warp; i < bp1 - bp0; i += kArnWarps) {
      const int p = spid[i];
      const int s = __ldg(a.piece_start + p), ls = spls[i], n = spls[i + 1] - ls;
      for (int q = lane; q < n; q += 32) snode[ls + q] = (unsigned short)(__ldg(a.perm + s + q) - R0);
    }
  }
  // FP32 basis: the coarse solve's static data for the cycle (the aggregates' piece ranges,
  // their scales, this block's rows of T^-1 when every warp has at most one) staged once in
  // shared memory, when it fits: past the rows of w's slice and past c, which the coarse solve
  // forms at the start of that slice (r entries, more than the rows of a small system's block)
  int* sap = nullptr;       // agg_piece, r + 1
  float* sus = nullptr;     // uscale, r
  float* stinv = nullptr;   // the block's rows of T^-1 (warp w: row (b - 1) + (G - 1) w)
  if constexpr (C32) {
    const int nwr = G == 1 ? kArnWarps : (G - 1) * kArnWarps;  // warps sharing the rows
    const int rows = (a.defl && bid > 0 && a.r <= nwr && bid - 1 < a.r)
                         ? min(kArnWarps, (a.r - (bid - 1) + G - 2) / (G - 1)) : 0;
    const size_t need = (size_t)(a.r + 1) * 4 + (size_t)a.r * 4 + (size_t)rows * a.r * 4;
    const long long at = nrows > a.r ? nrows : a.r;
    if (a.defl && G > 1 && a.RS > at && (size_t)(a.RS - at) * sizeof(TACC) >= need + 16) {
      sap = reinterpret_cast<int*>(Ws + at);
      sus = reinterpret_cast<float*>(sap + a.r + 1);
      stinv = rows > 0 ? sus + a.r : nullptr;
      for (int q = t; q <= a.r; q += kArnThreads) sap[q] = __ldg(a.agg_piece + q);
      for (int q = t; q < a.r; q += kArnThreads) sus[q] = (float)__ldg(a.uscale + q);
      for (int q = t; q < rows * a.r; q += kArnThreads) {
        const int w = q / a.r, b = q % a.r;
        stinv[q] = __ldg(a.tinv32 + (size_t)((bid - 1) + (G - 1) * w) * a.r + b);
      }
    }
  }
  bool waited = !a.pre;
  if constexpr (sizeof(TV) == 8) {  // the exponent of u_0: one more grid barrier per cycle
    if (!waited) {
      pdl_wait();
      pdl_trigger();
      waited = true;
    }
    int mx = 0;
    for (long long r = R0 + t; r < R1; r += kArnThreads) mx = max(mx, fx_mag(__ldcg(a.V + r)));
    mx = __reduce_max_sync(0xffffffffu, mx);
    if (lane == 0) smax[warp] = mx;
    __syncthreads();
    if (warp == 0) arn_put_max(ctl, bid, lane < kArnWarps ? smax[lane] : 0);
    if (!arn_grid_sync<CL>(a.gbar, gen++)) {
      arn_timeout(ctl);
      return;
    }
    if (warp == 0) {
      const int e = arn_get_max(ctl, G);
      if (lane == 0) sE[0] = e;
      if (lane == 0 && bid == 0) ctl.vexp[0] = e;
    }
  }
  __syncthreads();

  for (int j = 0; j < a.jmax; ++j) {
    const int k = j + 1;
    const TACC sig = (TACC)ssig[j];
    // the pairs per warp and column of an FP32, BF16 or double-FP32 multi-dot, which add up over
    // the super-tiles (fixed point stores its slots anew in each)
    if constexpr (sizeof(TV) < 8 || MODE == kArnLowsyncDf)
      for (int q = t; q < (int)(kArnScratch / sizeof(double)); q += kArnThreads) sbuf[q] = 0.0;
    arn_front<TV, TACC, ND, MODE>(a, g, j, sig, waited, j > 0, Ws, Us, Ss, sbuf, sE, semax, sred);
    waited = true;
    // per-block column sums (fixed order; a fixed-point multi-dot leaves them in sred)
    arn_block_sums<TV, MODE>(sbuf, NSET * k, k, R0 == R1, sred);
    // the partials: FP64 values, or double-FP32 pairs (two floats in the slot) for an FP32 or
    // BF16 basis, whose cross-block sums then run on the FP32 pipe
    for (int c = t; c < NSET * k; c += kArnThreads) __stcg(&ctl.part[(size_t)bid * ctl.ldp + c], sred[c]);
    // ---- 3. grid barrier; identical totals in every block -------------------------------
    if (!arn_grid_sync<CL>(a.gbar, gen++)) {
      arn_timeout(ctl);
      return;
    }
    if constexpr (sizeof(TV) < 8)
      // (a thread's 152 / 8 rows of partials in one batch of loads)
      arn_reduce_cols_df<24>(ctl.part, G, NSET * k, ctl.ldp, tot);  // ends with __syncthreads
    else
      arn_reduce_cols(ctl.part, G, NSET * k, ctl.ldp, tot);
    if constexpr (MODE == kArnCgs2) {
      // h = V^T w, first update and second multi-dot, one more barrier, h += h'
      for (int c = t; c < k; c += kArnThreads) {
        sg[c] = ssig[c] * tot[c];
        scoef[c] = (TACC)(ssig[c] * sg[c]);
      }
      if constexpr (sizeof(TV) == 8) {
        arn_pass2_fx(a.V, a.ldv, arn_shifts(a), a.w, a.N, a.RS, R0, R1, k, scoef, sE, Ws,
                     sbuf, semax, &sscale, sred);
      } else {
        arn_pass2_rows<TV, TACC, ND>(a, g, k, Ws, scoef, sbuf);
      }
      arn_block_sums<TV, MODE>(sbuf, k, k, R0 == R1, sred);
      // (columns of their own: another block may still be adding up the first dots' partials)
      double* const part2 = ctl.part + kMaxK;
      for (int c = t; c < k; c += kArnThreads) __stcg(&part2[(size_t)bid * ctl.ldp + c], sred[c]);
      if (!arn_grid_sync<CL>(a.gbar, gen++)) {
        arn_timeout(ctl);
        return;
      }
      if constexpr (sizeof(TV) < 8)
        arn_reduce_cols_df<24>(part2, G, k, ctl.ldp, tot);
      else
        arn_reduce_cols(part2, G, k, ctl.ldp, tot);
      for (int c = t; c < k; c += kArnThreads) {
        const double h2 = ssig[c] * tot[c];
        scoef[c] = (TACC)(ssig[c] * h2);
        if (bid == 0) ctl.h[c] = sg[c] + h2;
      }
      __syncthreads();
    } else {
      // (I + L) h = g; the new row of L: v_j . v_c = sigma_j sigma_c (u_j . u_c), c < j;
      // g_c = sigma_c (u_c . w)
      const double sj = ssig[k - 1];
      for (int c = t; c < k; c += kArnThreads) {
        if (c < k - 1) sL[(size_t)(k - 1) * kMaxK + c] = sj * ssig[c] * tot[k + c];
        sg[c] = ssig[c] * tot[c];
      }
      __syncthreads();
      if (warp == 0) {  // forward substitution: h_c final when reached (entries c, c+32, c+64)
        // sL[i][c] = 0 for c >= i, so rows at or above c take a zero update; only the
        // 32-row groups below k are touched (one FP64 FMA per group and column)
        const int nq = (k + 31) >> 5;
        double g[3];
#pragma unroll
        for (int q = 0; q < 3; ++q) g[q] = lane + 32 * q < k ? sg[lane + 32 * q] : 0.0;
        for (int c = 0; c < k; ++c) {
          const double hc = __shfl_sync(0xffffffffu, c < 32 ? g[0] : (c < 64 ? g[1] : g[2]), c & 31);
#pragma unroll
          for (int q = 0; q < 3; ++q) {
            const int i = lane + 32 * q;
            if (q < nq) g[q] -= (i < k ? sL[(size_t)i * kMaxK + c] : 0.0) * hc;
          }
        }
#pragma unroll
        for (int q = 0; q < 3; ++q) {
          const int i = lane + 32 * q;
          if (i < k) {
            scoef[i] = (TACC)(ssig[i] * g[q]);
            if (bid == 0) {
              ctl.h[i] = g[q];
              if (i < k - 1) ctl.L[(size_t)(k - 1) * kMaxK + i] = sL[(size_t)(k - 1) * kMaxK + i];
            }
          }
        }
      }
      __syncthreads();
    }
    // ---- 4. update u_{j+1} = w - V (sigma o h) and ||u_{j+1}||^2 ------------------------
    TV* __restrict__ vout = const_cast<TV*>(a.V) + (size_t)k * a.ldv;
    // a shared-memory copy of u_{j+1} for the piece sums when the block's rows fit one
    // super-tile (u_j's slice is dead by now)
    TACC* ush = (a.defl && k < a.jmax && R1 - R0 <= a.RS) ? Us : nullptr;
    double nrm;
    int mx = 0;
    if constexpr (sizeof(TV) == 8)
      nrm = arn_update_fx<MODE != kArnLowsyncDf>(
          a.V, a.ldv, arn_shifts(a), k < a.m ? vout : nullptr, a.w, a.N, R0, R1,
          MODE == kArnLowsync ? k - 1 : k, k, scoef, sE, sbuf, &sscale, ush, mx);
    else
      nrm = arn_update<TV, TACC, false>(a, g, k, Ws, scoef, ush, R0, R1,
                                          reinterpret_cast<float*>(sbuf));
    // ---- 5. norm partial; partial sums of u_{j+1} over this block's aggregate pieces ----
    {
      // the warp sums (formed by the update), then warp 0 adds the 16 of them (a block-wide
      // final loop would issue 16 FP64 adds in every warp)
      if (lane == 0) snrm[warp] = nrm;
      if constexpr (sizeof(TV) == 8) {
        mx = __reduce_max_sync(0xffffffffu, mx);
        if (lane == 0) smax[warp] = mx;
      }
      __syncthreads();  // also orders this block's stores of u_{j+1} before the piece sums
      if (warp == 0) {
        double bs = lane < kArnWarps ? snrm[lane] : 0.0;
#pragma unroll
        for (int o = kArnWarps / 2; o > 0; o >>= 1) bs += __shfl_xor_sync(0xffffffffu, bs, o);
        if (lane == 0) __stcg(&ctl.part[(size_t)bid * ctl.ldp + kArnNormCol], bs);
        if constexpr (sizeof(TV) == 8) arn_put_max(ctl, bid, lane < kArnWarps ? smax[lane] : 0);
      }
      if (a.defl && k < a.jmax) {
        if (staged && ush)
          arn_piece_sums_staged<C32>(ctl.cpart, ush, snode, spid, spls, bp1 - bp0);
        else
          arn_piece_sums<C32>(a, vout, ush, g);
      }
    }
    if (!arn_grid_sync<CL>(a.gbar, gen++)) {
      arn_timeout(ctl);
      return;
    }
    const bool coarse = a.defl && k < a.jmax && (bid > 0 || G == 1);
    // ---- 6. ||u_{j+1}|| and the plane rotations with the stopping tests (block 0); the next
    // step's coarse solve s' = U (|mu| T^-1 - I) U^T u_{j+1} (the other blocks) -------------
    const bool split0 = bid == 0 && G > 1;  // warp 0 alone: the others go on to the next SpMV
    if (bid == 0 && warp == 0) {
      double v = 0.0;
      for (int b = lane; b < G; b += 32) v += __ldcg(&ctl.part[(size_t)b * ctl.ldp + kArnNormCol]);
      givens_step(ctl, j, a.m, sqrt(warp_sum(v)));
      __syncwarp();
      if (CL) {
        if (split0) arn_cluster_arrive();
      } else if (split0 && lane == 0) {
        __threadfence();
        atomicAdd(&a.gbar[2], 1u);
      }
    }
    if (coarse) {
      // y = T^-1 c: a warp per row, the rows dealt round-robin over blocks 1 .. G-1 (warp w
      // of block b takes rows (b - 1) + (G - 1) (w + 16 i)) so that each block has few; all
      // to block 0 when it is alone.  TQ loads in flight per lane (a whole row up to 1024)
      constexpr int TQ = sizeof(TACC) == 4 && !C32 ? 16 : 32;
      const int gw = G == 1 ? warp : (bid - 1) + (G - 1) * warp;
      const int nw = G == 1 ? kArnWarps : (G - 1) * kArnWarps;
      if constexpr (!C32) {
        // c_a = uscale_a (sum of a's pieces, in piece order), every aggregate in every block
        for (int q = t; q < a.r; q += kArnThreads) {
          const int p0 = __ldg(a.agg_piece + q), p1 = __ldg(a.agg_piece + q + 1);
          double sum = 0.0;
          for (int pb = p0; pb < p1; pb += 8) {
            double v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = pb + u < p1 ? __ldcg(ctl.cpart + pb + u) : 0.0;
#pragma unroll
            for (int u = 0; u < 8; ++u) sum += v[u];
          }
          sc[q] = __ldg(a.uscale + q) * sum;
        }
        __syncthreads();
        const double mu = __ldcg(&ctl.scal[S_MU]);
        for (int row = gw; row < a.r; row += nw) {
          const double* tr = a.tinv + (size_t)row * a.r;
          double acc[2] = {0.0, 0.0};
          for (int b0 = 0; b0 < a.r; b0 += 32 * TQ) {
            double tv[TQ];
#pragma unroll
            for (int u = 0; u < TQ; ++u) {
              const int b = b0 + lane + 32 * u;
              tv[u] = b < a.r ? __ldg(tr + b) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < TQ; ++u) {
              const int b = b0 + lane + 32 * u;
              if (b < a.r) acc[u & 1] += tv[u] * sc[b];
            }
          }
          const double y = warp_sum(acc[0] + acc[1]);
          if (lane == 0) {
            const double sd = __ldg(a.uscale + row) * (mu * y - sc[row]);
            __stcg(ctl.sdefl + row, sd);
            __stcg(ctl.sdefl32 + row, (float)sd);
          }
        }
      } else {
        // FP32 basis: s' is used in FP32, so the coarse solve runs in FP32 too (c from the
        // double-FP32 piece pairs, rounded once; the FP32 copy of T^-1; FP32 sums)
        float* scf = reinterpret_cast<float*>(sc);
        for (int q = t; q < a.r; q += kArnThreads) {
          const int p0 = sap ? sap[q] : __ldg(a.agg_piece + q);
          const int p1 = sap ? sap[q + 1] : __ldg(a.agg_piece + q + 1);
          float hs = 0.f, hc = 0.f;
          for (int pb = p0; pb < p1; pb += 8) {
            float2 v[8];
#pragma unroll
            for (int u = 0; u < 8; ++u)
              v[u] = pb + u < p1 ? __ldcg(reinterpret_cast<const float2*>(ctl.cpart + pb + u))
                                 : make_float2(0.f, 0.f);
#pragma unroll
            for (int u = 0; u < 8; ++u) arn_df_add(hs, hc, v[u].x, v[u].y);
          }
          scf[q] = (sus ? sus[q] : (float)__ldg(a.uscale + q)) * (hs + hc);
        }
        __syncthreads();
        const float mu = (float)__ldcg(&ctl.scal[S_MU]);
        for (int row = gw; row < a.r; row += nw) {
          // the row from shared memory when staged (a plain load), else from global memory
          const float* tr = stinv ? stinv + (size_t)warp * a.r : a.tinv32 + (size_t)row * a.r;
          float acc[4] = {0.f, 0.f, 0.f, 0.f};
          for (int b0 = 0; b0 < a.r; b0 += 32 * TQ) {
            float tv[TQ];
#pragma unroll
            for (int u = 0; u < TQ; ++u) {
              const int b = b0 + lane + 32 * u;
              tv[u] = b < a.r ? tr[b] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < TQ; ++u) {
              const int b = b0 + lane + 32 * u;
              if (b < a.r) acc[u & 3] += tv[u] * scf[b];
            }
          }
          const float y = warp_sum((acc[0] + acc[1]) + (acc[2] + acc[3]));
          if (lane == 0) {
            const float sd = (sus ? sus[row] : (float)__ldg(a.uscale + row)) * (mu * y - scf[row]);
            __stcg(ctl.sdefl + row, (double)sd);
            __stcg(ctl.sdefl32 + row, sd);
          }
        }
      }
    }
    // this block's s' rows and (block 0) the rotations are published: arrive, then form the
    // diagonal part of the next step's SpMV for the first super-tile, which needs only
    // u_{j+1} (complete since the barrier), not s' or sigma_{j+1} (it overwrites c); then
    // wait for every block's arrival
    if (!split0) arn_arrive<CL>(&a.gbar[2]);
    else if (CL && warp > 0) arn_cluster_arrive();
    // the exponent of column j + 1 (one warp; the slots are written again only after this block's
    // next arrival)
    if constexpr (sizeof(TV) == 8) {
      if (warp == kArnWarps - 1) {
        const int e = arn_get_max(ctl, G);
        if (lane == 0) sE[k] = e;
        if (lane == 0 && bid == 0) ctl.vexp[k] = e;
      }
    }
    if (k < a.jmax && (!split0 || warp > 0))
      arn_diag<ND, TV, TACC>(a, k, R0, R0 + a.RS < R1 ? R0 + a.RS : R1, Ws, Us,
                             split0 ? t - 32 : t, split0 ? kArnThreads - 32 : kArnThreads);
    if (!arn_wait<CL>(&a.gbar[2], cbase + (unsigned)G * (unsigned)k)) {
      arn_timeout(ctl);
      return;
    }
    // the rotations' outputs are visible to every block: the same decision everywhere
    if (t == 0) ssig[k] = __ldcg(&ctl.sigma[k]);
    const int done = __ldcg(&ctl.flags[F_CYCLE_DONE]);
    __syncthreads();
    if (done) break;
  }
}

template <typename TV, typename TACC, int ND, int MODE>
__global__ void __launch_bounds__(kArnThreads, 1)
    k_arnoldi(const __grid_constant__ ArnArgs<TV, TACC> a) {
  arn_cycle<TV, TACC, ND, MODE, false>(a, (int)gridDim.x, (int)blockIdx.x);
}

// The cycles of many systems, a cluster of G blocks each: cluster c runs the c-th system of the list
// (list[0] systems still running, then their positions in args) when that count is in (lo, hi];
// deflation as the system's flag says
template <typename TV, typename TACC, int ND, int MODE>
__global__ void __launch_bounds__(kArnThreads, 1)
    k_arnoldi_batch(const ArnArgs<TV, TACC>* __restrict__ args, const int* __restrict__ list, int lo,
                    int hi, int G) {
  __shared__ ArnArgs<TV, TACC> a;
  const int n = __ldg(list), c = (int)blockIdx.x / G;
  if (n <= lo || n > hi || c >= n) return;  // the whole cluster
  const int* src = reinterpret_cast<const int*>(args + __ldg(list + 1 + c));
  for (int q = threadIdx.x; q < (int)(sizeof(a) / 4); q += kArnThreads)
    reinterpret_cast<int*>(&a)[q] = __ldg(src + q);
  __syncthreads();
  const int on = __ldcg(&a.ctl.flags[F_DEFL_ON]);
  __syncthreads();
  if (threadIdx.x == 0) a.defl = a.defl && on;
  __syncthreads();
  arn_cycle<TV, TACC, ND, MODE, true>(a, G, (int)(blockIdx.x % G));
}

// rows of a super-tile: w and u_j slices, s' and the reduction scratch in kArnSmem
inline long long arn_super_rows(int r, size_t esz) {
  const size_t fixed = ((size_t)r * esz + 127) / 128 * 128 + kArnScratch +
                       sizeof(double) * kMaxK * kMaxK + 256;
  if (fixed >= kArnSmem) return 0;
  return (long long)((kArnSmem - fixed) / (2 * esz)) / kArnUnit * kArnUnit;
}

template <typename TV, typename TACC>
struct Arn {
  using Args = ArnArgs<TV, TACC>;
  // many systems, a cluster of G blocks each (args, list: device arrays)
  template <int ND, int MODE>
  static cudaError_t batch_nd(const FusedBatch& f, int clusters, int lo, int hi, int G,
                              cudaStream_t st) {
    auto* kern = k_arnoldi_batch<TV, TACC, ND, MODE>;
    static cudaError_t prep = [&] {
      cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)kArnSmem);
      return e == cudaSuccess
                 ? cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)
                 : e;
    }();
    if (prep != cudaSuccess) return prep;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(clusters * G));
    cfg.blockDim = dim3((unsigned)kArnThreads);
    cfg.dynamicSmemBytes = kArnSmem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)G;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (clusters == 0) {  // query: the clusters of G blocks that fit the device at once
      cfg.gridDim = dim3((unsigned)G);
      int n = 0;
      const cudaError_t e = cudaOccupancyMaxActiveClusters(&n, kern, &cfg);
      if (e != cudaSuccess) {
        (void)cudaGetLastError();
        n = 0;
      }
      *f.fit = n;
      return cudaSuccess;
    }
    return cudaLaunchKernelEx(&cfg, kern, static_cast<const Args*>(f.args), f.list, lo, hi, G);
  }
  static cudaError_t batch(const FusedBatch& f, int clusters, int lo, int hi, int G,
                           cudaStream_t st) {
    if (f.ortho == GMRES_ORTHO_CGS2) return batch_op<kArnCgs2>(f, clusters, lo, hi, G, st);
    if constexpr (sizeof(TV) == sizeof(TACC))
      return batch_op<kArnLowsync>(f, clusters, lo, hi, G, st);
    else
      return cudaErrorInvalidValue;
  }
  template <int MODE>
  static cudaError_t batch_op(const FusedBatch& f, int clusters, int lo, int hi, int G,
                              cudaStream_t st) {
    return f.nd == 9  ? batch_nd<9, MODE>(f, clusters, lo, hi, G, st)
           : f.nd > 0 ? batch_nd<0, MODE>(f, clusters, lo, hi, G, st)
                      : batch_nd<kArnCsr, MODE>(f, clusters, lo, hi, G, st);
  }
  template <int ND, int MODE>
  static cudaError_t prepare() {
    return cudaFuncSetAttribute(k_arnoldi<TV, TACC, ND, MODE>,
                                cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kArnSmem);
  }
  template <int ND, int MODE>
  static cudaError_t launch_nd(const CycleArgs& c, const ArnArgs<TV, TACC>& p, cudaStream_t st) {
    static cudaError_t prep = prepare<ND, MODE>();
    if (prep != cudaSuccess) return prep;
    const int grid = p.units < c.sms ? p.units : c.sms;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)grid);
    cfg.blockDim = dim3((unsigned)kArnThreads);
    cfg.dynamicSmemBytes = kArnSmem;
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    // a cooperative launch with programmatic serialisation; should the runtime refuse the
    // pair, the kernel runs cooperatively in plain stream order from then on (same result)
    static bool pdl_ok = true;
    cfg.numAttrs = (c.pdl && pdl_ok) ? 2 : 1;
    cudaError_t e = cudaLaunchKernelEx(&cfg, k_arnoldi<TV, TACC, ND, MODE>, p);
    if (e != cudaSuccess && cfg.numAttrs == 2) {
      (void)cudaGetLastError();
      pdl_ok = false;
      cfg.numAttrs = 1;
      e = cudaLaunchKernelEx(&cfg, k_arnoldi<TV, TACC, ND, MODE>, p);
    }
    return e;
  }
  static Args fill(const CycleArgs& c, int jmax, bool defl) {
    Args p{};
    p.N = c.op.n;
    p.units = (int)(c.ldv / kArnUnit);
    p.fine = p.units < c.sms ? p.units : c.sms;
    p.jmax = jmax;
    p.m = c.m;
    p.pre = (defl && c.pdl) ? 1 : 0;
    p.defl = defl ? 1 : 0;
    p.r = defl ? c.op.defl.r : 0;
    p.RS = (int)arn_super_rows(p.r, sizeof(TACC));
    p.ldv = c.ldv;
    p.ldd = c.op.ldd;
    p.V = static_cast<const TV*>(c.V);
    p.w = static_cast<TACC*>(c.w);
    p.dia = c.op.dia;
    if constexpr (sizeof(TACC) == 8) {
      p.dval = c.op.dval;
      p.auval = c.op.defl.auval;
      p.aup_val = c.op.defl.aup_val;
      p.sdefl = c.ctl.sdefl;
    } else {
      p.dval = c.op.dval32;
      p.auval = c.op.defl.auval32;
      p.aup_val = c.op.defl.aup_val32;
      p.sdefl = c.ctl.sdefl32;
    }
    p.aurp = c.op.defl.aurp;
    p.aup_col = c.op.defl.aup_col;
    p.aucol = c.op.defl.aucol;
    p.perm = c.op.defl.perm;
    p.piece_start = c.op.defl.piece_start;
    p.agg_piece = c.op.defl.agg_piece;
    p.blk_piece_start = c.op.defl.blk_piece_start;
    p.blk_piece = c.op.defl.blk_piece;
    p.uscale = c.op.defl.uscale;
    p.tinv = c.op.defl.tinv;
    p.tinv32 = c.op.defl.tinv32;
    p.ctl = c.ctl;
    p.gbar = c.gbar;
    p.rowptr = c.op.rowptr;
    p.col = c.op.col;
    p.vec = c.op.vec;
    if constexpr (sizeof(TACC) == 8) p.val = c.op.val;
    else p.val = c.op.val32;
    return p;
  }
  static cudaError_t launch(const CycleArgs& c, int jmax, bool defl, cudaStream_t st) {
    const Args p = fill(c, jmax, defl);
    if (p.RS < kArnUnit) return cudaErrorInvalidValue;  // arnoldi_fusable rules this out
    if (c.ortho == GMRES_ORTHO_CGS2) return launch_op<kArnCgs2>(c, p, st);
    if constexpr (sizeof(TV) == 8) {
      // (a CSR operator takes the fixed-point multi-dot whatever dot_arith says)
      if (c.dot_arith == GMRES_DOT_DF32 && c.op.dia.nd > 0)
        return c.op.dia.nd == 9 ? launch_nd<9, kArnLowsyncDf>(c, p, st)
                                : launch_nd<0, kArnLowsyncDf>(c, p, st);
    }
    if constexpr (sizeof(TV) == sizeof(TACC)) return launch_op<kArnLowsync>(c, p, st);
    else return cudaErrorInvalidValue;
  }
  // the 9-point stencils of the Q1 systems take an unrolled instantiation
  template <int MODE>
  static cudaError_t launch_op(const CycleArgs& c, const ArnArgs<TV, TACC>& p, cudaStream_t st) {
    return c.op.dia.nd == 9  ? launch_nd<9, MODE>(c, p, st)
           : c.op.dia.nd > 0 ? launch_nd<0, MODE>(c, p, st)
                             : launch_nd<kArnCsr, MODE>(c, p, st);
  }
};

}  // namespace

}  // namespace gg
