// Shared pieces of the conjugate-gradient kernels (solve.cu, team.cu): FP64-
// grade dot products of FP32 vectors, block sums, the CG scalars, the
// iteration's record and the solve's starting point.
#pragma once

#include <cuda_runtime.h>

#include "common.cuh"

namespace casim {

// ---- FP64-grade dot products
// The CG dot products are accumulated to FP64 accuracy.  FP64 arithmetic is
// slow on this part (a dependent FP64 add takes about 64 cycles and an SM
// retires about two FP64 lanes per cycle, against 4.5 cycles and 128 lanes for
// FP32), so for FP32 vectors the per-row products and the in-block trees use
// double-word (float-float) arithmetic built from error-free transformations
// on the FP32 pipes:
//   TwoProd by FMA (the rounding error of a*b is fma(a, b, -a*b)),
//   TwoSum (Knuth) and Fast2Sum (Dekker),
//   the compensated dot product Dot2 of Ogita, Rump and Oishi (2005), kept
//   unrounded as a double word,
//   the double-word addition of Joldes, Muller and Popescu (2017) in its
//   11-operation form (below), relative error a few u^2 (u = 2^-24).
// Every operation is an explicitly rounded intrinsic, so the compiler can
// neither contract nor reassociate them.  Block partials are summed in block
// order (FP64 in the barrier kernels, double words in the team solver).
struct DW {
  float hi, lo;
};

__device__ __forceinline__ void two_sum_f(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  const float bb = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb));
}

// requires a == 0 or exponent(a) >= exponent(b)
__device__ __forceinline__ void fast_two_sum_f(float a, float b, float& s, float& e) {
  s = __fadd_rn(a, b);
  e = __fsub_rn(b, __fsub_rn(s, a));
}

// Sloppy double-word addition (Joldes, Muller, Popescu 2017, Algorithm 5):
// 11 operations; for operands of the same sign the relative error is at most
// 3u^2, otherwise the error is at most about u^2 (|x| + |y|), the same kind of
// bound as an FP64 sum has.
__device__ __forceinline__ DW dw_add_sloppy(DW x, DW y) {
  float sh, sl;
  two_sum_f(x.hi, y.hi, sh, sl);
  const float v = __fadd_rn(x.lo, y.lo);
  const float w = __fadd_rn(sl, v);
  DW z;
  fast_two_sum_f(sh, w, z.hi, z.lo);
  return z;
}

__device__ __forceinline__ DW dot3(float a0, float a1, float a2, float b0, float b1, float b2) {
  float p = __fmul_rn(a0, b0);
  float e = __fmaf_rn(a0, b0, -p);
  const float h1 = __fmul_rn(a1, b1), q1 = __fmaf_rn(a1, b1, -h1);
  const float h2 = __fmul_rn(a2, b2), q2 = __fmaf_rn(a2, b2, -h2);
  float s, t;
  two_sum_f(p, h1, s, t);
  p = s;
  e = __fadd_rn(e, __fadd_rn(q1, t));
  two_sum_f(p, h2, s, t);
  p = s;
  e = __fadd_rn(e, __fadd_rn(q2, t));
  DW z;
  two_sum_f(p, e, z.hi, z.lo);
  return z;
}

// Double-word product: the exact product of the high parts by TwoProd (FMA),
// the cross terms added in FP32, renormalised by Fast2Sum (relative error a
// few u^2; the neglected lo * lo term is below u^2 of the result).
__device__ __forceinline__ DW dw_mul(DW a, DW b) {
  const float p = __fmul_rn(a.hi, b.hi);
  float e = __fmaf_rn(a.hi, b.hi, -p);
  e = __fmaf_rn(a.hi, b.lo, e);
  e = __fmaf_rn(a.lo, b.hi, e);
  DW z;
  fast_two_sum_f(p, e, z.hi, z.lo);
  return z;
}
__device__ __forceinline__ DW dw_neg(DW a) { return DW{-a.hi, -a.lo}; }
// s += x for an FP32 x: the high parts by TwoSum, its error into the low part
// (renormalised once at the end by dw_norm).
__device__ __forceinline__ void dw_acc(DW& s, float x) {
  float h, e;
  two_sum_f(s.hi, x, h, e);
  s.hi = h;
  s.lo = __fadd_rn(s.lo, e);
}
// s += a b, the product exact by TwoProd (FMA)
__device__ __forceinline__ void dw_acc_prod(DW& s, float a, float b) {
  const float p = __fmul_rn(a, b);
  const float pe = __fmaf_rn(a, b, -p);
  float h, e;
  two_sum_f(s.hi, p, h, e);
  s.hi = h;
  s.lo = __fadd_rn(s.lo, __fadd_rn(e, pe));
}
__device__ __forceinline__ DW dw_norm(DW s) {
  DW z;
  fast_two_sum_f(s.hi, s.lo, z.hi, z.lo);
  return z;
}
// an FP64 value as a double word (hi = its FP32 rounding, lo = the rest rounded)
__device__ __forceinline__ DW dw_from(double x) {
  const float h = (float)x;
  return DW{h, (float)(x - (double)h)};
}


__device__ __forceinline__ double dot3(double a0, double a1, double a2, double b0, double b1, double b2) {
  return fma(a2, b2, fma(a1, b1, a0 * b0));
}

__device__ __forceinline__ DW acc_add(DW a, DW b) { return dw_add_sloppy(a, b); }
__device__ __forceinline__ double acc_add(double a, double b) { return a + b; }
__device__ __forceinline__ DW shfl_down(DW v, int o) {
  return DW{__shfl_down_sync(0xffffffffu, v.hi, o), __shfl_down_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ DW shfl_xor(DW v, int o) {
  return DW{__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ double shfl_down(double v, int o) { return __shfl_down_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double acc_to_f64(DW a) { return (double)a.hi + (double)a.lo; }
__device__ __forceinline__ double acc_to_f64(double a) { return a; }

template <typename A>
__device__ __forceinline__ A acc_zero();
template <>
__device__ __forceinline__ DW acc_zero<DW>() { return DW{0.0f, 0.0f}; }
template <>
__device__ __forceinline__ double acc_zero<double>() { return 0.0; }


// Block sums of NV per-thread values by fixed shuffle trees (within each warp,
// then over the NW warp sums, padded with zeros to a power of two); the FP64
// result is valid in lane 0 of warp 0.
// Contains one __syncthreads; sh holds at least 32 * NV doubles.
template <int NV, int NW, typename A>
__device__ __forceinline__ void block_sums(A (&v)[NV], double* sh, double (&bs)[NV]) {
  static_assert(sizeof(A) == sizeof(double), "accumulator must fit a double slot");
  static_assert(NW >= 1 && NW <= 32, "at most 32 warps per block");
  constexpr int NW2 = NW <= 1 ? 1 : NW <= 2 ? 2 : NW <= 4 ? 4 : NW <= 8 ? 8 : NW <= 16 ? 16 : 32;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  A* sa = reinterpret_cast<A*>(sh);
#pragma unroll
  for (int k = 0; k < NV; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[k] = acc_add(v[k], shfl_down(v[k], o));
  }
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) sa[k * 32 + wid] = v[k];
  }
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      A t = lane < NW ? sa[k * 32 + lane] : acc_zero<A>();
#pragma unroll
      for (int o = NW2 >> 1; o > 0; o >>= 1) t = acc_add(t, shfl_down(t, o));
      bs[k] = acc_to_f64(t);
    }
  }
}

// Warp sums of NV <= 4 double words by one butterfly that halves the values
// each lane carries at every level (a warp reduce-scatter): lanes exchange
// the half they give up at distance 16, then 8 (NV > 2), and every lane then
// finishes its one value with the remaining levels.  The pairs added are
// those of a shuffle-down tree over distances 16, 8, 4, 2, 1 (the sloppy
// addition is commutative bit for bit: TwoSum's error term is exact), so each
// sum equals that tree's, with 6 instead of 15 exchanges for NV = 3.  Value k
// ends in lanes [k L, (k + 1) L), L = 32 / (NV rounded up to a power of two).
template <int NV>
__device__ __forceinline__ DW warp_sums_dw_rs(const DW (&v)[NV]) {
  static_assert(NV >= 1 && NV <= 4, "one to four values");
  const int lane = threadIdx.x & 31;
  if constexpr (NV == 1) {
    DW x = v[0];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) x = dw_add_sloppy(x, shfl_xor(x, o));
    return x;
  } else if constexpr (NV == 2) {
    const bool up = lane & 16;
    DW x = dw_add_sloppy(up ? v[1] : v[0], shfl_xor(up ? v[0] : v[1], 16));
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) x = dw_add_sloppy(x, shfl_xor(x, o));
    return x;
  } else {
    const DW z{0.0f, 0.0f};
    const DW a2 = v[2], a3 = NV > 3 ? v[NV > 3 ? 3 : 0] : z;
    const bool up = lane & 16;
    const DW k0 = dw_add_sloppy(up ? a2 : v[0], shfl_xor(up ? v[0] : a2, 16));
    const DW k1 = dw_add_sloppy(up ? a3 : v[1], shfl_xor(up ? v[1] : a3, 16));
    const bool up8 = lane & 8;
    DW x = dw_add_sloppy(up8 ? k1 : k0, shfl_xor(up8 ? k0 : k1, 8));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) x = dw_add_sloppy(x, shfl_xor(x, o));
    return x;
  }
}

// Block sums of NV per-thread double words by fixed trees of sloppy
// double-word additions (the warp butterfly above, then warp 0 over the
// warps' sums); the double-word result is valid in lane 0 of warp 0.
// Contains one __syncthreads; sh holds at least 32 * NV doubles.
template <int NV, int NW>
__device__ __forceinline__ void block_sums_dw(DW (&v)[NV], double* sh, DW (&bs)[NV]) {
  static_assert(NW >= 1 && NW <= 32, "at most 32 warps per block");
  constexpr int NW2 = NW <= 1 ? 1 : NW <= 2 ? 2 : NW <= 4 ? 4 : NW <= 8 ? 8 : NW <= 16 ? 16 : 32;
  constexpr int L = NV == 1 ? 32 : NV == 2 ? 16 : 8;  // lanes per value after the butterfly
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  DW* sa = reinterpret_cast<DW*>(sh);
  const DW x = warp_sums_dw_rs<NV>(v);
  if (lane % L == 0 && lane / L < NV) sa[(lane / L) * 32 + wid] = x;
  __syncthreads();
  if (wid == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      DW t = lane < NW ? sa[k * 32 + lane] : DW{0.0f, 0.0f};
#pragma unroll
      for (int o = NW2 >> 1; o > 0; o >>= 1) t = dw_add_sloppy(t, shfl_down(t, o));
      bs[k] = t;
    }
  }
}

// End of an outer iteration (one thread): the energy into this iteration's
// record, the iteration count, and the per-iteration words reset.
template <typename T>
__device__ __forceinline__ void finalize_iteration(const Dev<T>& d, double energy) {
  Ctrl* c = d.ctrl;
  IterRec* rec = d.hist + (c->iter % d.hist_cap);
  rec->energy = energy;
  if (!isfinite(energy) && d.stats) c->status |= ST_NONFINITE;
  c->iter += 1;
  for (int j = 0; j < 3; ++j) {
    c->box_lo[j] = 0x7FFFFFFFFFFFFFFFLL;
    c->box_hi[j] = (long long)0x8000000000000000ULL;
  }
  IterRec* nx = d.hist + (c->iter % d.hist_cap);
  nx->energy = 0.0;
  nx->pcg_rel_residual = 0.0;
  nx->n_self_pairs = 0;
  nx->n_obstacle_pairs = 0;
  nx->n_springs = 0;
  nx->pcg_iters = 0;
  nx->knot_sig = 0;
  nx->spring_sig = 0;
}

// per-thread accumulator of the CG dot products for vectors of type T
template <typename T>
struct DotAcc;
template <>
struct DotAcc<float> {
  using type = DW;
};
template <>
struct DotAcc<double> {
  using type = double;
};

// (CG_LOST: the team PCG's step length is not positive)
enum { CG_CONTINUE = 0, CG_DONE = 1, CG_NONFINITE = 2, CG_ABORT = 3, CG_LOST = 4 };

// CG scalars after the reduction of (gamma_k, delta_k, rr), by all of warp 0
// (inputs read from lane 0, outputs in every lane).
// alpha_k = gamma_k / (delta_k - beta_k gamma_k / alpha_{k-1}) with
// beta_k = gamma_k / gamma_{k-1}, rearranged with q = gamma_{k-1} alpha_{k-1}
// to alpha_k = gamma_k q / (delta_k q - gamma_k^2); lanes 0 and 1 form
// alpha_k's and beta_k's quotients in the same division, so one FP64
// division lies on the dependent path.
__device__ __forceinline__ int cg_scalars_warp(const double (&t)[3], double bb_l0, double tol2, double& gamma,
                                               double& alpha, double& beta, double& rr) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const double gnew = __shfl_sync(full, t[0], 0), delta = __shfl_sync(full, t[1], 0);
  const double bb = __shfl_sync(full, bb_l0, 0);
  const double g = __shfl_sync(full, gamma, 0), a = __shfl_sync(full, alpha, 0);
  rr = __shfl_sync(full, t[2], 0);
  gamma = g;
  alpha = a;
  if (!isfinite(gnew) || !isfinite(delta) || !isfinite(rr)) return CG_NONFINITE;
  if (rr <= tol2 * bb) return CG_DONE;
  const double q = g * a;
  const double num = lane == 1 ? gnew : gnew * q;
  const double den = lane == 1 ? g : delta * q - gnew * gnew;
  const double quo = num / den;
  beta = __shfl_sync(full, quo, 1);
  alpha = __shfl_sync(full, quo, 0);
  gamma = gnew;
  return CG_CONTINUE;
}

// shared state of one block of a PCG kernel
template <typename T>
struct CgShared {
  double sh[96];
  T ta, tb;
  int flag;
  int ok;
};

template <typename T>
__device__ __forceinline__ R4<T> ld_cg(const R4<T>* a);
template <>
__device__ __forceinline__ R4<float> ld_cg<float>(const R4<float>* a) {
  const float4 v = __ldcg(reinterpret_cast<const float4*>(a));
  return R4<float>{v.x, v.y, v.z, v.w};
}
template <>
__device__ __forceinline__ R4<double> ld_cg<double>(const R4<double>* a) {
  const double2 v0 = __ldcg(reinterpret_cast<const double2*>(a));
  const double2 v1 = __ldcg(reinterpret_cast<const double2*>(a) + 1);
  return R4<double>{v0.x, v0.y, v1.x, v1.y};
}

__device__ __forceinline__ void write_pcg_record(const Ctrl* c, IterRec* hist, int cap, Ctrl* cw, int it, double rr,
                                                 double bb) {
  IterRec* rec = hist + (c->iter % cap);
  rec->pcg_iters = it;
  cw->total_pcg += it;
  rec->pcg_rel_residual = bb > 0.0 ? sqrt(rr / bb) : 0.0;
}

// The solve's starting point for free row i: x_i, plus the last outer
// iteration's step x_i - x_(i-1) where one is kept (an outer iteration's
// solve in MIXED mode; null otherwise).  The local-global iteration
// approaches its fixed point along a slowly turning direction, so
// x_i + (x_i - x_(i-1)) is a closer guess for x_(i+1) than x_i: the solve
// still stops at the same relative residual, from a smaller first one.  The
// same rounded sums in every row that reads it.
template <typename T>
__device__ __forceinline__ R4<T> warm_start(const Dev<T>& d, int i, R4<T> xi) {
  if (d.xstep) {
    const R4<T> s = d.xstep[i];
    xi.x += s.x;
    xi.y += s.y;
    xi.z += s.z;
  }
  return xi;
}

}  // namespace casim
