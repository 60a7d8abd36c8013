// Local step (Sec. III-A, Eq. 6, Eq. 7), right-hand-side gather and the
// global step solve (Sec. III-B, Eq. 8) on the GPU.
//
// Global step: the normal equations of Eq. 8 are A X = b with
//   A = L_w + k diag(mask),  L_w = sum_e w_e S_e^T N S_e  (3/4 w on the
//   diagonal, -1/4 w per shared edge), b = sum_e w_e S_e^T P_e^T + k c - A_fx x_fixed,
// the three coordinate columns sharing A.  They are solved together by
// Jacobi-preconditioned conjugate gradients in the single-reduction form of
// Chronopoulos and Gear (1989), inside one persistent cooperative kernel.
// Per iteration the neighbours' preconditioned residual u must be visible to
// the SpMV and one grid reduction produces (r.u, w.u, r.r) to FP64 accuracy:
// the kernels of this file publish u with a grid barrier; the team solver
// (team.cu), which outer iterations use where it fits, with epoch-tagged
// words that readers wait for.
#include <cooperative_groups.h>

#include <algorithm>
#include <type_traits>

#include "cg.cuh"
#include "common.cuh"
#include "kernels.h"
#include "svd3.cuh"

namespace casim {

// ---------------------------------------------------------------- local step
template <typename T>
__device__ __forceinline__ T cbrt_t(T x);
template <>
__device__ __forceinline__ float cbrt_t<float>(float x) { return cbrtf(x); }
template <>
__device__ __forceinline__ double cbrt_t<double>(double x) { return cbrt(x); }

__device__ __forceinline__ double w_table(const double* knots, int n, double eps, int& seg) {
  // piecewise linear through (eps_i, w_i), clamped at both ends; seg = the
  // interval used (0 below the first knot, i + 1 for [eps_i, eps_i+1), n above)
  seg = 0;
  if (eps <= knots[0]) return knots[1];
  for (int i = 0; i + 1 < n; ++i) {
    const double x0 = knots[2 * i], x1 = knots[2 * i + 2];
    if (eps < x1) {
      const double y0 = knots[2 * i + 1], y1 = knots[2 * i + 3];
      seg = i + 1;
      return y0 + (eps - x0) * (y1 - y0) / (x1 - x0);
    }
  }
  seg = n;
  return knots[2 * n - 1];
}

// The same table in FP32 (knots rounded to FP32), for FP32 positions.
__device__ __forceinline__ float w_table_f(const float* knots, int n, float eps, int& seg) {
  seg = 0;
  if (eps <= knots[0]) return knots[1];
  for (int i = 0; i + 1 < n; ++i) {
    const float x0 = knots[2 * i], x1 = knots[2 * i + 2];
    if (eps < x1) {
      const float y0 = knots[2 * i + 1], y1 = knots[2 * i + 3];
      seg = i + 1;
      return y0 + (eps - x0) * (y1 - y0) / (x1 - x0);
    }
  }
  seg = n;
  return knots[2 * n - 1];
}

// One thread per tet.  For FP32 positions the strain, w(eps) and the energy
// statistic stay on the FP32 pipes (FP32 strain and table, energy in double
// words); FP64 positions use FP64 throughout.
template <typename T, int SWEEPS, int BS>
__global__ void __launch_bounds__(BS) k_local(Dev<T> d) {
  constexpr bool F32 = std::is_same<T, float>::value;
  __shared__ double shd[32];
  __shared__ float s_kn[F32 ? 128 : 1];  // the knot table in FP32 (at most 64 knots)
  if constexpr (F32) {
    for (int k = threadIdx.x; k < 2 * d.n_knots; k += BS) s_kn[k] = (float)d.knots[k];
    __syncthreads();
  }
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  double en = 0.0;
  DW en_w{0.0f, 0.0f};
  unsigned long long ksig = 0;
  if (e < d.n_t) {
    const int4 t = chk_idx4(d.ctrl, d.tet[e], d.n_v);
    const R4<T> x0 = d.X[t.x], x1 = d.X[t.y], x2 = d.X[t.z], x3 = d.X[t.w];
    // centered deformed shape X_c = V^d N, formed from differences to x0
    T Xc[3][4];
    {
      const T r1[3] = {x1.x - x0.x, x1.y - x0.y, x1.z - x0.z};
      const T r2[3] = {x2.x - x0.x, x2.y - x0.y, x2.z - x0.z};
      const T r3[3] = {x3.x - x0.x, x3.y - x0.y, x3.z - x0.z};
      for (int i = 0; i < 3; ++i) {
        const T m = (r1[i] + r2[i] + r3[i]) * T(0.25);
        Xc[i][0] = -m;
        Xc[i][1] = r1[i] - m;
        Xc[i][2] = r2[i] - m;
        Xc[i][3] = r3[i] - m;
      }
    }
    const R4<T> tx = d.Tc[3 * (size_t)e], ty = d.Tc[3 * (size_t)e + 1], tz = d.Tc[3 * (size_t)e + 2];
    const T Tm[3][4] = {{tx.x, tx.y, tx.z, tx.w}, {ty.x, ty.y, ty.z, ty.w}, {tz.x, tz.y, tz.z, tz.w}};
    T D[3][3];
    for (int i = 0; i < 3; ++i)
      for (int j = 0; j < 3; ++j)
        D[i][j] = Xc[i][0] * Tm[j][0] + Xc[i][1] * Tm[j][1] + Xc[i][2] * Tm[j][2] + Xc[i][3] * Tm[j][3];
    T R[3][3], tr;
    rotation_fit<T, SWEEPS>(D, R, tr);
    T RT[3][4];
    for (int i = 0; i < 3; ++i)
      for (int k = 0; k < 4; ++k) RT[i][k] = R[i][0] * Tm[0][k] + R[i][1] * Tm[1][k] + R[i][2] * Tm[2][k];
    const R4<T> info = d.tinfo[e];
    const T omega = info.x, vol0 = info.y, tt = info.z;
    const int g = (int)info.w;
    T P[3][4];
    if (g >= 0) {
      // chamber element: every target vertex is the rest vertex scaled by cbrt(alpha_g)
      const T s = d.cbrt_alpha[g];
      for (int i = 0; i < 3; ++i)
        for (int k = 0; k < 4; ++k) P[i][k] = s * RT[i][k];
    } else {
      // body element: blend with w = R_omega(eps), then volume scaling (Eq. 6, Eq. 7)
      T mis = T(0);
      for (int i = 0; i < 3; ++i)
        for (int k = 0; k < 4; ++k) {
          const T q = Xc[i][k] - RT[i][k];
          mis += q * q;
        }
      int seg;
      T w;
      if constexpr (F32) {
        w = w_table_f(s_kn, d.n_knots, sqrtf(mis / tt), seg);
      } else {
        w = w_table(d.knots, d.n_knots, sqrt(mis / tt), seg);
      }
      if (d.stats) ksig = sig_mix((unsigned)e, (unsigned)seg);
      T B[3][4];
      for (int i = 0; i < 3; ++i)
        for (int k = 0; k < 4; ++k) B[i][k] = (T(1) - w) * Xc[i][k] + w * RT[i][k];
      const T a0 = B[0][1] - B[0][0], a1 = B[1][1] - B[1][0], a2 = B[2][1] - B[2][0];
      const T b0 = B[0][2] - B[0][0], b1 = B[1][2] - B[1][0], b2 = B[2][2] - B[2][0];
      const T c0 = B[0][3] - B[0][0], c1 = B[1][3] - B[1][0], c2 = B[2][3] - B[2][0];
      const T volB = (a0 * (b1 * c2 - b2 * c1) - a1 * (b0 * c2 - b2 * c0) + a2 * (b0 * c1 - b1 * c0)) / T(6);
      const T s = (volB > T(1e-3) * vol0) ? cbrt_t<T>(vol0 / volB) : T(1);
      for (int i = 0; i < 3; ++i)
        for (int k = 0; k < 4; ++k) P[i][k] = s * B[i][k];
    }
    if (d.stats) {
      if constexpr (F32) {
        // sum of (Xc - P)^2 with each difference exact as a double word
        DW acc{0.0f, 0.0f};
        for (int i = 0; i < 3; ++i)
          for (int k = 0; k < 4; ++k) {
            float qh, ql;
            two_sum_f(Xc[i][k], -P[i][k], qh, ql);
            dw_acc_prod(acc, qh, qh);
            acc.lo = __fmaf_rn(__fmul_rn(2.0f, qh), ql, acc.lo);
          }
        en_w = dw_mul(DW{omega, 0.0f}, dw_norm(acc));
      } else {
        double acc = 0.0;
        for (int i = 0; i < 3; ++i)
          for (int k = 0; k < 4; ++k) {
            const double q = (double)Xc[i][k] - (double)P[i][k];
            acc += q * q;
          }
        en = (double)omega * acc;
      }
    }
    R4<T>* out = d.P + 4 * (size_t)e;
    for (int k = 0; k < 4; ++k) {
      R4<T> c;
      c.x = omega * P[0][k];
      c.y = omega * P[1][k];
      c.z = omega * P[2][k];
      c.w = T(0);
      out[k] = c;
    }
  }
  if (d.stats) warp_add_u64(ksig, &(d.hist + (d.ctrl->iter % d.hist_cap))->knot_sig);
  if constexpr (F32) {
    DW v[1] = {en_w}, bs[1];
    block_sums_dw<1, BS / 32>(v, shd, bs);
    if (threadIdx.x == 0) d.e_partials[blockIdx.x] = acc_to_f64(bs[0]);
  } else {
    const double s = block_sum(en, shd);
    if (threadIdx.x == 0) d.e_partials[blockIdx.x] = s;
  }
}

// ------------------------------------------------------------ RHS gather
// b_v = sum over incident (e, slot) of w_e P_e[:, slot] + k mask_v c_v - bfix_v,
// accumulated in FP64 (the products of the FP32 targets need no rounding).
// The rows also carry the spring energy k mask_v |x_v - c_v|^2 (Eq. 5) of
// this iteration's springs (positions are unchanged since the spring update),
// summed per block in row order.
// One row of the right-hand side and of the diagonal: b_i, A_ii and the row's
// spring energy (see above).
template <typename T>
__device__ __forceinline__ void rhs_row(const Dev<T>& d, int i, R4<double>& b, T& diag, double& es) {
  double bx = 0.0, by = 0.0, bz = 0.0;
  const int k1 = d.inc_ptr[i + 1];
  for (int k = d.inc_ptr[i]; k < k1; ++k) {
    const R4<T> p = d.P[chk_idx(d.ctrl, d.inc[k], 4 * d.n_t)];
    bx += (double)p.x;
    by += (double)p.y;
    bz += (double)p.z;
  }
  const R4<double> sc = d.spring_c[i];
  const double km = d.k_spring * sc.w;
  const R4<double> bf = d.bfix[i];
  b = R4<double>{bx + km * sc.x - bf.x, by + km * sc.y - bf.y, bz + km * sc.z - bf.z, 0.0};
  diag = d.diagL[i] + (T)km;
  es = 0.0;
  if (sc.w != 0.0) {
    const R4<T> xi = d.X[i];
    const double ex = (double)xi.x - sc.x, ey = (double)xi.y - sc.y, ez = (double)xi.z - sc.z;
    es = km * (ex * ex + ey * ey + ez * ez);
  }
}

// The same row for FP32 positions with the FP32 terms added as double words
// (TwoSum) and the FP64 spring and fixed-vertex terms only on the rows that
// have them; the spring energy as a double word.
__device__ __forceinline__ void rhs_row_dw(const Dev<float>& d, int i, R4<double>& b, float& diag, DW& es) {
  DW bx{0.0f, 0.0f}, by{0.0f, 0.0f}, bz{0.0f, 0.0f};
  const int k1 = d.inc_ptr[i + 1];
#pragma unroll 4
  for (int k = d.inc_ptr[i]; k < k1; ++k) {
    const R4<float> p = d.P[chk_idx(d.ctrl, d.inc[k], 4 * d.n_t)];
    dw_acc(bx, p.x);
    dw_acc(by, p.y);
    dw_acc(bz, p.z);
  }
  bx = dw_norm(bx);
  by = dw_norm(by);
  bz = dw_norm(bz);
  b = R4<double>{(double)bx.hi + (double)bx.lo, (double)by.hi + (double)by.lo, (double)bz.hi + (double)bz.lo, 0.0};
  const R4<double> sc = d.spring_c[i];
  const double km = d.k_spring * sc.w;
  const R4<double> bf = d.bfix[i];
  diag = d.diagL[i] + (float)km;
  es = DW{0.0f, 0.0f};
  if (km != 0.0) {
    b.x += km * sc.x;
    b.y += km * sc.y;
    b.z += km * sc.z;
    const R4<float> xi = d.X[i];
    const double ex = (double)xi.x - sc.x, ey = (double)xi.y - sc.y, ez = (double)xi.z - sc.z;
    es = dw_from(km * (ex * ex + ey * ey + ez * ez));
  }
  if (bf.x != 0.0 || bf.y != 0.0 || bf.z != 0.0) {
    b.x -= bf.x;
    b.y -= bf.y;
    b.z -= bf.z;
  }
}

template <typename T, int BS>
__global__ void __launch_bounds__(BS) k_rhs(Dev<T> d) {
  __shared__ double shd[32];
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if constexpr (std::is_same<T, float>::value) {
    DW es[1] = {{0.0f, 0.0f}}, bs[1];
    if (i < d.n_free) {
      R4<double> b;
      float dg;
      rhs_row_dw(d, i, b, dg, es[0]);
      d.b[i] = b;
      d.diag[i] = dg;
    }
    block_sums_dw<1, BS / 32>(es, shd, bs);
    if (threadIdx.x == 0) d.e_partials[d.n_e_local + blockIdx.x] = acc_to_f64(bs[0]);
  } else {
    double es = 0.0;
    if (i < d.n_free) {
      R4<double> b;
      T dg;
      rhs_row(d, i, b, dg, es);
      d.b[i] = b;
      d.diag[i] = dg;
    }
    const double s = block_sum(es, shd);
    if (threadIdx.x == 0) d.e_partials[d.n_e_local + blockIdx.x] = s;
  }
}

// ------------------------------------------------------------------ PCG
//
// The PCG kernels solve for the correction d of the warm start x:
//   r0 = b - A x  in FP64 (FP32 products are exact in FP64),
//   A d = r0      by Jacobi-preconditioned CG in the working precision,
//   x <- x + d    once at the end,
// so that the rounding of the working precision applies to the small
// correction, not to the positions (one step of mixed-precision iterative
// refinement per outer iteration).  The stopping test ||r|| <= tol ||b|| is the
// same as for the plain system.
//
// Per CG iteration there are two grid barriers: one publishes the new
// preconditioned residual u for the neighbours' SpMV, one completes the
// reduction of (r.u, w.u, r.r).
//
// Grid barrier: one arrival counter whose top bit flips once per round.
// Block 0 adds 0x80000000 - (nblocks - 1) and every other block adds 1, so a
// full round adds exactly 0x80000000: the low bits return to their value and
// the top bit changes, which every block waits for (no reset, one atomic per
// block).  Every wait is bounded by a clock budget, after which the kernel
// records ST_TIMEOUT, raises the abort word and returns.
//
// Reductions: each block forms its sums (below), lane 0 of warp 0 stores them
// as the block's partials and arrives; after the barrier warp 0 alone adds the
// partials in block order (deterministic), computes the CG scalars once for
// the block and hands them to the other warps through shared memory.  Partials
// are stored value-major, partials[(parity * 4 + k) * nblocks + block], in two
// buffers chosen by the barrier count's parity.
struct GridCtx {
  Ctrl* ctrl;
  double* partials;
  unsigned nblocks;
  unsigned long long budget;
  unsigned extra;  // test-only: arrivals expected beyond the grid (never come)
};

// One thread of the block arrives and waits for the round to complete.
// Returns 0 when the wait gave up (timeout) or another block aborted.
__device__ __forceinline__ int arrive_and_wait(const GridCtx& g) {
  const unsigned add = blockIdx.x == 0 ? (0x80000000u - (g.nblocks - 1u + g.extra)) : 1u;
  __threadfence();
  const unsigned old = atomicAdd(&g.ctrl->bar_count, add);
  volatile unsigned* vc = &g.ctrl->bar_count;
  int ok = 1;
  if (((old ^ *vc) & 0x80000000u) == 0) {
    const long long t0 = clock64();
    unsigned spins = 0;
    while (((old ^ *vc) & 0x80000000u) == 0) {
      if ((++spins & 63u) == 0) {
        if (*(volatile int*)&g.ctrl->abort) {
          ok = 0;
          break;
        }
        if ((unsigned long long)(clock64() - t0) > g.budget) {
          atomicExch(&g.ctrl->abort, 1);
          atomicOr(&g.ctrl->status, ST_TIMEOUT);
          ok = 0;
          break;
        }
      }
    }
  }
  __threadfence();
  return ok;
}

// Plain grid barrier (makes every block's prior global writes visible).
__device__ __forceinline__ bool grid_barrier(const GridCtx& g, unsigned& epoch, int* shf) {
  ++epoch;
  __syncthreads();
  if (threadIdx.x == 0) *shf = arrive_and_wait(g);
  __syncthreads();
  return *shf != 0;
}

// Called by all of warp 0 after block_sums.  Lane 0 stores the block's sums
// as its partials, arrives and waits; the warp then adds the partials of
// blocks [b0, b1) in block order: each lane its blocks in increasing order,
// then a fixed shuffle tree.  tot is valid in lane 0.  Returns false
// (warp-uniform) when the wait gave up or another block aborted.
template <int NV>
__device__ __forceinline__ bool warp0_reduce(const GridCtx& g, unsigned& epoch, const double (&bs)[NV], int b0,
                                             int b1, double (&tot)[NV]) {
  ++epoch;
  const int lane = threadIdx.x & 31;
  const size_t nb = g.nblocks;
  const double* buf = g.partials + (size_t)(epoch & 1u) * 4 * nb;
  int ok = 1;
  if (lane == 0) {
    double* wb = g.partials + (size_t)(epoch & 1u) * 4 * nb;
#pragma unroll
    for (int k = 0; k < NV; ++k) wb[k * nb + blockIdx.x] = bs[k];
    ok = arrive_and_wait(g);
  }
  __syncwarp();
  ok = __shfl_sync(0xffffffffu, ok, 0);
  if (!ok) return false;
  double a[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) a[k] = 0.0;
#pragma unroll 2
  for (int b = b0 + lane; b < b1; b += 32) {
#pragma unroll
    for (int k = 0; k < NV; ++k) a[k] += __ldcg(buf + k * nb + b);
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a[k] += __shfl_down_sync(0xffffffffu, a[k], o);
    tot[k] = a[k];
  }
  return true;
}

// r_i = b_i - (A x)_i in FP64, x the solve's starting point, and ||b_i||^2,
// ||r_i||^2 (the first residual of the correction form; X is read-only while
// it is formed).
template <typename T>
__device__ __forceinline__ void residual_row_f64(const Dev<T>& d, int i, T dg, double (&rv)[3], double (&a0)[2],
                                                 const R4<double>* b_in = nullptr) {
  const R4<T> xi = warm_start(d, i, d.X[i]);
  double ax = (double)dg * xi.x, ay = (double)dg * xi.y, az = (double)dg * xi.z;
  const int sl = i >> 5, lane = i & 31;
  const int k1 = d.sl_ptr[sl + 1];
  for (int k = d.sl_ptr[sl] + lane; k < k1; k += 32) {
    const double a = (double)d.sl_val[k];
    const int col = chk_idx(d.ctrl, d.sl_col[k], d.n_free);
    const R4<T> xc = warm_start(d, col, d.X[col]);
    ax += a * xc.x;
    ay += a * xc.y;
    az += a * xc.z;
  }
  const R4<double> bi = b_in ? *b_in : d.b[i];
  rv[0] = bi.x - ax;
  rv[1] = bi.y - ay;
  rv[2] = bi.z - az;
  a0[0] += bi.x * bi.x + bi.y * bi.y + bi.z * bi.z;
  a0[1] += rv[0] * rv[0] + rv[1] * rv[1] + rv[2] * rv[2];
}

// Streaming variant: any number of rows per thread (grid-stride); vectors in
// HBM/L2, off-diagonals read from the sliced-ELL arrays every SpMV.
template <typename T>
__device__ __forceinline__ void spmv_row(const Dev<T>& d, int i, const R4<T>* __restrict__ src, T dg,
                                         const R4<T>& self, T& ax, T& ay, T& az) {
  ax = dg * self.x;
  ay = dg * self.y;
  az = dg * self.z;
  const int s = i >> 5, lane = i & 31;
  const int k1 = d.sl_ptr[s + 1];
  for (int k = d.sl_ptr[s] + lane; k < k1; k += 32) {
    const int c = chk_idx(d.ctrl, d.sl_col[k], d.n_v);
    const T a = d.sl_val[k];
    const R4<T> x = ld_cg<T>(src + c);
    ax += a * x.x;
    ay += a * x.y;
    az += a * x.z;
  }
}

template <typename T>
__global__ void __launch_bounds__(PCG_THREADS, 1) k_pcg(Dev<T> d) {
  using A = typename DotAcc<T>::type;
  constexpr int NW = PCG_THREADS / 32;
  __shared__ CgShared<T> cs;
  const GridCtx g{d.ctrl, d.partials, gridDim.x, d.wait_budget, d.bar_extra};
  unsigned epoch = 0;
  const int lane = threadIdx.x & 31;
  const bool w0 = threadIdx.x < 32;
  const int n = d.n_free;
  const int G = gridDim.x * blockDim.x;
  const int tid = blockIdx.x * blockDim.x + threadIdx.x;
  R4<T>* __restrict__ X = d.X;
  R4<T>* __restrict__ r = d.r;
  R4<T>* __restrict__ u = d.u;
  R4<T>* __restrict__ p = d.p;
  R4<T>* __restrict__ s = d.s;
  R4<T>* __restrict__ w = d.w;
  R4<T>* __restrict__ dx = d.dx;
  const R4<T> zero = {T(0), T(0), T(0), T(0)};
  // CG scalars: meaningful in lane 0 of warp 0
  double bb = 0.0, rr = 0.0, gamma = 0.0, alpha = 0.0, beta = 0.0;

  // r = b - A x in FP64, u = M^-1 r, d = 0
  double a0[2] = {0.0, 0.0};
  for (int i = tid; i < n; i += G) {
    const T dg = d.diag[i];
    double rv[3];
    residual_row_f64(d, i, dg, rv, a0);
    R4<T> ri, ui;
    ri.x = (T)rv[0]; ri.y = (T)rv[1]; ri.z = (T)rv[2]; ri.w = T(0);
    ui.x = ri.x / dg; ui.y = ri.y / dg; ui.z = ri.z / dg; ui.w = T(0);
    r[i] = ri;
    u[i] = ui;
    dx[i] = zero;
  }
  {
    double bs[2], t[2];
    block_sums<2, NW>(a0, cs.sh, bs);
    if (w0) {
      const bool ok = warp0_reduce<2>(g, epoch, bs, 0, gridDim.x, t);
      if (lane == 0) {
        bb = t[0];
        rr = t[1];
        cs.flag = !ok ? CG_ABORT : ((bb > 0.0 && rr > d.tol2 * bb) ? CG_CONTINUE : CG_DONE);
      }
    }
    __syncthreads();
  }
  if (cs.flag == CG_ABORT) return;
  int it = 0;
  if (cs.flag == CG_CONTINUE) {
    A a1[2] = {acc_zero<A>(), acc_zero<A>()};
    for (int i = tid; i < n; i += G) {
      const T dg = d.diag[i];
      const R4<T> ui = u[i], ri = r[i];
      T ax, ay, az;
      spmv_row(d, i, u, dg, ui, ax, ay, az);
      R4<T> wi;
      wi.x = ax; wi.y = ay; wi.z = az; wi.w = T(0);
      w[i] = wi;
      a1[0] = acc_add(a1[0], dot3(ri.x, ri.y, ri.z, ui.x, ui.y, ui.z));
      a1[1] = acc_add(a1[1], dot3(ax, ay, az, ui.x, ui.y, ui.z));
    }
    {
      double bs[2], t[2];
      block_sums<2, NW>(a1, cs.sh, bs);
      if (w0) {
        const bool ok = warp0_reduce<2>(g, epoch, bs, 0, gridDim.x, t);
        if (lane == 0) {
          if (ok) {
            gamma = t[0];
            alpha = gamma / t[1];
            cs.ta = (T)alpha;
            cs.tb = T(0);
          }
          cs.flag = ok ? CG_CONTINUE : CG_ABORT;
        }
      }
      __syncthreads();
    }
    if (cs.flag == CG_ABORT) return;
    T ta = cs.ta, tb = T(0);
    bool first = true;
    for (it = 1; it <= d.max_iter; ++it) {
      for (int i = tid; i < n; i += G) {
        const R4<T> ui = u[i], wi = w[i];
        R4<T> pi, si;
        if (first) {
          pi = ui;
          si = wi;
        } else {
          const R4<T> po = p[i], so = s[i];
          pi.x = ui.x + tb * po.x; pi.y = ui.y + tb * po.y; pi.z = ui.z + tb * po.z;
          si.x = wi.x + tb * so.x; si.y = wi.y + tb * so.y; si.z = wi.z + tb * so.z;
        }
        pi.w = T(0);
        si.w = T(0);
        p[i] = pi;
        s[i] = si;
        R4<T> di = dx[i], ri = r[i];
        di.x += ta * pi.x; di.y += ta * pi.y; di.z += ta * pi.z;
        ri.x -= ta * si.x; ri.y -= ta * si.y; ri.z -= ta * si.z;
        dx[i] = di;
        r[i] = ri;
        const T dg = d.diag[i];
        R4<T> un;
        un.x = ri.x / dg; un.y = ri.y / dg; un.z = ri.z / dg; un.w = T(0);
        u[i] = un;
      }
      if (!grid_barrier(g, epoch, &cs.ok)) return;
      A a2[3] = {acc_zero<A>(), acc_zero<A>(), acc_zero<A>()};
      for (int i = tid; i < n; i += G) {
        const T dg = d.diag[i];
        const R4<T> ui = u[i], ri = r[i];
        T ax, ay, az;
        spmv_row(d, i, u, dg, ui, ax, ay, az);
        R4<T> wi;
        wi.x = ax; wi.y = ay; wi.z = az; wi.w = T(0);
        w[i] = wi;
        a2[0] = acc_add(a2[0], dot3(ri.x, ri.y, ri.z, ui.x, ui.y, ui.z));
        a2[1] = acc_add(a2[1], dot3(ax, ay, az, ui.x, ui.y, ui.z));
        a2[2] = acc_add(a2[2], dot3(ri.x, ri.y, ri.z, ri.x, ri.y, ri.z));
      }
      {
        double bs[3], t[3];
        block_sums<3, NW>(a2, cs.sh, bs);
        if (w0) {
          const bool ok = warp0_reduce<3>(g, epoch, bs, 0, gridDim.x, t);
          int f = CG_ABORT;
          if (ok) f = cg_scalars_warp(t, bb, d.tol2, gamma, alpha, beta, rr);
          if (lane == 0) {
            if (ok) {
              if (f == CG_NONFINITE && blockIdx.x == 0) set_status(d.ctrl, ST_NONFINITE);
              cs.ta = (T)alpha;
              cs.tb = (T)beta;
            }
            cs.flag = f;
          }
        }
        __syncthreads();
      }
      const int f = cs.flag;
      if (f == CG_ABORT) return;
      if (f != CG_CONTINUE) break;
      ta = cs.ta;
      tb = cs.tb;
      first = false;
    }
    if (it > d.max_iter) {
      it = d.max_iter;
      if (tid == 0) set_status(d.ctrl, ST_PCG_MAXIT);
    }
    for (int i = tid; i < n; i += G) {
      R4<T> xi = X[i];
      const R4<T> di = dx[i];
      xi.x += di.x; xi.y += di.y; xi.z += di.z;
      X[i] = xi;
    }
  }
  if (tid == 0) write_pcg_record(d.ctrl, d.hist, d.hist_cap, d.ctrl, it, rr, bb);
}

// Register-resident variant: one row per thread.  The thread keeps its
// sliced-ELL row, diagonal and all CG vectors in registers for the whole
// solve; per iteration only the preconditioned residual u is written to
// memory and the neighbours' values are gathered from L2.
template <typename T, int MAXW>
__global__ void __launch_bounds__(PCG_RR_THREADS, 2) k_pcg_rr(Dev<T> d) {
  using A = typename DotAcc<T>::type;
  constexpr int NW = PCG_RR_THREADS / 32;
  __shared__ CgShared<T> cs;
  const GridCtx g{d.ctrl, d.partials, gridDim.x, d.wait_budget, d.bar_extra};
  unsigned epoch = 0;
  const int lane = threadIdx.x & 31;
  const bool w0 = threadIdx.x < 32;
  const int n = d.n_free;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = i < n;
  int col[MAXW];
  T val[MAXW];
  int width = 0;
  T dg = T(1);
  T x[3] = {T(0), T(0), T(0)};
  if (act) {
    const int sl = i >> 5, ln = i & 31;
    const int base = d.sl_ptr[sl];
    width = (d.sl_ptr[sl + 1] - base) >> 5;
#pragma unroll
    for (int j = 0; j < MAXW; ++j) {
      if (j < width) {
        col[j] = d.sl_col[base + j * 32 + ln];
        val[j] = d.sl_val[base + j * 32 + ln];
      } else {
        col[j] = i;
        val[j] = T(0);
      }
    }
    dg = d.diag[i];
    const R4<T> xi = d.X[i];
    x[0] = xi.x; x[1] = xi.y; x[2] = xi.z;
  }
  auto spmv = [&](const R4<T>* src, const T (&self)[3], T (&ax)[3]) {
    ax[0] = dg * self[0];
    ax[1] = dg * self[1];
    ax[2] = dg * self[2];
#pragma unroll
    for (int j = 0; j < MAXW; ++j) {
      if (j < width) {
        const R4<T> v = ld_cg<T>(src + col[j]);
        ax[0] += val[j] * v.x;
        ax[1] += val[j] * v.y;
        ax[2] += val[j] * v.z;
      }
    }
  };
  auto store_u = [&](const T (&uu)[3]) {
    R4<T> t;
    t.x = uu[0]; t.y = uu[1]; t.z = uu[2]; t.w = T(0);
    d.u[i] = t;
  };
  // CG scalars: meaningful in lane 0 of warp 0
  double bb = 0.0, rr = 0.0, gamma = 0.0, alpha = 0.0, beta = 0.0;
  T r[3], u[3], w[3], p[3], s[3], dd[3] = {T(0), T(0), T(0)};
  double a0[2] = {0.0, 0.0};
  if (act) {
    double rv[3];
    residual_row_f64(d, i, dg, rv, a0);
    for (int c = 0; c < 3; ++c) {
      r[c] = (T)rv[c];
      u[c] = r[c] / dg;
    }
    store_u(u);
  }
  {
    double bs[2], t[2];
    block_sums<2, NW>(a0, cs.sh, bs);
    if (w0) {
      const bool ok = warp0_reduce<2>(g, epoch, bs, 0, gridDim.x, t);
      if (lane == 0) {
        bb = t[0];
        rr = t[1];
        cs.flag = !ok ? CG_ABORT : ((bb > 0.0 && rr > d.tol2 * bb) ? CG_CONTINUE : CG_DONE);
      }
    }
    __syncthreads();
  }
  if (cs.flag == CG_ABORT) return;
  int it = 0;
  if (cs.flag == CG_CONTINUE) {
    A a1[2] = {acc_zero<A>(), acc_zero<A>()};
    if (act) {
      spmv(d.u, u, w);
      a1[0] = dot3(r[0], r[1], r[2], u[0], u[1], u[2]);
      a1[1] = dot3(w[0], w[1], w[2], u[0], u[1], u[2]);
      for (int c = 0; c < 3; ++c) {
        p[c] = u[c];
        s[c] = w[c];
      }
    }
    {
      double bs[2], t[2];
      block_sums<2, NW>(a1, cs.sh, bs);
      if (w0) {
        const bool ok = warp0_reduce<2>(g, epoch, bs, 0, gridDim.x, t);
        if (lane == 0) {
          if (ok) {
            gamma = t[0];
            alpha = gamma / t[1];
            cs.ta = (T)alpha;
          }
          cs.flag = ok ? CG_CONTINUE : CG_ABORT;
        }
      }
      __syncthreads();
    }
    if (cs.flag == CG_ABORT) return;
    T ta = cs.ta;
    for (it = 1; it <= d.max_iter; ++it) {
      if (act) {
        for (int c = 0; c < 3; ++c) {
          dd[c] += ta * p[c];
          r[c] -= ta * s[c];
          u[c] = r[c] / dg;
        }
        store_u(u);
      }
      if (!grid_barrier(g, epoch, &cs.ok)) return;
      A a2[3] = {acc_zero<A>(), acc_zero<A>(), acc_zero<A>()};
      if (act) {
        spmv(d.u, u, w);
        a2[0] = dot3(r[0], r[1], r[2], u[0], u[1], u[2]);
        a2[1] = dot3(w[0], w[1], w[2], u[0], u[1], u[2]);
        a2[2] = dot3(r[0], r[1], r[2], r[0], r[1], r[2]);
      }
      {
        double bs[3], t[3];
        block_sums<3, NW>(a2, cs.sh, bs);
        if (w0) {
          const bool ok = warp0_reduce<3>(g, epoch, bs, 0, gridDim.x, t);
          int f = CG_ABORT;
          if (ok) f = cg_scalars_warp(t, bb, d.tol2, gamma, alpha, beta, rr);
          if (lane == 0) {
            if (ok) {
              if (f == CG_NONFINITE && blockIdx.x == 0) set_status(d.ctrl, ST_NONFINITE);
              cs.ta = (T)alpha;
              cs.tb = (T)beta;
            }
            cs.flag = f;
          }
        }
        __syncthreads();
      }
      const int f = cs.flag;
      if (f == CG_ABORT) return;
      if (f != CG_CONTINUE) break;
      ta = cs.ta;
      const T tb = cs.tb;
      if (act)
        for (int c = 0; c < 3; ++c) {
          p[c] = u[c] + tb * p[c];
          s[c] = w[c] + tb * s[c];
        }
    }
    if (it > d.max_iter) {
      it = d.max_iter;
      if (i == 0) set_status(d.ctrl, ST_PCG_MAXIT);
    }
    if (act) {
      R4<T> t;
      t.x = x[0] + dd[0]; t.y = x[1] + dd[1]; t.z = x[2] + dd[2]; t.w = T(0);
      d.X[i] = t;
    }
  }
  if (i == 0) write_pcg_record(d.ctrl, d.hist, d.hist_cap, d.ctrl, it, rr, bb);
}

static constexpr int SEG_AGG_ROWS = 128;  // aggregate rows of the segmented batch kernel

// Segmented streaming variant for batches: block b works on a contiguous row
// range of one robot (every robot owns at least one block; blocks are given
// to robots in proportion to their rows), so each robot runs its own CG with
// its own scalars and stopping test while all robots share the two grid
// barriers of an iteration.  Robot totals are the sums of the partials of the
// robot's blocks in block order (deterministic).  A robot that has converged
// stops updating; the launch ends when every robot has converged (a counter
// that the robot's first block increments, read after the next barrier so
// every block sees the same value) or at the iteration cap.
// Per-robot coarse correction of the segmented kernel (COARSE): the same
// additive two-level preconditioner, per robot, over constants only, with
// aggregates of SEG_AGG_ROWS rows counted from the robot's first row and block
// boundaries on whole aggregates.  In a pass, round m of the block's threads
// covers the rows lo + 256 m + t, i.e. the block's local aggregates 2m (warps
// 0..3) and 2m + 1 (warps 4..7); each warp adds its rows' values by a fixed
// shuffle tree and the four warp sums of an aggregate are added in order.
static constexpr int SEG_WPA = SEG_AGG_ROWS / 32;  // warps per aggregate

template <int NV>
__device__ __forceinline__ void seg_agg_partial(const float (&v)[NV], int m, float (*zp)[PCG_SEG_THREADS / 32][6],
                                                int off) {
  float a[NV];
#pragma unroll
  for (int c = 0; c < NV; ++c) {
    a[c] = v[c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a[c] = __fadd_rn(a[c], __shfl_down_sync(0xffffffffu, a[c], o));
  }
  const int wid = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) {
    const int agg = 2 * m + wid / SEG_WPA;
    if (agg < PCG_SEG_AGG_MAX)
#pragma unroll
      for (int c = 0; c < NV; ++c) zp[agg][wid % SEG_WPA][off + c] = a[c];
  }
}

template <typename T, bool COARSE>
__global__ void __launch_bounds__(PCG_SEG_THREADS, 4) k_pcg_seg(Dev<T> d) {
  using A = typename DotAcc<T>::type;
  constexpr int NW = PCG_SEG_THREADS / 32;
  __shared__ CgShared<T> cs;
  // coarse state of the block's aggregates: warp partial sums of a pass,
  // fresh g(w) and g(r) of the last reduction, the carried g(s)
  __shared__ float s_zp[COARSE ? PCG_SEG_AGG_MAX : 1][PCG_SEG_THREADS / 32][6];
  __shared__ float s_gw[COARSE ? PCG_SEG_AGG_MAX : 1][3];
  __shared__ float s_gr[COARSE ? PCG_SEG_AGG_MAX : 1][3];
  __shared__ float s_gs[COARSE ? PCG_SEG_AGG_MAX : 1][3];
  const GridCtx g{d.ctrl, d.partials, gridDim.x, d.wait_budget, d.bar_extra};
  unsigned epoch = 0;
  const int lane = threadIdx.x & 31;
  const bool w0 = threadIdx.x < 32;
  const int b = blockIdx.x;
  const int lo = d.seg_lo[b], hi = d.seg_hi[b];
  const int rb0 = d.seg_rb0[b], rb1 = d.seg_rb1[b];
  const bool lead = b == rb0 && threadIdx.x == 0;  // the robot's first block, lane 0
  R4<T>* __restrict__ X = d.X;
  R4<T>* __restrict__ r = d.r;
  R4<T>* __restrict__ u = d.u;
  R4<T>* __restrict__ p = d.p;
  R4<T>* __restrict__ s = d.s;
  R4<T>* __restrict__ w = d.w;
  R4<T>* __restrict__ dx = d.dx;
  const R4<T> zero = {T(0), T(0), T(0), T(0)};
  // robot CG scalars: meaningful in lane 0 of warp 0
  double bb = 0.0, rr = 0.0, gamma = 0.0, alpha = 0.0, beta = 0.0;
  int it_done = 0;
  // coarse bookkeeping
  int rob = 0, r0 = 0, ga0 = 0, na_r = 0, na_b = 0;
  const float* ainv = nullptr;
  if constexpr (COARSE) {
    rob = d.seg_robot[b];
    r0 = d.robot_row[rob];
    na_r = d.seg_agg_base[rob + 1] - d.seg_agg_base[rob];
    ga0 = d.seg_agg_base[rob] + (lo - r0) / SEG_AGG_ROWS;
    na_b = (hi - lo + SEG_AGG_ROWS - 1) / SEG_AGG_ROWS;
    ainv = d.seg_ainv + d.seg_ainv_off[rob] + (size_t)((lo - r0) / SEG_AGG_ROWS) * na_r;
  }
  // the block's aggregate sums of this pass into the global exchange array
  // (call after a __syncthreads that follows the pass); which = 0 w, 1 r
  auto agg_store = [&](int which) {
    for (int k = threadIdx.x; k < na_b * 3; k += blockDim.x) {
      const int a = k / 3, c = k % 3;
      float t = s_zp[a][0][3 * which + c];
#pragma unroll
      for (int q = 1; q < SEG_WPA; ++q) t = __fadd_rn(t, s_zp[a][q][3 * which + c]);
      d.seg_aggsum[6 * (size_t)(ga0 + a) + 3 * which + c] = t;
    }
  };
  // g = A_c^-1 Z^T v for the block's aggregates from the robot's exchanged
  // sums (after the reduction made them visible): which = 0 w into s_gw, 1 r
  // into s_gr; one thread per (aggregate, column, which), robot-order sums
  auto agg_coarse = [&]() {
    const int base = d.seg_agg_base[rob];
    for (int k = threadIdx.x; k < na_b * 6; k += blockDim.x) {
      const int a = k / 6, which = (k % 6) / 3, c = k % 3;
      const float* row = ainv + (size_t)a * na_r;
      float t = 0.0f;
      for (int j = 0; j < na_r; ++j)
        t = __fmaf_rn(row[j], __ldcg(&d.seg_aggsum[6 * (size_t)(base + j) + 3 * which + c]), t);
      if (which == 0)
        s_gw[a][c] = t;
      else
        s_gr[a][c] = t;
    }
  };

  double a0[2] = {0.0, 0.0};
  for (int i = lo + (int)threadIdx.x, m = 0; i < hi || (COARSE && m * (int)blockDim.x < hi - lo);
       i += blockDim.x, ++m) {
    float rz[3] = {0.0f, 0.0f, 0.0f};
    if (i < hi) {
      const T dg = d.diag[i];
      double rv[3];
      residual_row_f64(d, i, dg, rv, a0);
      R4<T> ri, ui;
      ri.x = (T)rv[0]; ri.y = (T)rv[1]; ri.z = (T)rv[2]; ri.w = T(0);
      const T idg = T(1) / dg;
      ui.x = ri.x * idg; ui.y = ri.y * idg; ui.z = ri.z * idg; ui.w = T(0);
      r[i] = ri;
      u[i] = ui;
      dx[i] = zero;
      rz[0] = (float)ri.x; rz[1] = (float)ri.y; rz[2] = (float)ri.z;
    }
    if constexpr (COARSE) {
      const float wz[3] = {0.0f, 0.0f, 0.0f};
      seg_agg_partial<3>(wz, m, s_zp, 0);
      seg_agg_partial<3>(rz, m, s_zp, 3);
    }
  }
  if constexpr (COARSE) {
    __syncthreads();
    agg_store(0);
    agg_store(1);
  }
  {
    double bs[2], t[2];
    block_sums<2, NW>(a0, cs.sh, bs);
    if (w0) {
      const bool ok = warp0_reduce<2>(g, epoch, bs, rb0, rb1, t);
      if (lane == 0) {
        bb = t[0];
        rr = t[1];
        const bool conv = !(bb > 0.0 && rr > d.tol2 * bb);
        if (ok && conv && b == rb0) atomicAdd(&d.ctrl->queue, 1u);
        cs.flag = !ok ? CG_ABORT : (conv ? CG_DONE : CG_CONTINUE);
      }
    }
    __syncthreads();
  }
  if (cs.flag == CG_ABORT) return;
  bool done = cs.flag != CG_CONTINUE;
  if constexpr (COARSE) {
    // u_0 = D^-1 r_0 + Z g(r_0): one more pass and a grid barrier before the
    // first SpMV reads the neighbours' u
    if (!done) agg_coarse();
    __syncthreads();
    if (!done)
      for (int i = lo + (int)threadIdx.x; i < hi; i += blockDim.x) {
        const int a = (i - lo) / SEG_AGG_ROWS;
        R4<T> ui = u[i];
        ui.x += (T)s_gr[a][0];
        ui.y += (T)s_gr[a][1];
        ui.z += (T)s_gr[a][2];
        u[i] = ui;
      }
    if (!grid_barrier(g, epoch, &cs.ok)) return;
  }
  A a1[2] = {acc_zero<A>(), acc_zero<A>()};
  if (!done) {
    for (int i = lo + (int)threadIdx.x, m = 0; i < hi || (COARSE && m * (int)blockDim.x < hi - lo);
         i += blockDim.x, ++m) {
      float wz[3] = {0.0f, 0.0f, 0.0f}, rz[3] = {0.0f, 0.0f, 0.0f};
      if (i < hi) {
        const T dg = d.diag[i];
        const R4<T> ui = u[i], ri = r[i];
        T ax, ay, az;
        spmv_row(d, i, u, dg, ui, ax, ay, az);
        R4<T> wi;
        wi.x = ax; wi.y = ay; wi.z = az; wi.w = T(0);
        w[i] = wi;
        a1[0] = acc_add(a1[0], dot3(ri.x, ri.y, ri.z, ui.x, ui.y, ui.z));
        a1[1] = acc_add(a1[1], dot3(ax, ay, az, ui.x, ui.y, ui.z));
        wz[0] = (float)ax; wz[1] = (float)ay; wz[2] = (float)az;
        rz[0] = (float)ri.x; rz[1] = (float)ri.y; rz[2] = (float)ri.z;
      }
      if constexpr (COARSE) {
        seg_agg_partial<3>(wz, m, s_zp, 0);
        seg_agg_partial<3>(rz, m, s_zp, 3);
      }
    }
  }
  if constexpr (COARSE) {
    __syncthreads();
    if (!done) {
      agg_store(0);
      agg_store(1);
    }
  }
  {
    double bs[2], t[2];
    block_sums<2, NW>(a1, cs.sh, bs);
    if (w0) {
      const bool ok = warp0_reduce<2>(g, epoch, bs, rb0, rb1, t);
      if (lane == 0) {
        if (ok && !done) {
          gamma = t[0];
          alpha = gamma / t[1];
        }
        cs.ta = (T)alpha;
        cs.tb = T(0);
        cs.flag = ok ? CG_CONTINUE : CG_ABORT;
      }
    }
    __syncthreads();
  }
  if (cs.flag == CG_ABORT) return;
  T ta = cs.ta, tb = T(0);
  if constexpr (COARSE) {
    if (!done) agg_coarse();  // g(w_0), g(r_0)
    __syncthreads();
  }
  bool first = true;
  int it = 1;
  for (;; ++it) {
    if constexpr (COARSE) {
      // g(s_k) = g(w_k) + beta_k g(s_k-1); g(r_k+1) = g(r_k) - alpha_k g(s_k)
      if (!done)
        for (int k = threadIdx.x; k < na_b * 3; k += blockDim.x) {
          const int a = k / 3, c = k % 3;
          const float gs = first ? s_gw[a][c] : s_gw[a][c] + (float)tb * s_gs[a][c];
          s_gs[a][c] = gs;
          s_gr[a][c] = s_gr[a][c] - (float)ta * gs;
        }
      __syncthreads();
    }
    // r.u and r.r of the new residual are formed in the update pass, so the
    // SpMV pass does not read r again (same values, same order of rows)
    A a_ru = acc_zero<A>(), a_rr = acc_zero<A>();
    if (!done) {
      for (int i = lo + (int)threadIdx.x, m = 0; i < hi || (COARSE && m * (int)blockDim.x < hi - lo);
           i += blockDim.x, ++m) {
        float rz[3] = {0.0f, 0.0f, 0.0f};
        if (i < hi) {
          const R4<T> ui = u[i], wi = w[i];
          R4<T> pi, si;
          if (first) {
            pi = ui;
            si = wi;
          } else {
            const R4<T> po = p[i], so = s[i];
            pi.x = ui.x + tb * po.x; pi.y = ui.y + tb * po.y; pi.z = ui.z + tb * po.z;
            si.x = wi.x + tb * so.x; si.y = wi.y + tb * so.y; si.z = wi.z + tb * so.z;
          }
          pi.w = T(0);
          si.w = T(0);
          p[i] = pi;
          s[i] = si;
          R4<T> di = dx[i], ri = r[i];
          di.x += ta * pi.x; di.y += ta * pi.y; di.z += ta * pi.z;
          ri.x -= ta * si.x; ri.y -= ta * si.y; ri.z -= ta * si.z;
          dx[i] = di;
          r[i] = ri;
          const T idg = T(1) / d.diag[i];
          R4<T> un;
          un.x = ri.x * idg; un.y = ri.y * idg; un.z = ri.z * idg; un.w = T(0);
          if constexpr (COARSE) {
            const int a = (i - lo) / SEG_AGG_ROWS;
            un.x += (T)s_gr[a][0];
            un.y += (T)s_gr[a][1];
            un.z += (T)s_gr[a][2];
          }
          u[i] = un;
          a_ru = acc_add(a_ru, dot3(ri.x, ri.y, ri.z, un.x, un.y, un.z));
          a_rr = acc_add(a_rr, dot3(ri.x, ri.y, ri.z, ri.x, ri.y, ri.z));
          rz[0] = (float)ri.x; rz[1] = (float)ri.y; rz[2] = (float)ri.z;
        }
        if constexpr (COARSE) seg_agg_partial<3>(rz, m, s_zp, 3);
      }
    }
    if (!grid_barrier(g, epoch, &cs.ok)) return;
    // every block reads the same count: increments happen before this barrier
    const unsigned n_done = __ldcg(&d.ctrl->queue);
    if ((int)n_done >= d.n_robots || it > d.max_iter) break;
    A a2[3] = {a_ru, acc_zero<A>(), a_rr};
    if (!done) {
      for (int i = lo + (int)threadIdx.x, m = 0; i < hi || (COARSE && m * (int)blockDim.x < hi - lo);
           i += blockDim.x, ++m) {
        float wz[3] = {0.0f, 0.0f, 0.0f};
        if (i < hi) {
          const T dg = d.diag[i];
          const R4<T> ui = u[i];
          T ax, ay, az;
          spmv_row(d, i, u, dg, ui, ax, ay, az);
          R4<T> wi;
          wi.x = ax; wi.y = ay; wi.z = az; wi.w = T(0);
          w[i] = wi;
          a2[1] = acc_add(a2[1], dot3(ax, ay, az, ui.x, ui.y, ui.z));
          wz[0] = (float)ax; wz[1] = (float)ay; wz[2] = (float)az;
        }
        if constexpr (COARSE) seg_agg_partial<3>(wz, m, s_zp, 0);
      }
    }
    if constexpr (COARSE) {
      __syncthreads();
      if (!done) {
        agg_store(0);
        agg_store(1);
      }
    }
    {
      double bs[3], t[3];
      block_sums<3, NW>(a2, cs.sh, bs);
      if (w0) {
        const bool ok = warp0_reduce<3>(g, epoch, bs, rb0, rb1, t);
        int f = CG_ABORT;
        if (ok) f = done ? CG_DONE : cg_scalars_warp(t, bb, d.tol2, gamma, alpha, beta, rr);
        if (lane == 0) {
          if (ok) {
            if (!done) {
              if (f == CG_NONFINITE && b == rb0) set_status(d.ctrl, ST_NONFINITE);
              if (f != CG_CONTINUE) {
                it_done = it;
                if (b == rb0) atomicAdd(&d.ctrl->queue, 1u);
              }
            }
            cs.ta = (T)alpha;
            cs.tb = (T)beta;
          }
          cs.flag = f;
        }
      }
      __syncthreads();
    }
    const int f = cs.flag;
    if (f == CG_ABORT) return;
    if (f != CG_CONTINUE) done = true;
    ta = cs.ta;
    tb = cs.tb;
    first = false;
    if constexpr (COARSE) {
      if (!done) agg_coarse();  // g(w_k+1) and a fresh g(r_k+1)
      __syncthreads();
    }
  }
  if (!done && lead) {
    it_done = d.max_iter;
    set_status(d.ctrl, ST_PCG_MAXIT);
  }
  for (int i = lo + (int)threadIdx.x; i < hi; i += blockDim.x) {
    // x_(i+1) = start + correction; the step is kept for the next start
    const R4<T> x0 = X[i];
    R4<T> xi = warm_start(d, i, x0);
    const R4<T> di = dx[i];
    xi.x += di.x; xi.y += di.y; xi.z += di.z;
    X[i] = xi;
    if (d.xstep) d.xstep[i] = R4<T>{xi.x - x0.x, xi.y - x0.y, xi.z - x0.z, T(0)};
  }
  if (lead) {
    IterRec* rec = d.hist + (d.ctrl->iter % d.hist_cap);
    atomicMax(&rec->pcg_iters, it_done);
    atomicAdd(reinterpret_cast<unsigned long long*>(&d.ctrl->total_pcg), (unsigned long long)it_done);
    const double rel = bb > 0.0 ? sqrt(rr / bb) : 0.0;
    atomicMax(reinterpret_cast<unsigned long long*>(&rec->pcg_rel_residual),
              (unsigned long long)__double_as_longlong(rel));
  }
}

// Cluster variant: one thread-block cluster of PCG_CL_SIZE CTAs solves one
// robot's system at a time, taking robots from a work queue (one persistent
// launch serves any number of independent robots).  Each CTA owns a
// contiguous range of the robot's rows and keeps all of its CG vectors in
// shared memory; the preconditioned residual u of neighbouring rows is read
// from the owning CTA's shared memory (distributed shared memory), and the
// FP64 reductions exchange one partial per CTA through distributed shared
// memory.  All synchronisation is the cluster's hardware barrier.
namespace cgx = cooperative_groups;

template <typename T>
__global__ void __launch_bounds__(PCG_CL_THREADS, 1) k_pcg_cluster(Dev<T> d) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ double sh[96];
  __shared__ double part[4];
  __shared__ double tot[4];
  __shared__ int s_robot;
  cgx::cluster_group cl = cgx::this_cluster();
  const int crank = (int)cl.block_rank();
  const int csz = (int)cl.num_blocks();
  const int cap = d.cl_rows_cap;
  R4<T>* su = reinterpret_cast<R4<T>*>(smem);
  T* sr = reinterpret_cast<T*>(su + cap);
  T* sp = sr + 3 * cap;
  T* ss = sp + 3 * cap;
  T* sw = ss + 3 * cap;
  T* sd = sw + 3 * cap;
  T* sg = sd + 3 * cap;  // diagonal

  // cluster-wide FP64 sums of nv values: block sums in one shared-memory
  // round, one partial per CTA exchanged through distributed shared memory,
  // summed by a fixed shuffle tree over the ranks (deterministic)
  auto cluster_reduce = [&](const double* v, int nv) {
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    double t[3] = {0.0, 0.0, 0.0};
    for (int k = 0; k < nv; ++k) {
      t[k] = v[k];
      for (int o = 16; o > 0; o >>= 1) t[k] += __shfl_down_sync(0xffffffffu, t[k], o);
    }
    __syncthreads();
    if (lane == 0)
      for (int k = 0; k < nv; ++k) sh[k * 32 + wid] = t[k];
    __syncthreads();
    if (threadIdx.x < 3 && threadIdx.x < nv) {
      double a = 0.0;
      const int nw = (blockDim.x + 31) >> 5;
      for (int i = 0; i < nw; ++i) a += sh[threadIdx.x * 32 + i];
      part[threadIdx.x] = a;
    }
    cl.sync();
    if (threadIdx.x < 32) {
      double a[3] = {0.0, 0.0, 0.0};
      if (lane < csz) {
        const double* rp = cl.map_shared_rank(part, lane);
        for (int k = 0; k < nv; ++k) a[k] = rp[k];
      }
      for (int k = 0; k < nv; ++k) {
        for (int o = 16; o > 0; o >>= 1) a[k] += __shfl_down_sync(0xffffffffu, a[k], o);
        if (lane == 0) tot[k] = a[k];
      }
    }
    __syncthreads();
  };

  while (true) {
    if (crank == 0 && threadIdx.x == 0) s_robot = (int)atomicAdd(&d.ctrl->queue, 1u);
    cl.sync();
    const int robot = *cl.map_shared_rank(&s_robot, 0);
    cl.sync();  // every rank has read rank 0's word before any rank moves on or exits
    if (robot >= d.n_robots) break;
    const int row0 = d.robot_row[robot];
    const int n = d.robot_row[robot + 1] - row0;
    const int rpc = (((n + csz - 1) / csz) + 31) & ~31;  // rows per CTA (host checks rpc <= cap)
    const int my0 = crank * rpc;
    const int my1 = min(n, my0 + rpc);
    const int nmine = my1 > my0 ? my1 - my0 : 0;
    // SpMV of local rows: diag * own + sum of off-diagonals over neighbours' u
    auto spmv_u = [&](int j, T& ax, T& ay, T& az) {
      const int i = row0 + my0 + j;
      const T dg = sg[j];
      const R4<T> self = su[j];
      ax = dg * self.x;
      ay = dg * self.y;
      az = dg * self.z;
      const int sl = i >> 5, lane = i & 31;
      const int base = d.sl_ptr[sl] + lane;
      const int width = (d.sl_ptr[sl + 1] - d.sl_ptr[sl]) >> 5;
      // chunks of 8 entries: all column/value loads first, then the
      // distributed-shared-memory gathers, so the loads overlap
      for (int j0 = 0; j0 < width; j0 += 8) {
        int cc[8];
        T aa[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (j0 + q < width) {
            cc[q] = d.sl_col[base + (j0 + q) * 32];
            aa[q] = d.sl_val[base + (j0 + q) * 32];
          } else {
            cc[q] = row0 + my0 + j;
            aa[q] = T(0);
          }
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int c = cc[q] - row0;
          const int owner = c / rpc;
          const R4<T> v = cl.map_shared_rank(su, owner)[c - owner * rpc];
          ax += aa[q] * v.x;
          ay += aa[q] * v.y;
          az += aa[q] * v.z;
        }
      }
    };
    // r = b - A x in FP64, u = r / diag, correction d = 0
    double a0[2] = {0.0, 0.0};
    for (int j = threadIdx.x; j < nmine; j += blockDim.x) {
      const int i = row0 + my0 + j;
      const T dg = d.diag[i];
      sg[j] = dg;
      const R4<T> xi = d.X[i];
      double ax = (double)dg * xi.x, ay = (double)dg * xi.y, az = (double)dg * xi.z;
      const int sl = i >> 5, lane = i & 31;
      const int k1 = d.sl_ptr[sl + 1];
      for (int k = d.sl_ptr[sl] + lane; k < k1; k += 32) {
        const double a = (double)d.sl_val[k];
        const R4<T> xc = d.X[d.sl_col[k]];
        ax += a * xc.x;
        ay += a * xc.y;
        az += a * xc.z;
      }
      const R4<double> bi = d.b[i];
      const double rx = bi.x - ax, ry = bi.y - ay, rz = bi.z - az;
      sr[3 * j] = (T)rx;
      sr[3 * j + 1] = (T)ry;
      sr[3 * j + 2] = (T)rz;
      su[j] = R4<T>{sr[3 * j] / dg, sr[3 * j + 1] / dg, sr[3 * j + 2] / dg, T(0)};
      sd[3 * j] = sd[3 * j + 1] = sd[3 * j + 2] = T(0);
      a0[0] += bi.x * bi.x + bi.y * bi.y + bi.z * bi.z;
      a0[1] += rx * rx + ry * ry + rz * rz;
    }
    cluster_reduce(a0, 2);  // also publishes u
    const double bb = tot[0];
    double rr = tot[1];
    int it = 0;
    if (bb > 0.0 && rr > d.tol2 * bb) {
      double a1[2] = {0.0, 0.0};
      for (int j = threadIdx.x; j < nmine; j += blockDim.x) {
        T ax, ay, az;
        spmv_u(j, ax, ay, az);
        const R4<T> uj = su[j];
        sw[3 * j] = ax; sw[3 * j + 1] = ay; sw[3 * j + 2] = az;
        sp[3 * j] = uj.x; sp[3 * j + 1] = uj.y; sp[3 * j + 2] = uj.z;
        ss[3 * j] = ax; ss[3 * j + 1] = ay; ss[3 * j + 2] = az;
        a1[0] += (double)sr[3 * j] * uj.x + (double)sr[3 * j + 1] * uj.y + (double)sr[3 * j + 2] * uj.z;
        a1[1] += (double)ax * uj.x + (double)ay * uj.y + (double)az * uj.z;
      }
      cluster_reduce(a1, 2);
      double gamma = tot[0];
      double alpha = gamma / tot[1];
      for (it = 1; it <= d.max_iter; ++it) {
        const T ta = (T)alpha;
        for (int j = threadIdx.x; j < nmine; j += blockDim.x) {
          const T dg = sg[j];
          T un[3];
          for (int c = 0; c < 3; ++c) {
            sd[3 * j + c] += ta * sp[3 * j + c];
            sr[3 * j + c] -= ta * ss[3 * j + c];
            un[c] = sr[3 * j + c] / dg;
          }
          su[j] = R4<T>{un[0], un[1], un[2], T(0)};
        }
        cl.sync();  // u published to the cluster
        double a2[3] = {0.0, 0.0, 0.0};
        for (int j = threadIdx.x; j < nmine; j += blockDim.x) {
          T ax, ay, az;
          spmv_u(j, ax, ay, az);
          const R4<T> uj = su[j];
          sw[3 * j] = ax; sw[3 * j + 1] = ay; sw[3 * j + 2] = az;
          const T r0 = sr[3 * j], r1 = sr[3 * j + 1], r2 = sr[3 * j + 2];
          a2[0] += (double)r0 * uj.x + (double)r1 * uj.y + (double)r2 * uj.z;
          a2[1] += (double)ax * uj.x + (double)ay * uj.y + (double)az * uj.z;
          a2[2] += (double)r0 * r0 + (double)r1 * r1 + (double)r2 * r2;
        }
        cluster_reduce(a2, 3);
        const double gnew = tot[0], delta = tot[1];
        rr = tot[2];
        if (!isfinite(gnew) || !isfinite(delta) || !isfinite(rr)) {
          if (crank == 0 && threadIdx.x == 0) set_status(d.ctrl, ST_NONFINITE);
          break;
        }
        if (rr <= d.tol2 * bb) break;
        const double beta = gnew / gamma;
        alpha = gnew / (delta - beta * gnew / alpha);
        gamma = gnew;
        const T tb = (T)beta;
        for (int j = threadIdx.x; j < nmine; j += blockDim.x) {
          const R4<T> uj = su[j];
          const T uu[3] = {uj.x, uj.y, uj.z};
          for (int c = 0; c < 3; ++c) {
            sp[3 * j + c] = uu[c] + tb * sp[3 * j + c];
            ss[3 * j + c] = sw[3 * j + c] + tb * ss[3 * j + c];
          }
        }
      }
      if (it > d.max_iter) {
        it = d.max_iter;
        if (crank == 0 && threadIdx.x == 0) set_status(d.ctrl, ST_PCG_MAXIT);
      }
      for (int j = threadIdx.x; j < nmine; j += blockDim.x) {
        const int i = row0 + my0 + j;
        R4<T> xi = d.X[i];
        xi.x += sd[3 * j];
        xi.y += sd[3 * j + 1];
        xi.z += sd[3 * j + 2];
        d.X[i] = xi;
      }
    }
    if (crank == 0 && threadIdx.x == 0) {
      IterRec* rec = d.hist + (d.ctrl->iter % d.hist_cap);
      atomicMax(&rec->pcg_iters, it);
      atomicAdd(reinterpret_cast<unsigned long long*>(&d.ctrl->total_pcg), (unsigned long long)it);
      const double rel = bb > 0.0 ? sqrt(rr / bb) : 0.0;
      atomicMax(reinterpret_cast<unsigned long long*>(&rec->pcg_rel_residual),
                (unsigned long long)__double_as_longlong(rel));
    }
    cl.sync();  // shared memory is reused by the next robot
  }
}

// --------------------------------------------------------------- finalize
template <typename T>
__global__ void k_finalize(Dev<T> d) {
  __shared__ double sh[32];
  const int n = d.n_e_local + d.n_e_spring;
  // fixed-order sum: eight interleaved thread-strided chains (so that the
  // loads overlap), added in a fixed order, then a fixed tree
  constexpr int K = 8;
  double a[K];
#pragma unroll
  for (int k = 0; k < K; ++k) a[k] = 0.0;
  const int step = (int)blockDim.x * K;
  for (int i0 = threadIdx.x; i0 < n; i0 += step) {
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const int i = i0 + k * (int)blockDim.x;
      if (i < n) a[k] += d.e_partials[i];
    }
  }
  double at = 0.0;
#pragma unroll
  for (int k = 0; k < K; ++k) at += a[k];
  const double t = block_sum(at, sh);
  if (threadIdx.x == 0) finalize_iteration(d, t);
}

template <typename T>
__global__ void k_gather_positions(const R4<T>* X, const int* int_of_user, int n, T* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const R4<T> x = X[int_of_user[i]];
  out[3 * (size_t)i] = x.x;
  out[3 * (size_t)i + 1] = x.y;
  out[3 * (size_t)i + 2] = x.z;
}

// ---------------------------------------------------------------- launchers
int local_blocks(int n_t, int threads) { return (n_t + threads - 1) / threads; }
int rhs_blocks(int n_free, int threads) { return (n_free + threads - 1) / threads; }
int local_blocks(int n_t) { return local_blocks(n_t, LOCAL_THREADS); }
int rhs_blocks(int n_free) { return rhs_blocks(n_free, RHS_THREADS); }

// The block sizes are launch-shape choices of the autotuner: each allowed
// size is its own instantiation (compiled with its own launch bound).
template <typename T>
void launch_local(const Dev<T>& d, cudaStream_t st) {
  if (d.n_t == 0) return;
  const int bs = d.local_threads > 0 ? d.local_threads : LOCAL_THREADS;
  const int nb = local_blocks(d.n_t, bs);
  constexpr int SW = sizeof(T) == 4 ? 4 : 6;
  if (bs == 64)
    k_local<T, SW, 64><<<nb, 64, 0, st>>>(d);
  else if (bs == 256)
    k_local<T, SW, 256><<<nb, 256, 0, st>>>(d);
  else
    k_local<T, SW, 128><<<nb, 128, 0, st>>>(d);
}

template <typename T>
void launch_rhs(const Dev<T>& d, cudaStream_t st) {
  if (d.n_free == 0) return;
  const int bs = d.rhs_threads > 0 ? d.rhs_threads : RHS_THREADS;
  const int nb = rhs_blocks(d.n_free, bs);
  if (bs == 128)
    k_rhs<T, 128><<<nb, 128, 0, st>>>(d);
  else if (bs == 512)
    k_rhs<T, 512><<<nb, 512, 0, st>>>(d);
  else
    k_rhs<T, 256><<<nb, 256, 0, st>>>(d);
}

template <typename T>
int pcg_max_grid() {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pcg<T>, PCG_THREADS, 0);
  return sms * (per > 0 ? per : 1);
}

template <typename T>
int pcg_rr_max_rows() {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pcg_rr<T, PCG_RR_MAXW>, PCG_RR_THREADS, 0);
  return sms * per * PCG_RR_THREADS;
}

template <typename T>
cudaError_t launch_pcg(const Dev<T>& d, int grid, int variant, cudaStream_t st) {
  if (d.n_free == 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(variant == 2 ? PCG_RR_THREADS : PCG_THREADS);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (variant == 2) return cudaLaunchKernelEx(&cfg, k_pcg_rr<T, PCG_RR_MAXW>, d);
  return cudaLaunchKernelEx(&cfg, k_pcg<T>, d);
}

template <typename T>
void launch_finalize(const Dev<T>& d, cudaStream_t st) {
  k_finalize<T><<<1, 1024, 0, st>>>(d);
}

template <typename T>
void launch_gather_positions(const Dev<T>& d, const int* int_of_user, int n_user, T* out,
                             cudaStream_t st) {
  if (n_user == 0) return;
  k_gather_positions<T><<<(n_user + 255) / 256, 256, 0, st>>>(d.X, int_of_user, n_user, out);
}

template <typename T>
int pcg_cluster_rows_cap() {
  // per row: u (R4) + r, p, s, w, d, diag (3+3+3+3+3+1 values)
  const size_t per_row = sizeof(R4<T>) + 16 * sizeof(T);
  const size_t avail = 220 * 1024;
  return (int)((avail / per_row) & ~size_t(31));
}

template <typename T>
int pcg_cluster_max_clusters(int rows_cap) {
  const size_t smem = (sizeof(R4<T>) + 16 * sizeof(T)) * (size_t)rows_cap;
  if (cudaFuncSetAttribute(k_pcg_cluster<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return 0;
  if (cudaFuncSetAttribute(k_pcg_cluster<T>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(PCG_CL_SIZE);
  cfg.blockDim = dim3(PCG_CL_THREADS);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = PCG_CL_SIZE;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, k_pcg_cluster<T>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  return n;
}

template <typename T>
cudaError_t launch_pcg_cluster(const Dev<T>& d, int n_clusters, cudaStream_t st) {
  if (d.n_free == 0) return cudaSuccess;
  const size_t smem = (sizeof(R4<T>) + 16 * sizeof(T)) * (size_t)d.cl_rows_cap;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(PCG_CL_SIZE * n_clusters);
  cfg.blockDim = dim3(PCG_CL_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = PCG_CL_SIZE;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k_pcg_cluster<T>, d);
}

template <typename T>
int pcg_seg_max_blocks() {
  int dev = 0, sms = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_pcg_seg<T, std::is_same<T, float>::value>,
                                                PCG_SEG_THREADS, 0);
  return sms * per;
}

template <typename T>
cudaError_t launch_pcg_seg(const Dev<T>& d, int blocks, cudaStream_t st) {
  if (d.n_free == 0) return cudaSuccess;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(blocks);
  cfg.blockDim = dim3(PCG_SEG_THREADS);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if constexpr (std::is_same<T, float>::value) {
    if (d.seg_coarse) return cudaLaunchKernelEx(&cfg, k_pcg_seg<T, true>, d);
  }
  return cudaLaunchKernelEx(&cfg, k_pcg_seg<T, false>, d);
}

template int pcg_seg_max_blocks<float>();
template int pcg_seg_max_blocks<double>();
template cudaError_t launch_pcg_seg<float>(const Dev<float>&, int, cudaStream_t);
template cudaError_t launch_pcg_seg<double>(const Dev<double>&, int, cudaStream_t);
template int pcg_cluster_rows_cap<float>();
template int pcg_cluster_rows_cap<double>();
template int pcg_cluster_max_clusters<float>(int);
template int pcg_cluster_max_clusters<double>(int);
template cudaError_t launch_pcg_cluster<float>(const Dev<float>&, int, cudaStream_t);
template cudaError_t launch_pcg_cluster<double>(const Dev<double>&, int, cudaStream_t);
template void launch_local<float>(const Dev<float>&, cudaStream_t);
template void launch_local<double>(const Dev<double>&, cudaStream_t);
template void launch_rhs<float>(const Dev<float>&, cudaStream_t);
template void launch_rhs<double>(const Dev<double>&, cudaStream_t);
template cudaError_t launch_pcg<float>(const Dev<float>&, int, int, cudaStream_t);
template cudaError_t launch_pcg<double>(const Dev<double>&, int, int, cudaStream_t);
template int pcg_rr_max_rows<float>();
template int pcg_rr_max_rows<double>();
template int pcg_max_grid<float>();
template int pcg_max_grid<double>();
template void launch_finalize<float>(const Dev<float>&, cudaStream_t);
template void launch_finalize<double>(const Dev<double>&, cudaStream_t);
template void launch_gather_positions<float>(const Dev<float>&, const int*, int, float*, cudaStream_t);
template void launch_gather_positions<double>(const Dev<double>&, const int*, int, double*,
                                              cudaStream_t);

}  // namespace casim
