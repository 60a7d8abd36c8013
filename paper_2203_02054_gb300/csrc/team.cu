// Global step on teams of thread blocks (Sec. III-B, Eq. 8): one conjugate-
// gradient solve per robot, all CG vectors on chip.
//
// Every robot's free rows are cut into parts of consecutive rows; a thread
// block works on one part at a time and the blocks of a robot's parts form its
// team.  A row's CG vectors, diagonal and preconditioner data stay in
// registers for the whole solve.  There is no grid barrier:
//   * the preconditioned residual u that other parts read is published as
//     epoch-tagged words (a 16-bit tag over 48 bits of payload; aligned 8-byte
//     accesses are single-copy atomic, so a word whose tag matches holds that
//     epoch's payload) and readers re-read rows whose words are not yet
//     current;
//   * a part's contribution to the dot products is a slot of tagged words,
//     followed by one relaxed arrival on the team's counter; when the round is
//     complete every block of the team reads the team's slots and adds them in
//     part order.
// Words are double-buffered by epoch parity and zeroed before each launch.  No
// block can be more than one epoch ahead of a reader of its words (it cannot
// pass a reduction before the reader has arrived, after its last read of the
// older epoch), so a stale word's tag cannot match.  Robots of a batch neither
// wait for one another nor share scalars; with more parts than blocks a block
// works through its parts in order.  Every block takes its parts in the same
// global order (part p belongs to block p mod grid) and a robot has at most as
// many parts as the grid has blocks, so the oldest unfinished robot's team is
// always running: nothing can deadlock, and every wait is bounded all the
// same.
//
// Preconditioner: M^-1 = D^-1 + Z (A_c + sigma I)^-1 Z^T, Jacobi plus an
// additive coarse correction.  Z holds, for every part (a compact piece of the
// body), the constant and the three linear functions of the rest position,
// orthonormalised over the part (small MIXED robots: the constants of up to three
// pieces of it, without sigma); A_c = Z^T L Z is the Galerkin matrix of the
// spring-free Laplacian.  The springs add k Z^T diag(mask) Z to it, a
// different block-diagonal matrix every iteration; sigma = k (springs / rows)
// stands for it.  (Without it the coarse correction takes the body's soft
// modes for far softer than the springs leave them: M^-1 A then has a few
// eigenvalues in the hundreds, which FP32 rounding keeps re-exciting.)  The
// inverses for TEAM_LEVELS values of sigma, a factor 4 apart, are formed once at
// upload, and a solve takes the one for its number of springs.  CG iterations
// in a numpy model with FP32 vectors (1e-6, contact-bearing states; Jacobi,
// constants over 96 rows without sigma, this with the true spring matrix, this):
// gripper 86, 55, 37, 38 (parts of 288 rows), finger 79, 48, 26, 27 (96 rows),
// 80x16x16 finger 88, 56, 35, 36 (410 rows).
//
// Every block needs g(v) = (A_c + sigma I)^-1 Z^T v of its own functions for v =
// r_(k+1) before that iteration's SpMV.  From r_(k+1) = r_k - alpha_k s_k and
// s_k = w_k + beta_k s_(k-1) (w = A u): the slot carries Z^T w_k, every block
// forms g(w_k) from the slots after the round, and carries g(s) and g(r) by
// the same recurrences.  Every TEAM_REFRESH-th slot also carries Z^T r_k, from
// which g(r) is formed anew, so that its FP32 rounding cannot accumulate (a
// version that never refreshed stalled once the residual had fallen by 1e5).
#include <algorithm>
#include <type_traits>

#include "cg.cuh"
#include "common.cuh"
#include "kernels.h"

namespace casim {

static constexpr int TEAM_REFRESH = 8;  // iterations between fresh Z^T r sums
// The coarse correction is FP32 in FP64 solves too (it only preconditions),
// which makes the error that a solve leaves at its stopping test vary from
// input to input where an all-FP64 recurrence's is smooth; FP64 solves with it
// stop at 1/32 of the tolerance, so that finite differences of a run see no
// more of that error than before (about a tenth more iterations).
static constexpr double TEAM_STOP2_F64 = 1.0 / 1024.0;
static constexpr int TEAM_MAXQ = 5;  // dot slots per lane of warp 0
static_assert(32 * TEAM_MAXQ >= TEAM_MAX_PARTS, "a warp reads every slot of a team");

// ------------------------------------------------------------- tagged words
__device__ __forceinline__ void st_v2_relaxed(unsigned long long* p, unsigned long long a, unsigned long long b) {
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(a), "l"(b) : "memory");
}
__device__ __forceinline__ void ld_v2_relaxed(const unsigned long long* p, unsigned long long& a,
                                              unsigned long long& b) {
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p));
}
__device__ __forceinline__ unsigned long long tag_of(unsigned e) { return (unsigned long long)(e & 0xFFFFu) << 48; }
__device__ __forceinline__ bool has_tag(unsigned long long w, unsigned long long tag) {
  return (w & 0xFFFF000000000000ull) == tag;
}

// three floats as two words: w0 = tag | x | y[31:16], w1 = tag | y[15:0] | z
__device__ __forceinline__ void pack3(unsigned long long tag, float x, float y, float z, unsigned long long& w0,
                                      unsigned long long& w1) {
  const unsigned bx = __float_as_uint(x), by = __float_as_uint(y), bz = __float_as_uint(z);
  w0 = tag | ((unsigned long long)bx << 16) | (by >> 16);
  w1 = tag | ((unsigned long long)(by & 0xFFFFu) << 32) | bz;
}
__device__ __forceinline__ void unpack3(unsigned long long w0, unsigned long long w1, float& x, float& y, float& z) {
  x = __uint_as_float((unsigned)(w0 >> 16));
  y = __uint_as_float((((unsigned)w0 & 0xFFFFu) << 16) | ((unsigned)(w1 >> 32) & 0xFFFFu));
  z = __uint_as_float((unsigned)w1);
}

// three 64-bit values as four 48-bit chunks under one tag each
__device__ __forceinline__ void pack_192(unsigned long long tag, unsigned long long b0, unsigned long long b1,
                                         unsigned long long b2, unsigned long long (&w)[4]) {
  w[0] = tag | (b0 >> 16);
  w[1] = tag | ((b0 & 0xFFFFull) << 32) | (b1 >> 32);
  w[2] = tag | ((b1 & 0xFFFFFFFFull) << 16) | (b2 >> 48);
  w[3] = tag | (b2 & 0xFFFFFFFFFFFFull);
}
__device__ __forceinline__ void unpack_192(const unsigned long long (&w)[4], unsigned long long& b0,
                                           unsigned long long& b1, unsigned long long& b2) {
  const unsigned long long m48 = 0xFFFFFFFFFFFFull;
  const unsigned long long c0 = w[0] & m48, c1 = w[1] & m48, c2 = w[2] & m48, c3 = w[3] & m48;
  b0 = (c0 << 16) | (c1 >> 32);
  b1 = ((c1 & 0xFFFFFFFFull) << 32) | (c2 >> 16);
  b2 = ((c2 & 0xFFFFull) << 48) | c3;
}
__device__ __forceinline__ unsigned long long bits64(double v) { return (unsigned long long)__double_as_longlong(v); }
__device__ __forceinline__ unsigned long long bits64(DW v) {
  return ((unsigned long long)__float_as_uint(v.hi) << 32) | __float_as_uint(v.lo);
}
__device__ __forceinline__ void from_bits(unsigned long long b, double& v) { v = __longlong_as_double((long long)b); }
__device__ __forceinline__ void from_bits(unsigned long long b, DW& v) {
  v = DW{__uint_as_float((unsigned)(b >> 32)), __uint_as_float((unsigned)b)};
}

// Bounded polling: every 32nd poll checks the abort word and the clock budget
// (on expiry records ST_TIMEOUT and raises abort).  Returns false to stop.
struct TeamWait {
  long long t0 = 0;
  unsigned n = 0;
  __device__ __forceinline__ bool again(Ctrl* c, unsigned long long budget) {
    if ((++n & 31u) != 0) return true;
    if (*(volatile int*)&c->abort) return false;
    const long long now = clock64();
    if (t0 == 0) {
      t0 = now;
      return true;
    }
    if ((unsigned long long)(now - t0) > budget) {
      atomicExch(&c->abort, 1);
      atomicOr(&c->status, ST_TIMEOUT);
      return false;
    }
    return true;
  }
};

// One published value of u per thread: a row's three floats, or one FP64
// column of it (64 bits in two words of 48 and 16).
template <typename T>
struct Cols;
template <>
struct Cols<float> {
  static constexpr int N = 3;      // columns per thread
  static constexpr int PUBS = 1;   // published values per row
};
template <>
struct Cols<double> {
  static constexpr int N = 1;
  static constexpr int PUBS = 3;
};
__device__ __forceinline__ void publish_u(unsigned long long* p, unsigned long long tag, const float (&u)[3]) {
  unsigned long long a, b;
  pack3(tag, u[0], u[1], u[2], a, b);
  st_v2_relaxed(p, a, b);
}
__device__ __forceinline__ void publish_u(unsigned long long* p, unsigned long long tag, const double (&u)[1]) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(u[0]);
  st_v2_relaxed(p, tag | (b >> 16), tag | (b & 0xFFFFull));
}
__device__ __forceinline__ void unpack_u(unsigned long long a, unsigned long long b, float (&v)[3]) {
  unpack3(a, b, v[0], v[1], v[2]);
}
__device__ __forceinline__ void unpack_u(unsigned long long a, unsigned long long b, double (&v)[1]) {
  v[0] = __longlong_as_double((long long)((a << 16) | (b & 0xFFFFull)));
}

// The part's rows of u in shared memory: a float4 per row (one 16-byte load per
// matrix entry), or one array of doubles per column.
__device__ __forceinline__ void halo_put(void* h, int k, const float (&v)[3]) {
  static_cast<float4*>(h)[k] = make_float4(v[0], v[1], v[2], 0.0f);
}
__device__ __forceinline__ void halo_put(void* h, int k, const double (&v)[1]) { static_cast<double*>(h)[k] = v[0]; }
__device__ __forceinline__ void halo_axpy(const void* h, int k, float c, float (&o)[3]) {
  const float4 v = static_cast<const float4*>(h)[k];
  o[0] += c * v.x;
  o[1] += c * v.y;
  o[2] += c * v.z;
}
__device__ __forceinline__ void halo_axpy(const void* h, int k, double c, double (&o)[1]) {
  o[0] = fma(c, static_cast<const double*>(h)[k], o[0]);
}
static size_t halo_bytes(bool fp64, int rows) { return (size_t)rows * (fp64 ? 24 : 16); }

// dot product of a thread's columns, for one row or one column of it
__device__ __forceinline__ DW dot_cols(const float (&a)[3], const float (&b)[3]) {
  return dot3(a[0], a[1], a[2], b[0], b[1], b[2]);
}
__device__ __forceinline__ double dot_cols(const double (&a)[1], const double (&b)[1]) { return a[0] * b[0]; }

// ------------------------------------------------------------- warp sums
// Warp sums of N values by a butterfly in which the lanes hand over half of
// the values they still carry at every distance (16, 8, 4, 2, 1) and finish
// the rest: about N exchanges in all instead of 5 N.  Sum k is stored to
// dst[k] by the lane that ends with it.  The pairs added depend only on N.
template <int N, int O>
struct WarpScatterSum {
  static __device__ __forceinline__ void run(const float (&v)[N], int first, int count, bool owner, float* dst) {
    const int lane = threadIdx.x & 31;
    if constexpr (O == 0) {
#pragma unroll
      for (int k = 0; k < N; ++k)
        if (owner && k < count) dst[first + k] = v[k];
    } else if constexpr (N == 1) {
      const float x[1] = {__fadd_rn(v[0], __shfl_xor_sync(0xffffffffu, v[0], O))};
      WarpScatterSum<1, O / 2>::run(x, first, count, owner && !(lane & O), dst);
    } else {
      constexpr int H = (N + 1) / 2;
      const bool up = lane & O;
      float x[H];
#pragma unroll
      for (int k = 0; k < H; ++k) {
        const float hi = H + k < N ? v[H + k < N ? H + k : 0] : 0.0f;
        x[k] = __fadd_rn(up ? hi : v[k], __shfl_xor_sync(0xffffffffu, up ? v[k] : hi, O));
      }
      WarpScatterSum<H, O / 2>::run(x, first + (up ? H : 0), up ? count - H : (count < H ? count : H), owner, dst);
    }
  }
};
template <int N>
__device__ __forceinline__ void warp_scatter_sum(const float (&v)[N], float* dst) {
  WarpScatterSum<N, 16>::run(v, 0, N, true, dst);
}

// Addition inside a tree: double words are not renormalised (the low parts
// stay below n u of the sum of n terms; their rounding is of order u^2).
__device__ __forceinline__ DW tree_add(DW a, DW b) {
  DW z;
  float e;
  two_sum_f(a.hi, b.hi, z.hi, e);
  z.lo = __fadd_rn(e, __fadd_rn(a.lo, b.lo));
  return z;
}
__device__ __forceinline__ double tree_add(double a, double b) { return a + b; }
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }

// Warp sums of N <= 3 accumulators by one butterfly in which the lanes hand over
// half of the values they carry at distances 16 and 8: value k ends in lanes 8 k
// .. 8 k + 7 (N > 1).  Six exchanges for three values instead of fifteen: an
// FP64 addition occupies its scheduler's pipe for 64 cycles whatever the lanes.
template <int N, typename S>
__device__ __forceinline__ S warp_sums(const S (&v)[N]) {
  const int lane = threadIdx.x & 31;
  S x;
  if constexpr (N == 1) {
    x = tree_add(v[0], shfl_xor(v[0], 16));
    x = tree_add(x, shfl_xor(x, 8));
  } else {
    const S zero = acc_zero<S>();
    const bool up = lane & 16, up8 = lane & 8;
    const S v2 = N > 2 ? v[N > 2 ? 2 : 0] : zero;
    const S k0 = tree_add(up ? v2 : v[0], shfl_xor(up ? v[0] : v2, 16));
    const S k1 = tree_add(up ? zero : v[1], shfl_xor(up ? v[1] : zero, 16));
    x = tree_add(up8 ? k1 : k0, shfl_xor(up8 ? k0 : k1, 8));
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) x = tree_add(x, shfl_xor(x, o));
  return x;
}
// the warp's sums of values k0 .. k0 + N - 1 into sa[k][warp]
template <int N, typename S>
__device__ __forceinline__ void store_sums(const S (&v)[N], int k0, S (*sa)[32]) {
  const int lane = threadIdx.x & 31;
  const S x = warp_sums<N>(v);
  if ((lane & 7) == 0 && lane < 8 * N) sa[k0 + (lane >> 3)][threadIdx.x >> 5] = x;
}
// Sums of warps [q0, q1) in warp order, value min(lane, 2) in every lane
template <typename S>
__device__ __forceinline__ S add_sums3(const S (*sa)[32], int q0, int q1) {
  const int k = min((int)(threadIdx.x & 31), 2);
  S t = sa[k][q0];
#pragma unroll 4
  for (int q = q0 + 1; q < q1; ++q) t = tree_add(t, sa[k][q]);
  return t;
}
__device__ __forceinline__ DW acc_norm(DW a) { return dw_norm(a); }
__device__ __forceinline__ double acc_norm(double a) { return a; }
__device__ __forceinline__ DW shfl_at(DW v, int l) {
  return DW{__shfl_sync(0xffffffffu, v.hi, l), __shfl_sync(0xffffffffu, v.lo, l)};
}
__device__ __forceinline__ double shfl_at(double v, int l) { return __shfl_sync(0xffffffffu, v, l); }

// ------------------------------------------------------------- rounds
// A slot is ten pairs of words: two pairs for the dot products, then one per
// basis function for the three columns of Z^T w, then the same for Z^T r.  A
// team's slots are stored pair by pair, so that the threads that read one part
// each read whole lines.
static constexpr int SLOT_W = 2, SLOT_R = 6, SLOT_WORDS = 20;

template <typename T>
struct TeamCtx {
  const Dev<T>& d;
  TeamPart pt;
  int me;      // this part within its team
  int copies;  // copies of the slots and counters in use
  // pair p of part j's slot of epoch e
  __device__ __forceinline__ unsigned long long* slot(unsigned e, int copy, int p, int j) const {
    return d.tm_slot + (((size_t)copy * 2 + (e & 1u)) * d.tm_parts + pt.p0) * SLOT_WORDS + 2 * ((size_t)p * pt.np + j);
  }
  __device__ __forceinline__ unsigned* counter(int copy) const {
    return d.tm_count + 32 * ((size_t)copy * d.n_robots + pt.robot);
  }
};

// Warp 0: the block's dot sums (value k in lane k) and its coarse sums (which:
// bit 0 Z^T w, bit 1 Z^T r; sz: lane l's of the 24 sums) as the part's slot of
// epoch e, then the arrival and the wait for the round.  A team of more than
// 32 parts keeps its slots and its counter in TEAM_COPIES copies, and block b
// uses copy b mod TEAM_COPIES: every block reads every slot once per round and
// polls the counter, and spreading those reads over addresses in different L2
// slices shortens their queues.  The arrival is a fire-and-forget add: after
// round e of a launch (counted from 1) the counter's top bit equals e & 1,
// because it starts at zero and every complete round adds 2^31.  Returns false
// (warp-uniform) when the wait gave up or another block aborted.
template <typename T, typename S>
__device__ __forceinline__ bool team_publish(const TeamCtx<T>& c, unsigned e, S dots, int which, float sz) {
  const int lane = threadIdx.x & 31;
  const unsigned long long tag = tag_of(e);
  unsigned long long b[3], w[4];
#pragma unroll
  for (int k = 0; k < 3; ++k) b[k] = __shfl_sync(0xffffffffu, bits64(dots), k);
  pack_192(tag, b[0], b[1], b[2], w);
  // lanes 0..7: the pair of words of function lane & 3 (w, then r)
  const float z0 = __shfl_sync(0xffffffffu, sz, min(3 * lane, 21)), z1 = __shfl_sync(0xffffffffu, sz, min(3 * lane + 1, 22)),
              z2 = __shfl_sync(0xffffffffu, sz, min(3 * lane + 2, 23));
  unsigned long long a0 = 0, a1 = 0;
  int at = -1;
  if (lane >= 30) {
    a0 = lane == 30 ? w[0] : w[2];
    a1 = lane == 30 ? w[1] : w[3];
    at = lane - 30;
  } else if (c.d.tm_coarse && lane < 8 && (which >> (lane >> 2)) & 1) {
    pack3(tag, z0, z1, z2, a0, a1);
    at = SLOT_W + lane;
  }
  if (at >= 0)
    for (int k = 0; k < c.copies; ++k) st_v2_relaxed(c.slot(e, k, at, c.me), a0, a1);
  __syncwarp();
  if (lane < c.copies)
    atomicAdd(c.counter(lane), c.me == 0 ? (0x80000000u - ((unsigned)c.pt.np - 1u + c.d.bar_extra)) : 1u);
  int arrived = 1;
  if (lane == 0) {
    const unsigned want = (e & 1u) << 31;
    volatile unsigned* vc = c.counter(c.me % c.copies);
    TeamWait wt;
    while ((*vc & 0x80000000u) != want)
      if (!wt.again(c.d.ctrl, c.d.wait_budget)) {
        arrived = 0;
        break;
      }
  }
  return __shfl_sync(0xffffffffu, arrived, 0) != 0;
}

// After the round: N pairs of part j's slot from pair p on, read again until
// they are current; false when that wait gave up.
template <int N, typename T>
__device__ __forceinline__ bool team_read(const TeamCtx<T>& c, unsigned e, int p, int j, unsigned long long (&x)[2 * N]) {
  const unsigned long long* s = c.slot(e, c.me % c.copies, p, j);
  const unsigned long long tag = tag_of(e);
  TeamWait wt;
  for (;;) {
    bool ok = true;
#pragma unroll
    for (int k = 0; k < N; ++k) ld_v2_relaxed(s + 2 * (size_t)k * c.pt.np, x[2 * k], x[2 * k + 1]);
#pragma unroll
    for (int k = 0; k < 2 * N; ++k) ok = ok && has_tag(x[k], tag);
    if (ok) return true;
    if (!wt.again(c.d.ctrl, c.d.wait_budget)) return false;
  }
}
// part j's dot sums
template <typename T, typename S>
__device__ __forceinline__ bool team_read_dots(const TeamCtx<T>& c, unsigned e, int j, S (&v)[3]) {
  unsigned long long w[4], b0, b1, b2;
  const bool ok = team_read<2>(c, e, 0, j, w);
  unpack_192(w, b0, b1, b2);
  from_bits(b0, v[0]);
  from_bits(b1, v[1]);
  from_bits(b2, v[2]);
  return ok;
}
// part j's share of g = (A_c + sigma I)^-1 Z^T x for the block's four functions
// (ainv: their rows of the inverse, nd columns) from its sums z[m][k]
__device__ __forceinline__ void coarse_share(const float* ainv, int nd, int j, const float (&z)[4][3], float (&out)[12]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const float4 a = *reinterpret_cast<const float4*>(ainv + (size_t)i * nd + 4 * j);
#pragma unroll
    for (int k = 0; k < 3; ++k)
      out[3 * i + k] = __fmaf_rn(a.w, z[3][k], __fmaf_rn(a.z, z[2][k], __fmaf_rn(a.y, z[1][k], __fmul_rn(a.x, z[0][k]))));
  }
}

// the same from its slot, x's pairs from p on
template <typename T>
__device__ __forceinline__ bool team_read_coarse(const TeamCtx<T>& c, unsigned e, int p, int j, const float* ainv,
                                                 int nd, float (&out)[12]) {
  unsigned long long x[8];
  float z[4][3];
  const bool ok = team_read<4>(c, e, p, j, x);
#pragma unroll
  for (int k = 0; k < 4; ++k) unpack3(x[2 * k], x[2 * k + 1], z[k][0], z[k][1], z[k][2]);
  coarse_share(ainv, nd, j, z, out);
  return ok;
}

// Warp 0 of an FP32 solve: the team's dot sums, each lane its slots (lane, lane
// + 32, ...) in part order, then a fixed shuffle tree: value k ends in lanes 8 k
// to 8 k + 7.  False (per lane) when a wait gave up.
template <typename T, typename S>
__device__ __forceinline__ bool team_dots(const TeamCtx<T>& c, unsigned e, S& tot) {
  const int lane = threadIdx.x & 31;
  unsigned long long w[TEAM_MAXQ][4];
  const unsigned long long tag = tag_of(e);
  const unsigned long long* s = c.slot(e, c.me % c.copies, 0, lane);
  const size_t hi = 2 * (size_t)c.pt.np;
#pragma unroll
  for (int q = 0; q < TEAM_MAXQ; ++q)
    if (lane + 32 * q < c.pt.np) {
      ld_v2_relaxed(s + 64 * q, w[q][0], w[q][1]);
      ld_v2_relaxed(s + 64 * q + hi, w[q][2], w[q][3]);
    }
  S a[3] = {acc_zero<S>(), acc_zero<S>(), acc_zero<S>()};
  bool ok = true;
#pragma unroll
  for (int q = 0; q < TEAM_MAXQ; ++q)
    if (lane + 32 * q < c.pt.np) {
      S v[3];
      if (has_tag(w[q][0], tag) && has_tag(w[q][1], tag) && has_tag(w[q][2], tag) && has_tag(w[q][3], tag)) {
        unsigned long long b0, b1, b2;
        unpack_192(w[q], b0, b1, b2);
        from_bits(b0, v[0]);
        from_bits(b1, v[1]);
        from_bits(b2, v[2]);
      } else {
        ok = ok && team_read_dots(c, e, lane + 32 * q, v);
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) a[k] = tree_add(a[k], v[k]);
    }
  tot = warp_sums<3>(a);
  return ok;
}

// ---- teams of up to TEAM_CLUSTER parts: one thread-block cluster
// The blocks read one another's rows of u and write one another's slots in
// distributed shared memory, ordered by the cluster's hardware barrier: about
// 200 ns each instead of the two or three round trips through L2.
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ unsigned peer_addr(const void* p, int rank) {
  unsigned a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((unsigned)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ void peer_load(unsigned a, float (&v)[3]) {
  asm volatile(
      "{\n\t.reg .f32 pad;\n\t"
      "ld.shared::cluster.v4.f32 {%0, %1, %2, pad}, [%3];\n\t}"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2])
      : "r"(a)
      : "memory");
}
__device__ __forceinline__ void peer_load(unsigned a, double (&v)[1]) {
  asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v[0]) : "r"(a) : "memory");
}
__device__ __forceinline__ void peer_store(unsigned a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void peer_store(unsigned a, unsigned long long v) {
  asm volatile("st.shared::cluster.u64 [%0], %1;" ::"r"(a), "l"(v) : "memory");
}

// ------------------------------------------------ right-hand side of a row
// Everything of row i's right-hand side and first residual that does not
// depend on this iteration's springs: b0 = sum of the row's P_e columns -
// A_fx x_fixed and r0 = b0 - L x, x the solve's starting point.  A launch of
// its own beside the spring update and the ray casts (it needs only the local
// step's targets): inside the solver these gathers would run with one warp per
// scheduler on every block's path to the first reduction.  For FP32 positions
// in double words (two float4 per value: high and low parts), else in FP64.
__global__ void __launch_bounds__(256) k_team_rhs_f32(Dev<float> d) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= d.n_free) return;
  DW b[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
  const int k1 = d.inc_ptr[i + 1];
#pragma unroll 8
  for (int k = d.inc_ptr[i]; k < k1; ++k) {
    const R4<float> p = d.P[chk_idx(d.ctrl, d.inc[k], 4 * d.n_t)];
    dw_acc(b[0], p.x);
    dw_acc(b[1], p.y);
    dw_acc(b[2], p.z);
  }
  const R4<double> bf = d.bfix[i];
  if (bf.x != 0.0 || bf.y != 0.0 || bf.z != 0.0) {
    const double fv[3] = {bf.x, bf.y, bf.z};
    for (int c = 0; c < 3; ++c) b[c] = dw_add_sloppy(dw_norm(b[c]), dw_neg(dw_from(fv[c])));
  }
  const R4<float> xs = warm_start(d, i, d.X[i]);
  const float dg = d.diagL[i];
  DW ax[3] = {{0.0f, 0.0f}, {0.0f, 0.0f}, {0.0f, 0.0f}};
  dw_acc_prod(ax[0], dg, xs.x);
  dw_acc_prod(ax[1], dg, xs.y);
  dw_acc_prod(ax[2], dg, xs.z);
  const int sl = i >> 5, e1 = d.sl_ptr[sl + 1];
#pragma unroll 4
  for (int k = d.sl_ptr[sl] + (i & 31); k < e1; k += 32) {
    const int col = chk_idx(d.ctrl, d.sl_col[k], d.n_free);
    const float v = d.sl_val[k];
    const R4<float> xc = warm_start(d, col, d.X[col]);
    dw_acc_prod(ax[0], v, xc.x);
    dw_acc_prod(ax[1], v, xc.y);
    dw_acc_prod(ax[2], v, xc.z);
  }
  DW r[3];
  for (int c = 0; c < 3; ++c) {
    b[c] = dw_norm(b[c]);
    r[c] = dw_add_sloppy(b[c], dw_neg(dw_norm(ax[c])));
  }
  float4* bo = reinterpret_cast<float4*>(d.tm_b) + 2 * (size_t)i;
  float4* ro = reinterpret_cast<float4*>(d.tm_r) + 2 * (size_t)i;
  bo[0] = make_float4(b[0].hi, b[1].hi, b[2].hi, 0.0f);
  bo[1] = make_float4(b[0].lo, b[1].lo, b[2].lo, 0.0f);
  ro[0] = make_float4(r[0].hi, r[1].hi, r[2].hi, 0.0f);
  ro[1] = make_float4(r[0].lo, r[1].lo, r[2].lo, 0.0f);
}

__global__ void __launch_bounds__(128) k_team_rhs_f64(Dev<double> d) {
  // one thread per (row, column): the additions of a row are a chain of FP64
  // operations at tens of cycles each, so three threads share a row
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int i = t / 3, c = t - 3 * i;
  if (i >= d.n_free) return;
  const double* P = reinterpret_cast<const double*>(d.P);
  const double* X = reinterpret_cast<const double*>(d.X);
  double b0 = 0.0, b1 = 0.0;
  const int k0 = d.inc_ptr[i], k1 = d.inc_ptr[i + 1];
  int k = k0;
#pragma unroll 4
  for (; k + 1 < k1; k += 2) {
    b0 += P[4 * (size_t)chk_idx(d.ctrl, d.inc[k], 4 * d.n_t) + c];
    b1 += P[4 * (size_t)chk_idx(d.ctrl, d.inc[k + 1], 4 * d.n_t) + c];
  }
  if (k < k1) b0 += P[4 * (size_t)chk_idx(d.ctrl, d.inc[k], 4 * d.n_t) + c];
  const double b = b0 + b1 - reinterpret_cast<const double*>(d.bfix)[4 * (size_t)i + c];
  double a0 = d.diagL[i] * X[4 * (size_t)i + c], a1 = 0.0;
  const int sl = i >> 5, e1 = d.sl_ptr[sl + 1];
  int e = d.sl_ptr[sl] + (i & 31);
#pragma unroll 4
  for (; e + 32 < e1; e += 64) {
    a0 = fma(d.sl_val[e], X[4 * (size_t)chk_idx(d.ctrl, d.sl_col[e], d.n_free) + c], a0);
    a1 = fma(d.sl_val[e + 32], X[4 * (size_t)chk_idx(d.ctrl, d.sl_col[e + 32], d.n_free) + c], a1);
  }
  if (e < e1) a0 = fma(d.sl_val[e], X[4 * (size_t)chk_idx(d.ctrl, d.sl_col[e], d.n_free) + c], a0);
  reinterpret_cast<double*>(d.tm_b)[4 * (size_t)i + c] = b;
  reinterpret_cast<double*>(d.tm_r)[4 * (size_t)i + c] = b - (a0 + a1);
}

// The row's diagonal, first residual, and its terms of ||b||^2, ||r0||^2 and
// of the spring energy, from the arrays above and this iteration's springs;
// in the reverse pass (rhs_in_pcg 0) b and the diagonal are given and the
// start is zero.
__device__ __forceinline__ void team_row_start(const Dev<float>& d, int i, int, float& dg, float (&r)[3],
                                               DW (&a0)[3]) {
  if (!d.rhs_in_pcg) {
    const R4<double> bi = d.b[i];
    dg = d.diag[i];
    r[0] = (float)bi.x;
    r[1] = (float)bi.y;
    r[2] = (float)bi.z;
    const DW bb = dw_from(bi.x * bi.x + bi.y * bi.y + bi.z * bi.z);
    a0[0] = acc_add(a0[0], bb);
    a0[1] = acc_add(a0[1], bb);
    return;
  }
  const float4* bp = reinterpret_cast<const float4*>(d.tm_b) + 2 * (size_t)i;
  const float4* rp = reinterpret_cast<const float4*>(d.tm_r) + 2 * (size_t)i;
  const float4 bh = bp[0], rh = rp[0];
  const R4<double> sc = d.spring_c[i];
  const double km = d.k_spring * sc.w;
  dg = d.diagL[i] + (float)km;
  float b[3] = {bh.x, bh.y, bh.z};
  r[0] = rh.x;
  r[1] = rh.y;
  r[2] = rh.z;
  if (km != 0.0) {
    const float4 bl = bp[1], rl = rp[1];
    const R4<float> xi = d.X[i];
    const R4<float> xs = warm_start(d, i, xi);
    const double cv[3] = {sc.x, sc.y, sc.z};
    const float blo[3] = {bl.x, bl.y, bl.z}, rlo[3] = {rl.x, rl.y, rl.z}, xsv[3] = {xs.x, xs.y, xs.z};
    for (int c = 0; c < 3; ++c) {
      b[c] = dw_add_sloppy(DW{b[c], blo[c]}, dw_from(km * cv[c])).hi;
      r[c] = dw_add_sloppy(DW{r[c], rlo[c]}, dw_from(km * (cv[c] - (double)xsv[c]))).hi;
    }
    const double ex = (double)xi.x - sc.x, ey = (double)xi.y - sc.y, ez = (double)xi.z - sc.z;
    a0[2] = acc_add(a0[2], dw_from(km * (ex * ex + ey * ey + ez * ez)));
  }
  a0[0] = acc_add(a0[0], dot3(b[0], b[1], b[2], b[0], b[1], b[2]));
  a0[1] = acc_add(a0[1], dot3(r[0], r[1], r[2], r[0], r[1], r[2]));
}
__device__ __forceinline__ void team_row_start(const Dev<double>& d, int i, int c, double& dg, double (&r)[1],
                                               double (&a0)[3]) {
  const size_t k = 4 * (size_t)i + c;
  double b;
  if (!d.rhs_in_pcg) {
    b = r[0] = reinterpret_cast<const double*>(d.b)[k];
    dg = d.diag[i];
  } else {
    b = reinterpret_cast<const double*>(d.tm_b)[k];
    r[0] = reinterpret_cast<const double*>(d.tm_r)[k];
    dg = d.diagL[i];
    const double mask = d.spring_c[i].w;
    if (mask != 0.0) {
      const double km = d.k_spring * mask, x = reinterpret_cast<const double*>(d.spring_c)[k];
      const double ex = x - reinterpret_cast<const double*>(d.X)[k];
      dg += km;
      b += km * x;
      r[0] += km * ex;
      a0[2] += km * ex * ex;
    }
  }
  a0[0] += b * b;
  a0[1] += r[0] * r[0];
}

// CG scalars from a round's totals (gamma_k, delta_k, rr), by all of warp 0:
// alpha_k = gamma_k / (delta_k - beta_k gamma_k / alpha_(k-1)) with beta_k =
// gamma_k / gamma_(k-1), rearranged with q = gamma_(k-1) alpha_(k-1) (formed in
// the round before) to alpha_k = gamma_k q / (delta_k q - gamma_k^2).  FP32
// solves form them in double words (an FP64 division is a chain of operations
// at 64 cycles each); in FP64 lanes 0 and 1 share one division.
template <typename A>
struct CgState {
  A gamma, q, rr;  // gamma_(k-1), q, the last ||r||^2
  double bb, thr;  // ||b||^2, tol^2 ||b||^2
};
// Double-word quotient from the reciprocal y of b.hi: q = a.hi y, then two
// correction steps with the exact remainder a - q b (TwoProd), so that the
// rounded reciprocal costs no accuracy (relative error a few u^2).
__device__ __forceinline__ DW dw_div_fast(DW a, DW b) {
  const float y = __frcp_rn(b.hi);
  const float q = __fmul_rn(a.hi, y);
  const float p = __fmul_rn(q, b.hi);
  float r = __fsub_rn(__fsub_rn(a.hi, p), __fmaf_rn(q, b.hi, -p));
  r = __fmaf_rn(-q, b.lo, __fadd_rn(r, a.lo));
  const float c = __fmul_rn(r, y);
  r = __fmaf_rn(-c, b.hi, r);
  DW z;
  fast_two_sum_f(q, __fmaf_rn(r, y, c), z.hi, z.lo);
  return z;
}
__device__ __forceinline__ int team_scalars(const DW (&t)[3], bool first, CgState<DW>& cg, float& ta, float& tb) {
  if (!isfinite(t[0].hi) || !isfinite(t[1].hi) || !isfinite(t[2].hi)) return CG_NONFINITE;
  DW alpha;
  if (first) {
    alpha = dw_div_fast(t[0], t[1]);
    tb = 0.0f;
  } else {
    cg.rr = t[2];
    if (t[2].hi <= (float)cg.thr) return CG_DONE;
    // gamma brought to [1, 2) by a power of two, and the others with it: their
    // products, squares of squared residuals, would leave FP32's range for
    // residuals below 1e-10 or above 1e9
    const int e = min(max(((__float_as_int(t[0].hi) >> 23) & 255) - 127, -126), 126);
    const float sc = __int_as_float((127 - e) << 23);
    const DW g{t[0].hi * sc, t[0].lo * sc}, dl{t[1].hi * sc, t[1].lo * sc}, q{cg.q.hi * sc, cg.q.lo * sc};
    alpha = dw_div_fast(dw_mul(g, q), dw_add_sloppy(dw_mul(dl, q), dw_neg(dw_mul(g, g))));
    tb = dw_div_fast(t[0], cg.gamma).hi;
  }
  ta = alpha.hi;
  cg.gamma = t[0];
  cg.q = dw_mul(t[0], alpha);
  return CG_CONTINUE;
}
__device__ __forceinline__ int team_scalars(const double (&t)[3], bool first, CgState<double>& cg, double& ta,
                                            double& tb) {
  const int lane = threadIdx.x & 31;
  if (!isfinite(t[0]) || !isfinite(t[1]) || !isfinite(t[2])) return CG_NONFINITE;
  double alpha;
  bool lost = false;  // alpha is not positive (by the signs, beside the division)
  if (first) {
    alpha = t[0] / t[1];
    tb = 0.0;
  } else {
    cg.rr = t[2];
    if (t[2] <= cg.thr) return CG_DONE;
    // lane 0: gamma_k q / (delta_k q - gamma_k^2); lane 1: gamma_k / gamma_(k-1)
    const double n0 = t[0] * cg.q, d0 = fma(t[1], cg.q, -(t[0] * t[0]));
    const int hn = __double2hiint(n0), hd = __double2hiint(d0);
    lost = (hn ^ hd) < 0 || hn == 0 || hd == 0;
    const double num = lane == 1 ? t[0] : n0;
    const double den = lane == 1 ? cg.gamma : d0;
    const double quo = num / den;
    tb = __shfl_sync(0xffffffffu, quo, 1);
    alpha = __shfl_sync(0xffffffffu, quo, 0);
  }
  ta = alpha;
  cg.gamma = t[0];
  cg.q = t[0] * alpha;
  return lost ? CG_LOST : CG_CONTINUE;
}

// ------------------------------------------------------------- the solver
// FP32: a thread keeps R rows, row t + q rt of the part for q < R (rt =
// tm_row_threads, the threads that have rows).  FP64: a thread keeps one column
// of R rows, column t / rt of row t mod rt + q rt: an FP64 instruction occupies
// its scheduler for 64 cycles whatever its lanes, so a row's three columns go
// to three warps.  Threads beyond those help to read the halo and the slots.
//
// CL: the team is one thread-block cluster (a single robot of few parts).
//
// Matrix entries: with FP32 and R = 1 or with FP64 in registers, else in shared
// memory (columns as 16-bit indices into the halo).
template <typename T, int R, int NTMAX, bool CL>
__global__ void __launch_bounds__(NTMAX, 1) k_pcg_team(const __grid_constant__ Dev<T> d) {
  using A = typename DotAcc<T>::type;
  constexpr bool F32 = std::is_same<T, float>::value;
  constexpr int C = Cols<T>::N, PUBS = Cols<T>::PUBS;
  constexpr int MAXW = TEAM_MAX_WIDTH;
  constexpr int NWM = NTMAX / 32;
  constexpr bool REGS = !F32 || R == 1;  // matrix entries in registers
  constexpr int FETCH = 4;               // halo rows a thread has on their way at once
  constexpr int RV = REGS ? R : 1;
  // warp sums of the rows' and of the slots' dot products: (r.u, r.r, w.u),
  // in the first round (||b||^2, spring energy, ||r0||^2)
  __shared__ A s_row[3][32], s_slot[3][32];
  __shared__ float s_z[NWM][8 * C];          // warp sums of Z^T w, then Z^T r
  __shared__ float s_g[2][NWM][12];          // warp shares of g(w) and g(r)
  __shared__ __align__(16) float s_gr[NWM][12];  // g(r), a copy per warp
  __shared__ A c_dots[3][CL ? TEAM_CLUSTER : 1];    // CL: the parts' dot sums and coarse sums of this round
  __shared__ float c_z[CL ? 24 : 1][CL ? TEAM_CLUSTER : 1];
  __shared__ double s_es;
  __shared__ T s_ta, s_tb;
  __shared__ int s_flag, s_ok, s_lost;
  extern __shared__ __align__(16) unsigned char dyn[];
  const int t = threadIdx.x, nt = blockDim.x, lane = t & 31, wid = t >> 5;
  const bool w0 = wid == 0;
  const int n = d.n_free;
  const int rt = d.tm_row_threads;
  const int col = F32 ? 0 : t / rt;                     // FP64: this thread's column
  const int lt = F32 ? t : t - col * rt;                // its place among the rows' threads
  const bool rows_here = F32 ? t < rt : col < 3;        // warp-uniform: rt is a multiple of 32
  unsigned char* halo = dyn + (F32 ? 0 : (size_t)8 * d.tm_halo_max * min(col, 2));
  float* ainv = reinterpret_cast<float*>(dyn + d.tm_ainv_off);
  T* va_sh = reinterpret_cast<T*>(dyn + d.tm_val_off);
  unsigned short* lc_sh = reinterpret_cast<unsigned short*>(dyn + d.tm_lcol_off);
  const size_t ustride = (size_t)2 * PUBS * n;  // words of one parity buffer of u
  const double tol2 = F32 || !d.tm_coarse ? d.tol2 : d.tol2 * TEAM_STOP2_F64;

  for (int part = blockIdx.x; part < d.tm_parts; part += gridDim.x) {
    TeamCtx<T> c{d, d.tm_part[part], 0, 1};
    c.me = part - c.pt.p0;
    c.copies = c.pt.np > 32 ? TEAM_COPIES : 1;
    const int nrow = c.pt.nrow, row0 = c.pt.row0;
    const int nd = 4 * c.pt.np;  // coarse functions of the team
    __syncthreads();             // the previous part's shared state is free
    if (d.tm_coarse) {
      // the inverse for this solve's springs: the first level with sigma at
      // least 0.7 of theirs (the iteration counts hardly grow when sigma is too
      // large by a factor 4, by a third when it is too small by that)
      const int n_spr = d.tm_springs[c.pt.robot];
      const float sigma = 0.7f * (float)n_spr / (float)(d.robot_row[c.pt.robot + 1] - d.robot_row[c.pt.robot]);
      int lvl = n_spr > 0 && d.tm_levels > 1 ? 1 : 0;
      for (float v = TEAM_SIGMA_1; lvl > 0 && lvl < d.tm_levels - 1 && v < sigma; v *= 4.0f) ++lvl;
      const float4* src = reinterpret_cast<const float4*>(d.tm_ainv + (size_t)lvl * d.tm_ainv_level + c.pt.ainv);
      const bool stiff = n_spr > 0 && d.tm_stiff;  // zero: Jacobi alone (see make_dev)
      for (int k = t; k < nd; k += nt)
        reinterpret_cast<float4*>(ainv)[k] = stiff ? make_float4(0.0f, 0.0f, 0.0f, 0.0f) : src[k];
    }
    bool act[R];
    int width[R];
    T dg[R], idg[R];
    float4 z[R];
    T val[RV][REGS ? MAXW : 1];
    unsigned lc[RV][REGS ? MAXW / 2 : 1];
    T r[R][C], u[R][C], w[R][C], p[R][C], s[R][C], dd[R][C];
    A a0[3] = {acc_zero<A>(), acc_zero<A>(), acc_zero<A>()};
#pragma unroll
    for (int q = 0; q < R; ++q) {
      const int li = lt + q * rt, i = row0 + li;
      act[q] = rows_here && li < nrow;
      width[q] = 0;
      dg[q] = idg[q] = T(1);
      z[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll
      for (int k = 0; k < C; ++k) r[q][k] = u[q][k] = w[q][k] = p[q][k] = s[q][k] = dd[q][k] = T(0);
      if constexpr (REGS) {
#pragma unroll
        for (int j = 0; j < MAXW; ++j) val[q][j] = T(0);
#pragma unroll
        for (int j = 0; j < MAXW / 2; ++j) lc[q][j] = 0;
      }
      if (act[q]) {
        const int sl = i >> 5, base = d.sl_ptr[sl] + (i & 31);
        width[q] = (d.sl_ptr[sl + 1] - d.sl_ptr[sl]) >> 5;
        if constexpr (REGS) {
#pragma unroll
          for (int j = 0; j < MAXW; ++j)
            if (j < width[q]) {
              val[q][j] = d.sl_val[base + 32 * j];
              lc[q][j / 2] |= (unsigned)chk_idx(d.ctrl, d.tm_lcol[base + 32 * j], d.tm_halo_max) << (16 * (j & 1));
            }
        } else {
#pragma unroll 4
          for (int j = 0; j < width[q]; ++j) {
            va_sh[j * (R * rt) + li] = d.sl_val[base + 32 * j];
            lc_sh[j * (R * rt) + li] = (unsigned short)chk_idx(d.ctrl, d.tm_lcol[base + 32 * j], d.tm_halo_max);
          }
        }
        if (d.tm_coarse) z[q] = d.tm_z[i];
        team_row_start(d, i, col, dg[q], r[q], a0);
        idg[q] = T(1) / dg[q];
      }
    }
    const int n_oth = c.pt.n_other;
    const int* hrow = d.tm_halo + c.pt.halo0;
    // warp 0, lane 3 m + k (+ 12): the coarse sum of function m, column k of w
    // (of r) over the warps [z_q0, z_q1)
    const int z_h = lane >= 12, z_m = (lane - 12 * z_h) / 3, z_k = (lane - 12 * z_h) % 3;
    const int z_q0 = F32 ? 0 : z_k * (rt >> 5), z_q1 = z_q0 + (rt >> 5);
    const int z_at = F32 ? 12 * z_h + 3 * z_m + z_k : 4 * z_h + z_m;
    const int zwarps = F32 ? rt >> 5 : 3 * (rt >> 5);  // warps with rows
    // One pass of this loop is one round.  Pass -1 sums ||b||^2, ||r0||^2, the
    // spring energy and Z^T r0; pass 0 forms u_0 = M^-1 r0 and w_0; pass it > 0
    // is CG iteration it.  (One loop, so that every part of it exists once: the
    // code stays in the instruction cache and its state in registers.)
    const int part_len = d.tm_part[c.pt.p0].nrow;  // of every part but the last
    unsigned peer[CL ? FETCH : 1];                 // CL: where this thread's halo rows live
    auto peer_row = [&](int k) {
      const int cc = F32 ? 0 : k / n_oth, row = hrow[F32 ? k : k - cc * n_oth] - d.robot_row[c.pt.robot];
      const int rank = row / part_len, li = row - rank * part_len;
      return peer_addr(dyn + (F32 ? (size_t)16 * li : (size_t)8 * (d.tm_halo_max * cc + li)), rank);
    };
    if constexpr (CL) {
#pragma unroll
      for (int b = 0; b < FETCH; ++b) peer[b] = t + b * nt < PUBS * n_oth ? peer_row(t + b * nt) : 0;
      cluster_arrive();  // every block of the cluster is running
      cluster_wait();
    }
    CgState<A> cg{acc_zero<A>(), acc_zero<A>(), acc_zero<A>(), 0.0, 0.0};  // in warp 0
    T ta = T(0), tb = T(0);
    float gs = 0.0f, gr = 0.0f;  // lane l < 12 of every warp: g(s) and g(r)
    int it = -1, f = CG_CONTINUE;
    bool lost = false;  // a wait gave up
    for (;; ++it) {
      const unsigned e = (unsigned)it + 2u;  // epoch of this pass's u and round
      const bool coarse = it <= d.tm_coarse_last;
      A a[3];
      int which = 2;
      if (it < 0) {
#pragma unroll
        for (int k = 0; k < 3; ++k) a[k] = a0[k];
      } else {
        which = it > 0 && it % TEAM_REFRESH == 0 ? 3 : 1;
        a[0] = a[1] = a[2] = acc_zero<A>();
        unsigned long long* ubuf = d.tm_u + (size_t)(e & 1u) * ustride;
        const unsigned long long tag = tag_of(e);
        if (rows_here) {
          float gv[12];
#pragma unroll
          for (int k = 0; k < 12; ++k) gv[k] = 0.0f;
          if (coarse) {
#pragma unroll
            for (int k = 0; k < 3; ++k) {
              const float4 v = reinterpret_cast<const float4*>(s_gr[wid])[k];
              gv[4 * k] = v.x;
              gv[4 * k + 1] = v.y;
              gv[4 * k + 2] = v.z;
              gv[4 * k + 3] = v.w;
            }
          }
#pragma unroll
          for (int q = 0; q < R; ++q) {
            const float zz[4] = {z[q].x, z[q].y, z[q].z, z[q].w};
#pragma unroll
            for (int k = 0; k < C; ++k) {
              dd[q][k] += ta * p[q][k];
              r[q][k] -= ta * s[q][k];
              u[q][k] = r[q][k] * idg[q];
              if (coarse) {
                const int cc = F32 ? k : col;
                float g = 0.0f;
#pragma unroll
                for (int m = 0; m < 4; ++m)
                  g = __fmaf_rn(zz[m], F32 ? gv[3 * m + k] : (cc == 0 ? gv[3 * m] : cc == 1 ? gv[3 * m + 1] : gv[3 * m + 2]),
                                g);
                u[q][k] += (T)g;
              }
            }
            if (act[q]) {
              if constexpr (!CL) publish_u(ubuf + (size_t)2 * ((size_t)col * n + row0 + lt + q * rt), tag, u[q]);
              halo_put(halo, lt + q * rt, u[q]);
            }
          }
        }
        // the halo: own rows from registers (above), the other parts' rows as
        // they become current; r.u and r.r are summed while the first loads
        // are on their way
        const int n_fetch = PUBS * n_oth;
        auto at = [&](int k) {
          const int cc = F32 ? 0 : k / n_oth;
          return ubuf + (size_t)2 * ((size_t)cc * n + chk_idx(d.ctrl, hrow[F32 ? k : k - cc * n_oth], n));
        };
        auto put_v = [&](int k, const T(&v)[C]) {
          const int cc = F32 ? 0 : k / n_oth;
          halo_put(dyn + (F32 ? 0 : (size_t)8 * d.tm_halo_max * cc), nrow + (F32 ? k : k - cc * n_oth), v);
        };
        auto put = [&](int k, unsigned long long x, unsigned long long y) {
          T v[C];
          unpack_u(x, y, v);
          put_v(k, v);
        };
        unsigned long long fx[FETCH], fy[FETCH];
        if constexpr (CL) {
          cluster_arrive();  // own rows are in place
        } else {
#pragma unroll
          for (int b = 0; b < FETCH; ++b)
            if (t + b * nt < n_fetch) ld_v2_relaxed(at(t + b * nt), fx[b], fy[b]);
        }
        if (rows_here) {
#pragma unroll
          for (int q = 0; q < R; ++q) {
            a[0] = acc_add(a[0], dot_cols(r[q], u[q]));
            a[2] = acc_add(a[2], dot_cols(r[q], r[q]));
          }
          const A early[2] = {a[0], a[2]};
          store_sums<2>(early, 0, s_row);
        }
        if constexpr (CL) {
          cluster_wait();
          T v[FETCH][C];
#pragma unroll
          for (int b = 0; b < FETCH; ++b)
            if (t + b * nt < n_fetch) peer_load(peer[b], v[b]);
#pragma unroll
          for (int b = 0; b < FETCH; ++b)
            if (t + b * nt < n_fetch) put_v(t + b * nt, v[b]);
#pragma unroll 1
          for (int k = t + FETCH * nt; k < n_fetch; k += nt) {
            peer_load(peer_row(k), v[0]);
            put_v(k, v[0]);
          }
        } else {
        TeamWait wt;
#pragma unroll
        for (int b = 0; b < FETCH; ++b)
          if (t + b * nt < n_fetch) {
            while (!(has_tag(fx[b], tag) && has_tag(fy[b], tag)) && wt.again(d.ctrl, d.wait_budget))
              ld_v2_relaxed(at(t + b * nt), fx[b], fy[b]);
            put(t + b * nt, fx[b], fy[b]);
          }
#pragma unroll 1
        for (int k = t + FETCH * nt; k < n_fetch; k += nt) {
          unsigned long long x, y;
          do {
            ld_v2_relaxed(at(k), x, y);
          } while (!(has_tag(x, tag) && has_tag(y, tag)) && wt.again(d.ctrl, d.wait_budget));
          put(k, x, y);
        }
        // (a wait that gave up leaves the abort word raised: the waits that
        // follow give up at once and every block leaves)
        }
        __syncthreads();
        if (rows_here) {
#pragma unroll
          for (int q = 0; q < R; ++q) {
#pragma unroll
            for (int k = 0; k < C; ++k) w[q][k] = dg[q] * u[q][k];
            if constexpr (REGS) {
              T w2[C];
#pragma unroll
              for (int k = 0; k < C; ++k) w2[k] = T(0);
              // four entries at a time (entries beyond the row's width are
              // zeros at halo index 0): their loads go out together
#pragma unroll
              for (int j0 = 0; j0 < MAXW; j0 += 4)
                if (j0 < width[q]) {
#pragma unroll
                  for (int j = j0; j < j0 + 4; ++j) {
                    const int at = (lc[q][j / 2] >> (16 * (j & 1))) & 0xFFFFu;
                    if (!F32 && (j & 1))
                      halo_axpy(halo, at, val[q][j], w2);
                    else
                      halo_axpy(halo, at, val[q][j], w[q]);
                  }
                }
              if (!F32)
#pragma unroll
                for (int k = 0; k < C; ++k) w[q][k] += w2[k];
            } else {
#pragma unroll 4
              for (int j = 0; j < width[q]; ++j)
                halo_axpy(halo, lc_sh[j * (R * rt) + lt + q * rt], va_sh[j * (R * rt) + lt + q * rt], w[q]);
            }
            a[1] = acc_add(a[1], dot_cols(w[q], u[q]));
          }
        }
      }
      // ---- the round: the block's sums, its slot, the team's totals and g(w)
      // and g(r) (its barriers also let the halo be rewritten)
      if (rows_here) {
        if (coarse) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (!(which & (1 << h))) continue;
            float v[4 * C];
#pragma unroll
            for (int q = 0; q < R; ++q) {
              const float zz[4] = {z[q].x, z[q].y, z[q].z, z[q].w};
#pragma unroll
              for (int k = 0; k < 4 * C; ++k) {
                const float x = h ? (float)r[q][k % C] : (float)w[q][k % C];
                v[k] = q > 0 ? __fmaf_rn(zz[k / C], x, v[k]) : __fmul_rn(zz[k / C], x);
              }
            }
            warp_scatter_sum(v, &s_z[wid][4 * C * h]);
          }
        }
        if (it < 0) {
          const A early[2] = {a[0], a[2]};
          store_sums<2>(early, 0, s_row);
        }
        const A late[1] = {a[1]};
        store_sums<1>(late, 2, s_row);
      }
      __syncthreads();
      A dots = acc_zero<A>();
      if (w0) {
        dots = add_sums3(s_row, 0, zwarps);
        float sz = 0.0f;
        if (coarse && lane < 24 && (which >> (lane >= 12)) & 1) {
          sz = s_z[z_q0][z_at];
#pragma unroll 4
          for (int q = z_q0 + 1; q < z_q1; ++q) sz = __fadd_rn(sz, s_z[q][z_at]);
        }
        if constexpr (CL) {
          // lane l < 24: coarse sum l; lane 24 + k: dot sum k, to every block
          const unsigned long long db = __shfl_sync(0xffffffffu, bits64(dots), max(lane - 24, 0));
          for (int q = 0; q < c.pt.np; ++q) {
            if (lane < 24)
              peer_store(peer_addr(&c_z[lane][c.me], q), sz);
            else if (lane < 27)
              peer_store(peer_addr(&c_dots[lane - 24][c.me], q), db);
          }
        } else {
          const bool ok = team_publish(c, e, dots, coarse ? which : 0, sz);
          if (lane == 0) {
            s_ok = ok;
            s_lost = 0;
          }
        }
      }
      if constexpr (CL) {
        cluster_arrive();
        cluster_wait();
      } else {
        __syncthreads();
        lost = !s_ok;
        if (lost) break;
      }
      {
        // The team's totals and the shares of g(w) and g(r).  FP32: warp 0
        // adds the dot sums and forms the CG scalars while the next gw warps
        // read the coarse sums, one part per thread.  FP64: those warps read
        // the dot sums too (a warp's FP64 addition costs 64 cycles, so one
        // warp adding 150 slots would be the longest piece of the round), and
        // warp 0 adds the warps' sums.
        const int j = t - 32, gw = (c.pt.np + 31) >> 5;
        const int sel = coarse ? which : 0;
        bool ok = true;
        A tot = acc_zero<A>();
        if (wid >= 1 && wid <= gw) {
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            if (!(sel & (1 << h))) continue;
            float g[12];
#pragma unroll
            for (int k = 0; k < 12; ++k) g[k] = 0.0f;
            if constexpr (CL) {
              if (j < c.pt.np) {
                float x[4][3];
#pragma unroll
                for (int m = 0; m < 12; ++m) x[m / 3][m % 3] = c_z[12 * h + m][j];
                coarse_share(ainv, nd, j, x, g);
              }
            } else {
              if (j < c.pt.np) ok = team_read_coarse(c, e, h ? SLOT_R : SLOT_W, j, ainv, nd, g) && ok;
            }
            warp_scatter_sum(g, s_g[h][wid]);
          }
          if constexpr (!F32 && !CL) {
            A v[3] = {acc_zero<A>(), acc_zero<A>(), acc_zero<A>()};
            if (j < c.pt.np) ok = team_read_dots(c, e, j, v) && ok;
            store_sums<3>(v, 0, s_slot);
          }
          if (!ok) s_lost = 1;
        }
        if constexpr (!F32 && !CL) __syncthreads();
        if (w0) {
          A t0, t1, t2;
          if constexpr (F32 || CL) {
            if constexpr (CL) {
              A v[3];
#pragma unroll
              for (int k = 0; k < 3; ++k) v[k] = lane < c.pt.np ? c_dots[k][lane] : acc_zero<A>();
              tot = warp_sums<3>(v);
            } else {
              if (!team_dots(c, e, tot)) s_lost = 1;
            }
            tot = acc_norm(tot);
            t0 = shfl_at(tot, 0);
            t2 = shfl_at(tot, 8);
            t1 = shfl_at(tot, 16);
          } else {
            tot = add_sums3(s_slot, 1, gw + 1);
            t0 = shfl_at(tot, 0);
            t2 = shfl_at(tot, 1);
            t1 = shfl_at(tot, 2);
          }
          if (it < 0) {
            cg.bb = acc_to_f64(t0);
            cg.thr = tol2 * cg.bb;
            cg.rr = t1;
            if (t == 0) {
              s_es = acc_to_f64(t2);
              // a batch's energy is added up by the finalize launch: the
              // robot's in its first part's place
              if (d.n_robots > 1 && d.rhs_in_pcg) d.e_partials[d.n_e_local + part] = c.me == 0 ? s_es : 0.0;
            }
            f = (cg.bb > 0.0 && acc_to_f64(t1) > cg.thr) ? CG_CONTINUE : CG_DONE;
          } else {
            const A tot3[3] = {t0, t1, t2};
            f = team_scalars(tot3, it == 0 || it == d.tm_coarse_last + 1, cg, ta, tb);
            // An FP64 residual that falls by 1e5 or more in a few iterations is less
            // than the FP32 rounding that g has kept; the products with u then have any
            // sign.  Such a pass moves nothing, and the CG starts anew with the next
            // (there alpha is gamma / delta and beta 2^-60); g is formed anew before long.
            if constexpr (!F32)
              if (f == CG_LOST) {
                f = CG_CONTINUE;
                if (coarse) {
                  ta = tb = T(0);
                  cg.gamma = cg.q = 0x1p60 * t0;
                }
              }
          }
          if (f == CG_NONFINITE && c.me == 0 && t == 0) set_status(d.ctrl, ST_NONFINITE);
          if (t == 0) {
            s_ta = ta;
            s_tb = tb;
            s_flag = f;
          }
        }
        __syncthreads();
        if constexpr (!CL) {
          lost = s_lost;
          if (lost) break;
        }
        ta = s_ta;
        tb = s_tb;
        f = s_flag;
        auto shares = [&](const float(*g)[12]) {
          float x = 0.0f;
          if (lane < 12) {
            float y[TEAM_MAXQ];
#pragma unroll
            for (int q = 0; q < TEAM_MAXQ; ++q) y[q] = q < gw ? g[1 + q][lane] : 0.0f;
#pragma unroll
            for (int q = 0; q < TEAM_MAXQ; ++q) x = __fadd_rn(x, y[q]);
          }
          return x;
        };
        if (f != CG_CONTINUE) break;
        if (coarse) {
          if (which & 2) gr = shares(s_g[1]);
          if (it >= 0) {
            gs = shares(s_g[0]) + (float)tb * gs;  // g(s_k) = g(w_k) + beta_k g(s_k-1)
            gr -= (float)ta * gs;                  // g(r_k+1)
          }
          if (lane < 12) s_gr[wid][lane] = gr;
          __syncwarp();
        }
      }
      if (it == d.tm_cap) {
        if (c.me == 0 && t == 0) set_status(d.ctrl, ST_PCG_MAXIT);
        break;
      }
      if (it >= 0 && rows_here) {
#pragma unroll
        for (int q = 0; q < R; ++q)
#pragma unroll
          for (int k = 0; k < C; ++k) {
            p[q][k] = u[q][k] + tb * p[q][k];
            s[q][k] = w[q][k] + tb * s[q][k];
          }
      }
    }
    if (lost) {
      // the positions stay as they are; the iteration's record is closed all the
      // same (a batch's by the finalize launch)
      if (d.n_robots == 1 && d.rhs_in_pcg && c.me == 0 && t == 0) finalize_iteration(d, 0.0);
      return;
    }
    it = max(it, 0);
    if (it > 0 || d.xstep) {
#pragma unroll
      for (int q = 0; q < R; ++q)
        if (act[q]) {
          // x_(i+1) = start + correction (zero if the start already meets the
          // tolerance: that is where its residual was formed); the step x_(i+1) -
          // x_i is kept for the next outer iteration's start
          const int i = row0 + lt + q * rt;
          if constexpr (F32) {
            const R4<T> x0 = d.X[i];
            R4<T> x = warm_start(d, i, x0);
            x.x += dd[q][0];
            x.y += dd[q][1];
            x.z += dd[q][2];
            d.X[i] = x;
            if (d.xstep) d.xstep[i] = R4<T>{x.x - x0.x, x.y - x0.y, x.z - x0.z, T(0)};
          } else {
            reinterpret_cast<T*>(d.X)[4 * (size_t)i + col] += dd[q][0];
          }
        }
    }
    if (c.me == 0) {
      // the robot's solve into the record of this outer iteration; with one
      // robot also what a finalize launch would do: the Eq. 8 energy (the
      // local step's partials in a fixed order plus the spring energy of the
      // first round), the iteration count, the per-iteration words reset
      if (d.n_robots > 1) {
        if (t == 0) {
          IterRec* rec = d.hist + (d.ctrl->iter % d.hist_cap);
          atomicMax(&rec->pcg_iters, it);
          atomicAdd(reinterpret_cast<unsigned long long*>(&d.ctrl->total_pcg), (unsigned long long)it);
          const double rel = cg.bb > 0.0 ? sqrt(acc_to_f64(cg.rr) / cg.bb) : 0.0;
          atomicMax(reinterpret_cast<unsigned long long*>(&rec->pcg_rel_residual),
                    (unsigned long long)__double_as_longlong(rel));
        }
      } else {
        __shared__ double s_e[32];
        double el = 0.0;
        if (d.rhs_in_pcg && d.stats)
          for (int k = t; k < d.n_e_local; k += nt) el += d.e_partials[k];
        const double en = block_sum(el, s_e);
        if (t == 0) {
          write_pcg_record(d.ctrl, d.hist, d.hist_cap, d.ctrl, it, acc_to_f64(cg.rr), cg.bb);
          if (d.rhs_in_pcg) finalize_iteration(d, d.stats ? en + s_es : 0.0);
        }
      }
    }
  }
}

// ---------------------------------------------- inverse of the coarse matrices
// In-place inverse of SPD matrices (row-major FP64, one per robot) by blocked
// Gauss-Jordan elimination without pivoting: for every 32-wide pivot block,
// its inverse D, the pivot rows D A_k*, the rank-32 update of all other rows,
// and the pivot column -A_*k D.  On the device because the coarse matrix of a
// large robot has up to 640 rows (4 TEAM_MAX_PARTS): 2 n^3 operations for each
// robot and level.
static constexpr int GJ = 32;

__device__ __forceinline__ double* gj_mat(double* A, const long long* off, const int* dim, int r, int& n) {
  n = dim[r];
  return A + off[r];
}

__global__ void __launch_bounds__(GJ* GJ) k_gj_pivot(double* A, const long long* off, const int* dim, int kb, double* D,
                                                     int* bad) {
  __shared__ double m[GJ][GJ + 1];
  int n;
  double* a = gj_mat(A, off, dim, blockIdx.x, n);
  const int k0 = kb * GJ;
  if (k0 >= n) return;
  const int i = threadIdx.y, j = threadIdx.x, nb = min(GJ, n - k0);
  m[i][j] = (i < nb && j < nb) ? a[(size_t)(k0 + i) * n + k0 + j] : (i == j ? 1.0 : 0.0);
  __syncthreads();
  for (int k = 0; k < GJ; ++k) {
    const double piv = m[k][k], ik = m[i][k], kj = m[k][j], ij = m[i][j];
    __syncthreads();
    if (!(piv > 0.0) && i == 0 && j == 0) bad[blockIdx.x] = 1;
    const double q = 1.0 / piv;
    double v;
    if (i == k && j == k)
      v = q;
    else if (i == k)
      v = kj * q;
    else if (j == k)
      v = -ik * q;
    else
      v = ij - ik * (kj * q);
    m[i][j] = v;
    __syncthreads();
  }
  D[((size_t)blockIdx.x * GJ + i) * GJ + j] = m[i][j];
}

// the old pivot column into C, the pivot rows D A_k* into place
__global__ void __launch_bounds__(GJ* GJ) k_gj_row(double* A, const long long* off, const int* dim, int kb,
                                                   const double* D, double* C, int cmax) {
  __shared__ double sd[GJ][GJ + 1], sa[GJ][GJ + 1];
  int n;
  const int r = blockIdx.y;
  double* a = gj_mat(A, off, dim, r, n);
  const int k0 = kb * GJ, j0 = blockIdx.x * GJ;
  if (k0 >= n || j0 >= n) return;
  const int i = threadIdx.y, j = threadIdx.x, nb = min(GJ, n - k0);
  // column panel rows j0.. (old values), transposed use below
  double* c = C + (size_t)r * cmax * GJ;
  if (j0 + i < n) c[(size_t)(j0 + i) * GJ + j] = j < nb ? a[(size_t)(j0 + i) * n + k0 + j] : 0.0;
  if (blockIdx.x == kb) return;
  sd[i][j] = D[((size_t)r * GJ + i) * GJ + j];
  sa[i][j] = (i < nb && j0 + j < n) ? a[(size_t)(k0 + i) * n + j0 + j] : 0.0;
  __syncthreads();
  double v = 0.0;
  for (int k = 0; k < GJ; ++k) v = fma(sd[i][k], sa[k][j], v);
  if (i < nb && j0 + j < n) a[(size_t)(k0 + i) * n + j0 + j] = v;
}

__global__ void __launch_bounds__(256) k_gj_update(double* A, const long long* off, const int* dim, int kb,
                                                   const double* D, const double* C, int cmax) {
  __shared__ double sc[2 * GJ][GJ + 1], sb[GJ][2 * GJ + 1];
  int n;
  const int r = blockIdx.z;
  double* a = gj_mat(A, off, dim, r, n);
  const int k0 = kb * GJ, i0 = blockIdx.y * 2 * GJ, j0 = blockIdx.x * 2 * GJ;
  if (k0 >= n || i0 >= n || j0 >= n) return;
  const int nb = min(GJ, n - k0);
  const double* c = C + (size_t)r * cmax * GJ;
  for (int q = threadIdx.x; q < 2 * GJ * GJ; q += 256) {
    const int ii = q / GJ, kk = q % GJ;
    sc[ii][kk] = i0 + ii < n ? c[(size_t)(i0 + ii) * GJ + kk] : 0.0;
    const int k2 = q / (2 * GJ), jj = q % (2 * GJ), gj = j0 + jj;
    double v = 0.0;
    if (gj < n && k2 < nb)
      v = (gj >= k0 && gj < k0 + nb) ? D[((size_t)r * GJ + k2) * GJ + gj - k0] : a[(size_t)(k0 + k2) * n + gj];
    sb[k2][jj] = v;
  }
  __syncthreads();
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  double v[4][4] = {};
  for (int k = 0; k < GJ; ++k) {
    double x[4], y[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      x[q] = sc[ty + 16 * q][k];
      y[q] = sb[k][tx + 16 * q];
    }
#pragma unroll
    for (int p = 0; p < 4; ++p)
#pragma unroll
      for (int q = 0; q < 4; ++q) v[p][q] = fma(x[p], y[q], v[p][q]);
  }
#pragma unroll
  for (int p = 0; p < 4; ++p)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int gi = i0 + ty + 16 * p, gj = j0 + tx + 16 * q;
      if (gi >= n || gj >= n) continue;
      const bool prow = gi >= k0 && gi < k0 + nb, pcol = gj >= k0 && gj < k0 + nb;
      double* o = a + (size_t)gi * n + gj;
      if (prow && pcol)
        *o = D[((size_t)r * GJ + gi - k0) * GJ + gj - k0];
      else if (!prow)
        *o = pcol ? -v[p][q] : *o - v[p][q];
    }
}

// the inverse in FP32, symmetrised
__global__ void k_gj_float(const double* A, const long long* off, const int* dim, float* out, int* bad) {
  const int r = blockIdx.y;
  const long long n = dim[r];
  const double* a = A + off[r];
  for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n * n; q += (long long)gridDim.x * blockDim.x) {
    const long long i = q / n, j = q - i * n;
    const double v = 0.5 * (a[i * n + j] + a[j * n + i]);
    if (!isfinite(v)) bad[r] = 1;
    out[off[r] + q] = (float)v;
  }
}

__global__ void k_shift(double* A, const long long* off, const int* dim, double sigma) {
  const long long n = dim[blockIdx.y];
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i < n) A[off[blockIdx.y] + i * (n + 1)] += sigma;
}

// Largest absolute row sums (one warp to a row) into norm[r], which is zero before.
__global__ void __launch_bounds__(256) k_matrix_norm(const double* A, const long long* off, const int* dim, double* norm) {
  const int r = blockIdx.y, n = dim[r], i = blockIdx.x * 8 + (threadIdx.x >> 5);
  if (i >= n) return;
  double s = 0.0;
  for (int j = threadIdx.x & 31; j < n; j += 32) s += fabs(A[off[r] + (long long)i * n + j]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  // (non-negative doubles order like their bits; a NaN ends above them)
  if ((threadIdx.x & 31) == 0) atomicMax(reinterpret_cast<unsigned long long*>(norm + r), bits64(s));
}

// Calls f(first, count) for n_mat matrices (a batch has TEAM_LEVELS a robot) in
// slices that fit a grid's y and z dimensions.
template <typename F>
static void for_slices(int n_mat, F f) {
  for (int s = 0; s < n_mat; s += INVERT_SLICE) f(s, std::min(INVERT_SLICE, n_mat - s));
}

void launch_shift(double* A, const long long* off, const int* dim, int n_mat, double sigma, cudaStream_t st) {
  for_slices(n_mat, [&](int s, int m) {
    k_shift<<<dim3((4 * TEAM_MAX_PARTS + 255) / 256, m), 256, 0, st>>>(A, off + s, dim + s, sigma);
  });
}

void launch_matrix_norm(const double* A, const long long* off, const int* dim, int n_mat, int max_dim, double* norm,
                        cudaStream_t st) {
  for_slices(n_mat, [&](int s, int m) {
    if (max_dim > 0) k_matrix_norm<<<dim3((max_dim + 7) / 8, m), 256, 0, st>>>(A, off + s, dim + s, norm + s);
  });
}

// Inverts n_mat matrices at A + off[r] (dim[r] rows, at most max_dim) into out
// (same offsets).  C holds m x max_dim x 32 doubles, D m x 32 x 32 for m matrices,
// n_mat or INVERT_SLICE if that is less;
// bad[r] becomes 1 for a matrix that is not positive definite.
void launch_invert(double* A, const long long* off, const int* dim, int n_mat, int max_dim, double* C, double* D,
                   float* out, int* bad, cudaStream_t st) {
  const int nk = (max_dim + GJ - 1) / GJ, nt = (max_dim + 2 * GJ - 1) / (2 * GJ);
  for_slices(n_mat, [&](int s, int m) {
    const long long* o = off + s;
    const int* n = dim + s;
    for (int kb = 0; kb < nk; ++kb) {
      k_gj_pivot<<<m, dim3(GJ, GJ), 0, st>>>(A, o, n, kb, D, bad + s);
      k_gj_row<<<dim3(nk, m), dim3(GJ, GJ), 0, st>>>(A, o, n, kb, D, C, max_dim);
      k_gj_update<<<dim3(nt, nt, m), 256, 0, st>>>(A, o, n, kb, D, C, max_dim);
    }
    k_gj_float<<<dim3(std::min(((max_dim * max_dim) + 255) / 256, 1024), m), 256, 0, st>>>(A, o, n, out, bad + s);
  });
}

// ---------------------------------------------------------------- launchers
template <typename T>
void launch_team_rhs(const Dev<T>& d, cudaStream_t st) {
  if (d.n_free == 0) return;
  if constexpr (std::is_same<T, float>::value)
    k_team_rhs_f32<<<(d.n_free + 255) / 256, 256, 0, st>>>(d);
  else
    k_team_rhs_f64<<<(3 * d.n_free + 127) / 128, 128, 0, st>>>(d);
}

// Words that every solve finds at zero: the tagged words of u, the slots and
// the teams' counters (one allocation, tm_u first).
template <typename T>
cudaError_t launch_team_clear(const Dev<T>& d, cudaStream_t st) {
  return cudaMemsetAsync(d.tm_u, 0, d.tm_zero_bytes, st);
}

size_t team_words(bool fp64, int n_free, int parts, int robots, size_t& slot_off, size_t& count_off) {
  const size_t u = (size_t)2 * n_free * (fp64 ? 6 : 2);
  const size_t slot = (size_t)TEAM_COPIES * 2 * parts * SLOT_WORDS;
  slot_off = (u + 1) & ~size_t(1);
  count_off = slot_off + slot;
  return count_off + (size_t)16 * TEAM_COPIES * robots;  // counters 128 bytes apart
}

size_t team_smem(bool fp64, int rows, int r, int halo_max, int max_np, bool coarse, int max_width,
                 int& ainv_off, int& val_off, int& lcol_off) {
  size_t s = (halo_bytes(fp64, halo_max) + 15) & ~size_t(15);
  ainv_off = (int)s;
  if (coarse) s += sizeof(float) * 16 * (size_t)max_np;
  const bool regs = fp64 || r == 1;
  val_off = (int)s;
  if (!regs) s += sizeof(float) * max_width * rows;
  lcol_off = (int)s;
  if (!regs) s += sizeof(unsigned short) * max_width * rows;
  return s;
}

// The instance for a plan: FP64 with 1, 2 or 3 rows per thread, FP32 with 1 or
// 3, in one cluster with 1.
template <typename F>
static auto with_team_kernel(bool fp64, int r, bool cluster, F f) {
  if (fp64) {
    if (cluster) return f(k_pcg_team<double, 1, TEAM_NT_F64, true>);
    if (r == 1) return f(k_pcg_team<double, 1, TEAM_NT_F64, false>);
    if (r == 2) return f(k_pcg_team<double, 2, TEAM_NT_F64, false>);
    return f(k_pcg_team<double, 3, TEAM_NT_F64, false>);
  }
  if (cluster) return f(k_pcg_team<float, 1, TEAM_NT_1, true>);
  if (r == 1) return f(k_pcg_team<float, 1, TEAM_NT_1, false>);
  return f(k_pcg_team<float, 3, TEAM_NT_3, false>);
}

static cudaLaunchConfig_t team_config(int grid, int threads, size_t smem, bool cluster, cudaLaunchAttribute* attr,
                                      cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  if (cluster) {
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = grid;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
  } else {
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
  }
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cfg;
}

// Raises the kernel's shared-memory limit (and allows its cluster size); false
// when it cannot be resident.  The limit belongs to the kernel and every handle's
// launches share it: always the same, so that no upload lowers another's.
bool team_prepare(bool fp64, int r, bool cluster, int grid, int threads, size_t smem) {
  const bool ok = with_team_kernel(fp64, r, cluster, [&](auto k) {
    int n = 0;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TEAM_SMEM_MAX) != cudaSuccess) return false;
    if (!cluster)
      return cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, k, threads, smem) == cudaSuccess && n >= 1;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess) return false;
    cudaLaunchAttribute attr[1];
    const cudaLaunchConfig_t cfg = team_config(grid, threads, smem, true, attr, nullptr);
    return cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n >= 1;
  });
  if (!ok) cudaGetLastError();
  return ok;
}

template <typename T>
cudaError_t launch_pcg_team(const Dev<T>& d, cudaStream_t st) {
  if (d.n_free == 0) return cudaSuccess;
  cudaLaunchAttribute attr[1];
  const cudaLaunchConfig_t cfg = team_config(d.tm_grid, d.tm_threads, d.tm_smem, d.tm_cluster, attr, st);
  if constexpr (std::is_same<T, float>::value) {
    if (d.tm_cluster) return cudaLaunchKernelEx(&cfg, k_pcg_team<float, 1, TEAM_NT_1, true>, d);
    return d.tm_r_per == 1 ? cudaLaunchKernelEx(&cfg, k_pcg_team<float, 1, TEAM_NT_1, false>, d)
                           : cudaLaunchKernelEx(&cfg, k_pcg_team<float, 3, TEAM_NT_3, false>, d);
  } else {
    if (d.tm_cluster) return cudaLaunchKernelEx(&cfg, k_pcg_team<double, 1, TEAM_NT_F64, true>, d);
    return d.tm_r_per == 1   ? cudaLaunchKernelEx(&cfg, k_pcg_team<double, 1, TEAM_NT_F64, false>, d)
           : d.tm_r_per == 2 ? cudaLaunchKernelEx(&cfg, k_pcg_team<double, 2, TEAM_NT_F64, false>, d)
                             : cudaLaunchKernelEx(&cfg, k_pcg_team<double, 3, TEAM_NT_F64, false>, d);
  }
}

template void launch_team_rhs<float>(const Dev<float>&, cudaStream_t);
template void launch_team_rhs<double>(const Dev<double>&, cudaStream_t);
template cudaError_t launch_team_clear<float>(const Dev<float>&, cudaStream_t);
template cudaError_t launch_team_clear<double>(const Dev<double>&, cudaStream_t);
template cudaError_t launch_pcg_team<float>(const Dev<float>&, cudaStream_t);
template cudaError_t launch_pcg_team<double>(const Dev<double>&, cudaStream_t);

}  // namespace casim
