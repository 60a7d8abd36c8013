// Collision check (Sec. II-B, Eq. 3, Eq. 4) and spring update (Sec. II-C,
// Eq. 5, Sec. III-A.3) kernels.
//
// Broad phase: a spatial hash of the query vertices (lists) and one of the
// boundary faces (counting sort), rebuilt every iteration from the current
// positions.  A point strictly inside a tet lies in the tet's closed bounding
// box, whose cell range covers the point's cell, so a walk over the cells of
// every tet's box meets every pair.
//
// Narrow phase: one thread per tet tests the vertices listed in its cells with
// exact orientation signs (predicates.cuh), so the pair set equals the
// brute-force definition bit for bit.
//
// Spring update: one thread per non-fixed boundary vertex for obstacle
// targets (closed form) and the paper's release condition; self-collision
// targets by a ray cast along -n(v) (3D-DDA cell walk of Amanatides and Woo
// 1987 over the face hash, Moller-Trumbore 1997 ray-triangle test), eight
// lanes per casting vertex.  All spring geometry is evaluated in FP64.
#include <algorithm>

#include "bvh.cuh"
#include "common.cuh"
#include "kernels.h"
#include "predicates.cuh"

namespace casim {

static constexpr int MAX_CELLS_PER_ITEM = 4096;
static constexpr int MAX_DDA_STEPS = 4096;

template <typename T>
__device__ __forceinline__ void load3(const R4<T>* X, int v, double& x, double& y, double& z) {
  const R4<T> a = X[v];
  x = (double)a.x;
  y = (double)a.y;
  z = (double)a.z;
}

// Bounding box of up to four corners in the positions' own precision; false if
// one is not finite.
template <typename T, int NV>
__device__ __forceinline__ bool corner_box(const R4<T> (&c)[NV], T lo[3], T hi[3]) {
  bool ok = true;
  lo[0] = hi[0] = c[0].x;
  lo[1] = hi[1] = c[0].y;
  lo[2] = hi[2] = c[0].z;
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const T a[3] = {c[k].x, c[k].y, c[k].z};
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      ok = ok && isfinite(a[j]);
      if (k == 0) continue;
      lo[j] = fmin(lo[j], a[j]);
      hi[j] = fmax(hi[j], a[j]);
    }
  }
  return ok;
}

// Cell coordinate in FP32 for FP32 positions, used for the tets and for the
// narrow phase's point lookups only: it is monotone in x, so the cells of a
// tet's box corners bound the cell of every point in the box, the property
// the point-in-tet search needs.  The boundary faces keep FP64 cells
// (cell_coord), the model of the ray walk and of the shell search.
__device__ __forceinline__ int cell_coord_f(float x, float inv_cell) {
  float c = floorf(x * inv_cell);
  c = fminf(fmaxf(c, -1.0e6f), 1.0e6f);
  return (int)c;
}

// Block-reduced bounding box of the valid item boxes (count pass only).
// Warps without a valid item skip the shuffles, and blocks without one skip
// the atomics (only the boundary faces' blocks contribute).
__device__ __forceinline__ void reduce_box(Ctrl* c, bool valid, const double lo[3], const double hi[3]) {
  __shared__ long long s_lo[3][8], s_hi[3][8];
  constexpr long long kLo = 0x7FFFFFFFFFFFFFFFLL, kHi = (long long)0x8000000000000000ULL;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const bool any = __any_sync(0xffffffffu, valid);
  for (int j = 0; j < 3; ++j) {
    long long a = kLo, b = kHi;
    if (any) {
      a = valid ? order_code(lo[j]) : kLo;
      b = valid ? order_code(hi[j]) : kHi;
      for (int o = 16; o > 0; o >>= 1) {
        a = min(a, __shfl_down_sync(0xffffffffu, a, o));
        b = max(b, __shfl_down_sync(0xffffffffu, b, o));
      }
    }
    if (lane == 0) {
      s_lo[j][wid] = a;
      s_hi[j][wid] = b;
    }
  }
  __syncthreads();
  if (threadIdx.x < 3) {
    const int j = threadIdx.x;
    long long a = s_lo[j][0], b = s_hi[j][0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
      a = min(a, s_lo[j][w]);
      b = max(b, s_hi[j][w]);
    }
    if (a != kLo) atomicMin(&c->box_lo[j], a);
    if (b != kHi) atomicMax(&c->box_hi[j], b);
  }
}

// Adds one block's number of hash entries to the iteration's total; a total
// above the declared capacity is an overflow.
template <typename T>
__device__ __forceinline__ void add_entries(const Dev<T>& d, unsigned long long n) {
  if (n == 0) return;
  if (atomicAdd(d.entries, n) + n > (unsigned long long)d.cap_items) set_status(d.ctrl, ST_OVERFLOW);
}

// ---- hash of the boundary faces: count, place the cells, fill ----
static constexpr int FACE_THREADS = 256;

template <typename T, bool FILL>
__global__ void __launch_bounds__(FACE_THREADS) k_faces(Dev<T> d) {
  const int f = blockIdx.x * FACE_THREADS + threadIdx.x;
  T lo[3] = {0, 0, 0}, hi[3] = {0, 0, 0};
  bool ok = false;
  if (f < d.n_f) {
    const int4 fv = chk_face(d.ctrl, d.faces[f], d.n_v);
    const R4<T> c[3] = {d.X[fv.x], d.X[fv.y], d.X[fv.z]};
    ok = corner_box<T, 3>(c, lo, hi);
  }
  // (converted exactly)
  const double lod[3] = {(double)lo[0], (double)lo[1], (double)lo[2]},
               hid[3] = {(double)hi[0], (double)hi[1], (double)hi[2]};
  // the box of the boundary faces bounds the ray walks (no face lies beyond it)
  if (!FILL) reduce_box(d.ctrl, ok, lod, hid);
  if (f >= d.n_f) return;
  if (!ok) {
    if (!FILL) set_status(d.ctrl, ST_NONFINITE);
    return;
  }
  int c0[3], c1[3];
  for (int j = 0; j < 3; ++j) {
    c0[j] = cell_coord(lod[j], d.inv_cell);
    c1[j] = cell_coord(hid[j], d.inv_cell);
  }
  const long long ncell =
      (long long)(c1[0] - c0[0] + 1) * (c1[1] - c0[1] + 1) * (c1[2] - c0[2] + 1);
  if (ncell > MAX_CELLS_PER_ITEM) {
    if (!FILL) set_status(d.ctrl, ST_OVERFLOW);
    return;
  }
  const int robot = d.robot_of_face ? d.robot_of_face[f] : 0;
  for (int cz = c0[2]; cz <= c1[2]; ++cz)
    for (int cy = c0[1]; cy <= c1[1]; ++cy)
      for (int cx = c0[0]; cx <= c1[0]; ++cx) {
        const unsigned h = hash_cell(cx, cy, cz, robot) & (d.H_f - 1u);
        if (!FILL) {
          atomicAdd(&d.cell_count[h], 1);
        } else {
          const int pos = atomicAdd(&d.cell_range[h].y, 1);
          if (pos < d.cap_items) d.items[pos] = f;
        }
      }
}

// ---- exclusive scan (three small kernels) ----
static constexpr int SCAN_THREADS = 256;
static constexpr int SCAN_PER_THREAD = 8;
static constexpr int SCAN_TILE = SCAN_THREADS * SCAN_PER_THREAD;

__global__ void k_scan_tiles(const int* __restrict__ in, int* __restrict__ out, int* __restrict__ tile_sums,
                             int n) {
  __shared__ int sh[SCAN_THREADS];
  const int base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_PER_THREAD;
  int v[SCAN_PER_THREAD];
  int s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_PER_THREAD; ++k) {
    v[k] = (base + k < n) ? in[base + k] : 0;
    s += v[k];
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int off = 1; off < SCAN_THREADS; off <<= 1) {
    int t = (threadIdx.x >= off) ? sh[threadIdx.x - off] : 0;
    __syncthreads();
    sh[threadIdx.x] += t;
    __syncthreads();
  }
  int run = sh[threadIdx.x] - s;  // exclusive prefix of this thread
#pragma unroll
  for (int k = 0; k < SCAN_PER_THREAD; ++k) {
    if (base + k < n) out[base + k] = run;
    run += v[k];
  }
  if (threadIdx.x == SCAN_THREADS - 1) tile_sums[blockIdx.x] = sh[threadIdx.x];
}

// Single block: exclusive scan of the tile sums in place, total into *total.
__global__ void k_scan_top(int* tile_sums, int n_tiles, int* total_out) {
  __shared__ int sh[1024];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < n_tiles; base += 1024) {
    const int i = base + threadIdx.x;
    const int v = (i < n_tiles) ? tile_sums[i] : 0;
    sh[threadIdx.x] = v;
    __syncthreads();
    for (int off = 1; off < 1024; off <<= 1) {
      int t = (threadIdx.x >= off) ? sh[threadIdx.x - off] : 0;
      __syncthreads();
      sh[threadIdx.x] += t;
      __syncthreads();
    }
    if (i < n_tiles) tile_sums[i] = carry + sh[threadIdx.x] - v;
    __syncthreads();
    if (threadIdx.x == 1023) carry += sh[1023];
    __syncthreads();
  }
  if (threadIdx.x == 0) *total_out = carry;
}

__global__ void k_scan_add(int* out, const int* tile_sums, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] += tile_sums[i / SCAN_TILE];
}

// Places the face cells in the item array, (start, start) for each: the cells
// only need disjoint ranges, in whatever order, so a block takes the range of
// its tile with one addition to a global counter instead of waiting for the
// tiles before it, and the fill moves the end.
template <typename T>
__global__ void __launch_bounds__(SCAN_THREADS) k_place_cells(Dev<T> d) {
  __shared__ int s_warp[SCAN_THREADS / 32], s_base;
  const int base = blockIdx.x * SCAN_TILE + threadIdx.x * SCAN_PER_THREAD, n = (int)d.H_f;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int v[SCAN_PER_THREAD];
  int s = 0;
#pragma unroll
  for (int k = 0; k < SCAN_PER_THREAD; ++k) {
    v[k] = (base + k < n) ? d.cell_count[base + k] : 0;
    s += v[k];
  }
  int incl = s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) s_warp[wid] = incl;
  __syncthreads();
  int before = 0, total = 0;
#pragma unroll
  for (int w = 0; w < SCAN_THREADS / 32; ++w) {
    if (w < wid) before += s_warp[w];
    total += s_warp[w];
  }
  if (threadIdx.x == 0) {
    s_base = total ? atomicAdd(d.cell_total, total) : 0;
    add_entries(d, (unsigned long long)total);
  }
  __syncthreads();
  int run = s_base + before + incl - s;
#pragma unroll
  for (int k = 0; k < SCAN_PER_THREAD; ++k) {
    if (base + k < n) d.cell_range[base + k] = make_int2(run, run);
    run += v[k];
  }
}

// ---- narrow phase ----
__device__ __forceinline__ int orient_t(float ax, float ay, float az, float bx, float by, float bz, float cx, float cy,
                                        float cz, float dx, float dy, float dz) {
  return orient_sign_f(ax, ay, az, bx, by, bz, cx, cy, cz, dx, dy, dz);
}
__device__ __forceinline__ int orient_t(double ax, double ay, double az, double bx, double by, double bz, double cx,
                                        double cy, double cz, double dx, double dy, double dz) {
  return orient_sign(ax, ay, az, bx, by, bz, cx, cy, cz, dx, dy, dz);
}

template <typename T>
__device__ __forceinline__ T min4(T a, T b, T c, T e) {
  return fmin(fmin(a, b), fmin(c, e));
}
template <typename T>
__device__ __forceinline__ T max4(T a, T b, T c, T e) {
  return fmax(fmax(a, b), fmax(c, e));
}

// p strictly inside tet t, evaluated in the positions' own precision (the
// box reject compares exactly; the orientation signs are exact).
template <typename T>
__device__ __forceinline__ bool strictly_inside_at(const R4<T>* X, T px, T py, T pz, int4 t) {
  const R4<T> a = X[t.x], b = X[t.y], c = X[t.z], e = X[t.w];
  // A point strictly inside a tet lies strictly inside its box: the tet
  // reaches its extreme coordinates only on its boundary.  The open box test
  // is exact and rejects the many points on a box face (vertices of
  // axis-aligned meshes), whose orientation signs would be exact zeros.
  if (!(px > min4(a.x, b.x, c.x, e.x) && px < max4(a.x, b.x, c.x, e.x))) return false;
  if (!(py > min4(a.y, b.y, c.y, e.y) && py < max4(a.y, b.y, c.y, e.y))) return false;
  if (!(pz > min4(a.z, b.z, c.z, e.z) && pz < max4(a.z, b.z, c.z, e.z))) return false;
  // p strictly inside iff each sub-tet with one vertex replaced by p is
  // positive; for FP32 positions every sign first gets the FP32 filter, so a
  // certified negative sign ends the test before any FP64 or exact work
  if constexpr (std::is_same<T, float>::value) {
    const int s0 = orient_filter_f(px, py, pz, b.x, b.y, b.z, c.x, c.y, c.z, e.x, e.y, e.z);
    const int s1 = orient_filter_f(a.x, a.y, a.z, px, py, pz, c.x, c.y, c.z, e.x, e.y, e.z);
    const int s2 = orient_filter_f(a.x, a.y, a.z, b.x, b.y, b.z, px, py, pz, e.x, e.y, e.z);
    const int s3 = orient_filter_f(a.x, a.y, a.z, b.x, b.y, b.z, c.x, c.y, c.z, px, py, pz);
    if (s0 < 0 || s1 < 0 || s2 < 0 || s3 < 0) return false;
  }
  if (orient_t(px, py, pz, b.x, b.y, b.z, c.x, c.y, c.z, e.x, e.y, e.z) <= 0) return false;
  if (orient_t(a.x, a.y, a.z, px, py, pz, c.x, c.y, c.z, e.x, e.y, e.z) <= 0) return false;
  if (orient_t(a.x, a.y, a.z, b.x, b.y, b.z, px, py, pz, e.x, e.y, e.z) <= 0) return false;
  if (orient_t(a.x, a.y, a.z, b.x, b.y, b.z, c.x, c.y, c.z, px, py, pz) <= 0) return false;
  return true;
}
// The same behind a call: where it is rare, its registers stay out of the caller.
template <typename T>
__device__ __noinline__ bool strictly_inside_call(const R4<T>* X, T px, T py, T pz, int4 t) {
  return strictly_inside_at(X, px, py, pz, t);
}

// Obstacle tests of one query point (Eq. 4): the sphere whose signed surface
// distance |x - c_j| - r_j is smallest among those strictly containing it
// (ties: lowest j), how many spheres contain it, and how many tetrahedra of
// the rigid tetrahedral obstacle strictly contain it (exact signs, AABB tree
// of the obstacle).  Spheres use the fixed FP64 evaluation order.
template <typename T>
__device__ __forceinline__ void sphere_tests(const Dev<T>& d, T px, T py, T pz, int& best, int& n_sph) {
  best = -1;
  n_sph = 0;
  if (d.collision < 2) return;
  double bestd = 0.0;
  for (int j = 0; j < d.n_spheres; ++j) {
    // FP32 reject first: a point farther than r from the centre along one axis
    // is outside; the margins (1e-5 relative to the magnitudes involved) cover
    // the FP32 rounding of the centre, the radius and the difference, so only
    // points near the sphere reach the FP64 test (on this part an FP64
    // instruction costs about as much in one lane as in thirty-two)
    {
      const float rf = d.spheres_f[4 * j + 3];
      const float cf[3] = {d.spheres_f[4 * j], d.spheres_f[4 * j + 1], d.spheres_f[4 * j + 2]};
      const float pf[3] = {(float)px, (float)py, (float)pz};
      bool far = false;
#pragma unroll
      for (int k = 0; k < 3; ++k)
        far |= fabsf(pf[k] - cf[k]) > rf * 1.00001f + 1e-5f * (fabsf(cf[k]) + fabsf(pf[k]));
      if (far) continue;
    }
    const double cx = d.spheres[4 * j], cy = d.spheres[4 * j + 1], cz = d.spheres[4 * j + 2];
    const double r = d.spheres[4 * j + 3];
    const double dx = __dsub_rn((double)px, cx), dy = __dsub_rn((double)py, cy), dz = __dsub_rn((double)pz, cz);
    const double d2 = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
    if (d2 < __dmul_rn(r, r)) {
      ++n_sph;
      const double dist = sqrt(d2) - r;
      if (best < 0 || dist < bestd) {
        best = j;
        bestd = dist;
      }
    }
  }
}
template <typename T>
__device__ __forceinline__ void obstacle_tests(const Dev<T>& d, T px, T py, T pz, int& best, int& n_sph,
                                               int& n_mesh) {
  n_mesh = 0;
  sphere_tests(d, px, py, pz, best, n_sph);
  if (d.collision >= 2 && d.ot.n > 0)
    bvh_point_query(d.ot, 0, (double)px, (double)py, (double)pz, [&](int e) {
      if (strictly_inside_call(d.OX, px, py, pz, d.ot.prim[e])) ++n_mesh;
    });
}

// Block totals of one spring-update launch into this iteration's record: self
// pairs, finished springs and the springs' signature.
template <typename T>
__device__ __forceinline__ void spring_block_totals(const Dev<T>& d, int n_self, int n_spr, unsigned long long ssig,
                                                    int* shi) {
  if (d.stats) warp_add_u64(ssig, &(d.hist + (d.ctrl->iter % d.hist_cap))->spring_sig);
  const int s1 = block_sum_int(n_self, shi);
  const int s2 = block_sum_int(n_spr, shi);
  if (threadIdx.x == 0 && (s1 | s2)) {
    IterRec* rec = d.hist + (d.ctrl->iter % d.hist_cap);
    if (s1) atomicAdd(&rec->n_self_pairs, s1);
    if (s2) atomicAdd(&rec->n_springs, s2);
  }
}

// l1 norm, and triple product a . (b x c), in FP32.
__device__ __forceinline__ float l1(const float (&a)[3]) { return fabsf(a[0]) + fabsf(a[1]) + fabsf(a[2]); }
__device__ __forceinline__ float triple(const float (&a)[3], const float (&b)[3], const float (&c)[3]) {
  return a[0] * (b[1] * c[2] - b[2] * c[1]) + a[1] * (b[2] * c[0] - b[0] * c[2]) + a[2] * (b[0] * c[1] - b[1] * c[0]);
}

// FP32 test of a point against a tet, corners given as differences from the
// point: false only if one of the four orientation signs of the exact test is
// certainly negative.  Each sign is a triple product of differences, whose FP32
// rounding error is below 8 u times the product of the factors' 1-norms
// (u = 2^-24; 1e-6 = 16.8 u is used); dl bounds the error that rounded FP64
// positions add to a difference.  The constant covers underflow; differences
// above 1e9 (products that could overflow) and NaN pass, like every value
// within its bound.
__device__ __forceinline__ bool may_be_inside(const float (&a)[3], const float (&b)[3], const float (&c)[3],
                                              const float (&e)[3], float dl) {
  const float na = l1(a) + dl, nb = l1(b) + dl, nc = l1(c) + dl, ne = l1(e) + dl;
  if (!(na + nb + nc + ne < 1e9f)) return true;
  const float tiny = 1e-25f, k = 1e-6f;
  const float ab = na * nb, ce = nc * ne;
  const float e0 = k * nb * ce + dl * (nb * nc + ce + nb * ne) + tiny, e1 = k * na * ce + dl * (na * nc + ce + na * ne) + tiny,
              e2 = k * ab * ne + dl * (ab + na * ne + nb * ne) + tiny, e3 = k * ab * nc + dl * (ab + na * nc + nb * nc) + tiny;
  return !(triple(b, c, e) < -e0 || triple(a, c, e) > e1 || triple(a, b, e) < -e2 || triple(a, b, c) > e3);
}

// The same with the dl of tet t's rounded corners.
template <typename T>
__device__ __forceinline__ bool may_be_inside_at(const R4<T>* X, const float (&p)[3], int4 t) {
  const R4<T> c[4] = {X[t.x], X[t.y], X[t.z], X[t.w]};
  float e[4][3], dl = 0.0f;
  if constexpr (!std::is_same<T, float>::value) dl = l1(p);
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float x[3] = {(float)c[k].x, (float)c[k].y, (float)c[k].z};
    if constexpr (!std::is_same<T, float>::value) dl += l1(x);
#pragma unroll
    for (int j = 0; j < 3; ++j) e[k][j] = x[j] - p[j];
  }
  return may_be_inside(e[0], e[1], e[2], e[3], 0x1p-22f * dl);
}

// Zeroes the iteration's ray-cast list length and spring counts, which the spring
// update counts up and the casts and the solve read; by the threads of the first
// launch of the contact check, so whatever an iteration that ended early (a solve
// that gave up, a launch that failed) left there is gone.
template <typename T>
__device__ __forceinline__ void start_counts(const Dev<T>& d) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t == 0) d.ctrl->n_cast = 0;
  if (d.tm_springs)
    for (int r = t; r < d.n_robots; r += gridDim.x * blockDim.x) d.tm_springs[r] = 0;
}

static constexpr int BRICK = 3;  // edge of the bricks of cells that k_tets looks up at once

// Empty slot of a pair list (above every tet id).
static constexpr int NO_PAIR = 0x7FFFFFFF;

// Enters query vertex qi at position p (internal vertex v, robot rv) into the
// list of its cell, and clears its pair list.
template <typename T>
__device__ __forceinline__ void bin_query(const Dev<T>& d, int qi, int v, int rv, R4<T> p) {
  d.pair_count[qi] = 0;
  int* out = d.pair_tet + (size_t)qi * d.max_pairs;
  for (int k = 0; k < d.max_pairs; ++k) out[k] = NO_PAIR;
  if (!(d.collision >= 1 && isfinite(p.x) && isfinite(p.y) && isfinite(p.z))) return;
  const float inv = (float)d.inv_cell, x = (float)p.x, y = (float)p.y, z = (float)p.z;
  const int cx = cell_coord_f(x, inv), cy = cell_coord_f(y, inv), cz = cell_coord_f(z, inv);
  d.q_pos[qi] = make_float4(x, y, z, __int_as_float(v));
  d.q_next[qi] = atomicExch(&d.q_head[hash_cell(cx, cy, cz, rv) & (d.H_q - 1u)], qi + 1);
  // (a word's 32 cells overlap the next word's first 16, see k_tets; only the
  // first BRICK - 1 of those are looked up there)
  const unsigned words = d.H_q / 8 - 1u;
  atomicOr(&d.q_bits[hash_cell(cx >> 4, cy, cz, rv) & words], 1u << (cx & 15));
  if ((cx & 15) < BRICK - 1) atomicOr(&d.q_bits[hash_cell((cx >> 4) - 1, cy, cz, rv) & words], 0x10000u << (cx & 15));
}

static constexpr int QUERY_THREADS = 128;

// One thread per query vertex: its cell's list, and its obstacle tests.
template <typename T>
__global__ void __launch_bounds__(QUERY_THREADS, 4) k_queries(Dev<T> d) {
  __shared__ int shi[32];
  const int qi = blockIdx.x * QUERY_THREADS + threadIdx.x;
  start_counts(d);
  int n_obs = 0;
  if (qi < d.n_q) {
    const int v = d.q_verts[qi];
    const R4<T> p = d.X[v];
    bin_query(d, qi, v, d.robot_of_vert ? d.robot_of_vert[v] : 0, p);
    int best, n_sph, n_mesh;
    obstacle_tests(d, p.x, p.y, p.z, best, n_sph, n_mesh);
    n_obs = n_sph + n_mesh;
    d.obs_sphere[qi] = best;
    if (d.obs_mesh) d.obs_mesh[qi] = n_mesh;
  }
  if (d.collision < 2) return;
  const int s = block_sum_int(n_obs, shi);
  if (threadIdx.x == 0 && s) atomicAdd(&(d.hist + (d.ctrl->iter % d.hist_cap))->n_obstacle_pairs, s);
}

// Enters tet e into the pair list of query vertex qi: slot k keeps the smallest
// id it is given and passes the other on, so the list ends as the smallest
// max_pairs ids in ascending order whatever the order of arrival.
template <typename T>
__device__ __forceinline__ void add_pair(const Dev<T>& d, int qi, int e) {
  if (atomicAdd(&d.pair_count[qi], 1) >= d.max_pairs) set_status(d.ctrl, ST_PAIRS_TRUNC);
  int* out = d.pair_tet + (size_t)qi * d.max_pairs;
  for (int k = 0; k < d.max_pairs; ++k) {
    const int old = atomicMin(&out[k], e);
    if (old == NO_PAIR) break;
    e = max(old, e);
  }
}

__device__ __forceinline__ bool finite_t(float x) { return isfinite(x); }
__device__ __forceinline__ bool finite_t(double x) { return (__double2hiint(x) & 0x7FF00000) != 0x7FF00000; }

// Narrow phase, one lane per tet, over the cells of the tet's box: tests the
// query vertices listed in them whose own cell is the visited one (so every
// vertex of the box is met once).
//
// The lists hold the boundary vertices alone, far fewer entries than a hash of
// the tets needs.  Most cells are empty; a table of one bit per cell, small
// enough for the first-level cache, shows which, for a brick of 3 x 3 x 3 cells
// with nine independent reads (a word holds 32 cells along x, starting every 16,
// so that three neighbours always share one).  What is left is uneven, so each
// warp works it off together: its lanes append (tet, cell, first vertex) for the
// occupied cells to a queue, then each takes one entry, tests its vertex in FP32
// (own cell, box, signs) and appends the next one of the list.  The vertices that
// pass go to a second queue, and the exact tests, which may need FP64 or longer
// arithmetic, run on 32 of them at a time.
// CHECK: the tets are a caller's and their vertex ids are tested first.
// Measured (k_tets with k_queries, the faces' hash beside them) against a hash of
// all tets (count, scan, fill) and one warp per vertex: 117 and 321 us for
// 983,040 tets, 37 and 98 us for 193,920, 42 and 140 us for 51,840 in FP64.  Two
// to five blocks of 256 threads to an SM measured alike; blocks of 64 or 128
// threads, which each need the same shared memory, are slower at large sizes.
static constexpr int TETS_MAX_THREADS = 256;

template <typename T, bool CHECK>
__global__ void __launch_bounds__(TETS_MAX_THREADS, 4) k_tets(Dev<T> d, int per_warp) {
  constexpr unsigned FULL = 0xffffffffu;
  constexpr int WARPS = TETS_MAX_THREADS / 32;
  __shared__ unsigned s_entries;
  __shared__ int4 s_visits[WARPS][64], s_tet[WARPS][32];  // (cell, 32 x list entry + lane); vertex ids
  __shared__ int2 s_pairs[WARPS][64];                     // (tet, query vertex)
  __shared__ float s_x[WARPS][12][32];                    // corners
  if (threadIdx.x == 0) s_entries = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int i0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5) * per_warp;
  const int i = lane < per_warp ? i0 + lane : d.n_t;
  const unsigned before = (1u << lane) - 1u;
  int c0[3] = {0, 0, 0}, n[3] = {1, 1, 1}, ncell = 0;
  const float inv = (float)d.inv_cell;
  if (i < d.n_t) {
    int4 t = d.tet[i];
    bool valid = true;
    if (CHECK) {
      const unsigned nv = (unsigned)d.n_v;
      valid = (unsigned)t.x < nv && (unsigned)t.y < nv && (unsigned)t.z < nv && (unsigned)t.w < nv;
      if (!valid) set_status(d.ctrl, ST_BAD_INPUT);
    } else {
      t = chk_idx4(d.ctrl, t, d.n_v);
    }
    if (valid) {
      const R4<T> p[4] = {d.X[t.x], d.X[t.y], d.X[t.z], d.X[t.w]};
      // (rounding is monotone: the rounded box holds the rounded image of every
      // point of the tet, and so do the cells of its corners)
      float lo[3], hi[3];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        valid = valid && finite_t(p[k].x) && finite_t(p[k].y) && finite_t(p[k].z);
        const float x[3] = {(float)p[k].x, (float)p[k].y, (float)p[k].z};
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          s_x[wid][3 * k + j][lane] = x[j];
          lo[j] = k ? fminf(lo[j], x[j]) : x[j];
          hi[j] = k ? fmaxf(hi[j], x[j]) : x[j];
        }
      }
      if (!valid) {
        set_status(d.ctrl, ST_NONFINITE);
      } else {
        s_tet[wid][lane] = t;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          c0[j] = cell_coord_f(lo[j], inv);
          n[j] = cell_coord_f(hi[j], inv) - c0[j] + 1;
        }
        const long long m = (long long)n[0] * n[1] * n[2];
        if (m > MAX_CELLS_PER_ITEM) set_status(d.ctrl, ST_OVERFLOW);
        else ncell = (int)m;
      }
    }
  }
  {
    const unsigned m = __reduce_add_sync(FULL, (unsigned)ncell);
    if (lane == 0 && m) atomicAdd(&s_entries, m);
    __syncthreads();
    if (threadIdx.x == 0) add_entries(d, (unsigned long long)s_entries);
  }
  const int rt = d.robot_of_tet && i < d.n_t ? d.robot_of_tet[i] : 0;
  int bx = 0, by = 0, bz = ncell > 0 ? 0 : n[2];  // this lane's next brick (relative to the box),
  int ox = 0, oy = 0, oz = 0;                     //   the one before it,
  unsigned occ = 0;                               //   and that one's occupied cells not yet queued
  int n_visits = 0, n_pairs = 0;  // queued (the same in all lanes)
  for (;;) {
    while (n_visits < 32) {
      if (!__any_sync(FULL, occ || bz < n[2])) break;
      if (!occ && bz < n[2]) {
        const int cx = c0[0] + bx, shift = cx & 15;
        const unsigned keep = (1u << min(BRICK, n[0] - bx)) - 1u;
        unsigned row[BRICK * BRICK];
#pragma unroll
        for (int r = 0; r < BRICK * BRICK; ++r) {
          const int y = by + r % BRICK, z = bz + r / BRICK;
          row[r] = y < n[1] && z < n[2]
                       ? __ldg(&d.q_bits[hash_cell(cx >> 4, c0[1] + y, c0[2] + z, rt) & (d.H_q / 8 - 1u)])
                       : 0u;
        }
#pragma unroll
        for (int r = 0; r < BRICK * BRICK; ++r) occ |= (row[r] >> shift & keep) << (BRICK * r);
        ox = bx, oy = by, oz = bz;
        if ((bx += BRICK) >= n[0]) {
          bx = 0;
          if ((by += BRICK) >= n[1]) {
            by = 0;
            bz += BRICK;
          }
        }
      }
      int head = 0;
      int4 visit = make_int4(0, 0, 0, 0);
      if (occ) {
        const int b = __ffs(occ) - 1;
        occ &= occ - 1;
        visit = make_int4(c0[0] + ox + b % BRICK, c0[1] + oy + b / BRICK % BRICK, c0[2] + oz + b / (BRICK * BRICK), 0);
        head = __ldg(&d.q_head[hash_cell(visit.x, visit.y, visit.z, rt) & (d.H_q - 1u)]);
      }
      const unsigned who = __ballot_sync(FULL, head);
      visit.w = head * 32 + lane;
      if (head) s_visits[wid][n_visits + __popc(who & before)] = visit;
      n_visits += __popc(who);
    }
    __syncwarp();
    // one vertex to each lane
    const int take = min(n_visits, 32);
    const bool mine = lane < take;
    int4 visit = make_int4(0, 0, 0, 0);
    if (mine) visit = s_visits[wid][n_visits - 1 - lane];
    __syncwarp();
    n_visits -= take;
    bool cand = false;
    int qi = 0, next = 0;
    const int src = visit.w & 31;
    if (mine) {
      qi = chk_idx(d.ctrl, (int)((unsigned)visit.w >> 5) - 1, d.n_q);
      const float4 p = __ldg(&d.q_pos[qi]);
      next = __ldg(&d.q_next[qi]);
      const int v = __float_as_int(p.w);
      const int4 t = s_tet[wid][src];
      if (cell_coord_f(p.x, inv) == visit.x && cell_coord_f(p.y, inv) == visit.y && cell_coord_f(p.z, inv) == visit.z &&
          t.x != v && t.y != v && t.z != v && t.w != v) {
        // corners relative to the vertex (a difference of floats has its exact
        // sign, so the closed box test is exact; the exact test has the open one)
        float e[4][3], dl = 0.0f;
        const float pp[3] = {p.x, p.y, p.z};
        bool in_box = true;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float x = s_x[wid][3 * k + j][src];
            e[k][j] = x - pp[j];
            if constexpr (!std::is_same<T, float>::value) dl += fabsf(x);
          }
          if constexpr (!std::is_same<T, float>::value) dl += fabsf(pp[j]);
          in_box = in_box && min4(e[0][j], e[1][j], e[2][j], e[3][j]) <= 0.0f && max4(e[0][j], e[1][j], e[2][j], e[3][j]) >= 0.0f;
        }
        cand = in_box && may_be_inside(e[0], e[1], e[2], e[3], 0x1p-22f * dl);
      }
    }
    const unsigned again = __ballot_sync(FULL, next), who = __ballot_sync(FULL, cand);
    visit.w = next * 32 + src;
    if (next) s_visits[wid][n_visits + __popc(again & before)] = visit;
    n_visits += __popc(again);
    if (cand) s_pairs[wid][n_pairs + __popc(who & before)] = make_int2(i0 + src, qi);
    n_pairs += __popc(who);
    const bool last = take == 0;
    if (n_pairs >= 32 || last) {
      __syncwarp();
      const int m = min(n_pairs, 32);
      if (lane < m) {
        const int2 pr = s_pairs[wid][n_pairs - 1 - lane];
        const int v = d.q_verts[pr.y];
        if (!d.robot_of_tet || d.robot_of_vert[v] == d.robot_of_tet[pr.x]) {
          // (strictly_inside_at, with the four signs in a loop around one inlined
          // copy of the exact arithmetic: a call would cost the walk its registers)
          const R4<T> x = d.X[v];
          const int4 pt = d.tet[pr.x];
          const R4<T> p[4] = {d.X[pt.x], d.X[pt.y], d.X[pt.z], d.X[pt.w]};
          bool in = x.x > min4(p[0].x, p[1].x, p[2].x, p[3].x) && x.x < max4(p[0].x, p[1].x, p[2].x, p[3].x) &&
                    x.y > min4(p[0].y, p[1].y, p[2].y, p[3].y) && x.y < max4(p[0].y, p[1].y, p[2].y, p[3].y) &&
                    x.z > min4(p[0].z, p[1].z, p[2].z, p[3].z) && x.z < max4(p[0].z, p[1].z, p[2].z, p[3].z);
#pragma unroll 1
          for (int s = 0; s < 4 && in; ++s) {
            const R4<T> a = s == 0 ? x : p[0], b = s == 1 ? x : p[1], e = s == 2 ? x : p[2], f = s == 3 ? x : p[3];
            int sign = 0;
            if constexpr (std::is_same<T, float>::value)
              sign = orient_filter_f(a.x, a.y, a.z, b.x, b.y, b.z, e.x, e.y, e.z, f.x, f.y, f.z);
            if (sign == 0) sign = orient_filter(a.x, a.y, a.z, b.x, b.y, b.z, e.x, e.y, e.z, f.x, f.y, f.z);
            if (sign == 0) sign = orient_exact_inline(a.x, a.y, a.z, b.x, b.y, b.z, e.x, e.y, e.z, f.x, f.y, f.z);
            in = sign > 0;
          }
          if (in) add_pair(d, pr.y, pr.x);
        }
      }
      __syncwarp();
      n_pairs -= m;
      if (last && n_pairs == 0) break;
    }
  }
}

// ---- AABB trees: refit and point queries ----
// Refit after the positions moved (the tree's structure is kept, Sec. II-B):
// one thread per leaf computes its box and climbs; at every internal node the
// first of the two arriving threads stops, the second forms the union of the
// two children's boxes (the sibling's box was written before its arrival,
// fenced) and continues toward the root.
template <typename T>
__global__ void __launch_bounds__(256) k_bvh_refit(BvhDev b, const R4<T>* __restrict__ X) {
  const int p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= b.n) return;
  float4 lo, hi;
  prim_box(b, X, p, lo, hi);
  int me = ~p;
  int node = b.parent[b.n - 1 + p];
  while (node >= 0) {
    __threadfence();
    if (atomicAdd(&b.flag[node], 1) == 0) return;
    __threadfence();
    const int2 c = b.child[node];
    const int other = c.x == me ? c.y : c.x;
    float4 olo, ohi;
    if (other < 0) {
      prim_box(b, X, ~other, olo, ohi);
    } else {
      olo = __ldcg(&b.lo[other]);
      ohi = __ldcg(&b.hi[other]);
    }
    lo = make_float4(fminf(lo.x, olo.x), fminf(lo.y, olo.y), fminf(lo.z, olo.z), 0.0f);
    hi = make_float4(fmaxf(hi.x, ohi.x), fmaxf(hi.y, ohi.y), fmaxf(hi.z, ohi.z), 0.0f);
    __stcg(&b.lo[node], lo);
    __stcg(&b.hi[node], hi);
    me = node;
    node = b.parent[node];
  }
}

// Tree queries by teams of eight lanes: the nodes still to be visited wait on a
// stack in shared memory, and a round takes up to eight of them, one to a lane.
// A descent by one thread is a chain of dependent reads (a node's children, then
// their boxes) of some 60 to 100 nodes; a team's is about as long as the tree is
// deep.  Measured on a finger of 51,840 tets with a box of 768 as obstacle, one
// thread per query and eight lanes: narrow phase with the spring update 330 and
// 99 us (57 of them the tree queries, 36 the obstacle's closest faces), casts 572
// and 60 us.  (The four teams of a warp go round together; each on its own, their
// reads queue up behind one another: 75, 42 and 94 us.)
static constexpr int TEAM_LANES = 8;
static constexpr int TEAM_STACK = 128;
struct TeamStack {
  int node[TEAM_STACK];
  float key[TEAM_STACK];  // ray parameter or squared distance at which the node's box begins
  int cand[3 * TEAM_LANES];    // primitives that wait for their FP64 test,
  float cand_key[3 * TEAM_LANES];  // and a lower bound of their key
};
// Nodes of the next round with n on the stack: a node leaves at most two, so the
// stack stays within its size (one by one it grows by the tree's depth at most,
// for which 64 places are kept).
__device__ __forceinline__ int team_take(int n) { return min(min(TEAM_LANES, n), max(1, TEAM_STACK - BVH_STACK - n)); }
// Pushes ch of the lanes that have one; all lanes of the warp take part.
__device__ __forceinline__ void team_push(TeamStack& s, int& n, bool push, int ch, float key) {
  const int lane = threadIdx.x & 31;
  const unsigned who = __ballot_sync(0xffffffffu, push) & (0xFFu << (lane & 24));
  const int at = n + __popc(who & ((1u << lane) - 1u));
  if (push && at < TEAM_STACK) {
    s.node[at] = ch;
    s.key[at] = key;
  }
  n = min(n + __popc(who), TEAM_STACK);
}

// Calls leaf(p), by some lane of the team, for every primitive whose ancestors'
// boxes all contain the team's point (search: it has one).  The four teams of a
// warp go round together, so that their reads are in flight together.
template <typename Leaf>
__device__ __forceinline__ void team_point_query(const BvhDev& b, int tree, bool search, const PtF& pf, TeamStack& s,
                                                 Leaf leaf) {
  constexpr unsigned FULL = 0xffffffffu;
  const int tl = threadIdx.x & (TEAM_LANES - 1);
  const int root = search && b.n > 0 ? (b.root ? b.root[tree] : 0) : BVH_EMPTY;
  int n = 0;
  if (root >= 0) {
    if (box_has(b.lo[root], b.hi[root], pf)) n = 1;
    if (tl == 0) s.node[0] = root;
  } else if (root != BVH_EMPTY && tl == 0) {
    leaf(~root);
  }
  __syncwarp();
  while (__any_sync(FULL, n > 0)) {
    const int take = team_take(n);
    const int node = tl < take ? s.node[n - 1 - tl] : -1;
    __syncwarp();
    n -= take;
    int2 c = make_int2(0, 0);
    if (node >= 0) c = b.child[node];
    bool push[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int ch = k ? c.y : c.x;
      push[k] = node >= 0 && ch >= 0 && box_has(b.lo[ch], b.hi[ch], pf);
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int ch = k ? c.y : c.x;
      if (node >= 0 && ch < 0) leaf(~ch);
      team_push(s, n, push[k], ch, 0.0f);
    }
    __syncwarp();
  }
}

// Narrow phase over the robot's AABB tree (broad phase 1), a team per query
// vertex: the boxes containing it, then an FP32 test of the tets at the leaves,
// then the exact one; the same sorted pair list as the hash path's (at most
// max_pairs, the smallest tet ids).
static constexpr int NARROW_BVH_THREADS = 128;

template <typename T>
__global__ void __launch_bounds__(NARROW_BVH_THREADS, 4) k_narrow_bvh(Dev<T> d) {
  __shared__ int shi[32];
  __shared__ TeamStack s_stack[NARROW_BVH_THREADS / TEAM_LANES];
  const int qi = (blockIdx.x * NARROW_BVH_THREADS + threadIdx.x) / TEAM_LANES;
  const int tl = threadIdx.x & (TEAM_LANES - 1);
  TeamStack& stack = s_stack[threadIdx.x / TEAM_LANES];
  start_counts(d);
  int n_obs = 0;
  const bool valid = qi < d.n_q;
  const int v = valid ? d.q_verts[qi] : 0;
  const R4<T> pv = d.X[v];
  const T px = pv.x, py = pv.y, pz = pv.z;
  const float pf[3] = {(float)px, (float)py, (float)pz};
  if (valid) {
    if (tl == 0) d.pair_count[qi] = 0;
    for (int k = tl; k < d.max_pairs; k += TEAM_LANES) d.pair_tet[(size_t)qi * d.max_pairs + k] = NO_PAIR;
  }
  __syncwarp();
  const int rv = d.robot_of_vert ? d.robot_of_vert[v] : 0;
  const bool finite = isfinite(px) && isfinite(py) && isfinite(pz);
  if (valid && !finite && tl == 0) set_status(d.ctrl, ST_NONFINITE);
  const PtF q = pt_f((double)px, (double)py, (double)pz);
  team_point_query(d.bt, rv, valid && finite && d.collision >= 1, q, stack, [&](int e) {
    const int4 t = chk_idx4(d.ctrl, d.tet[e], d.n_v);
    if (d.robot_of_tet && d.robot_of_tet[e] != rv) return;
    if (t.x == v || t.y == v || t.z == v || t.w == v) return;
    if (may_be_inside_at(d.X, pf, t) && strictly_inside_call(d.X, px, py, pz, t)) add_pair(d, qi, e);
  });
  int best = -1, n_sph = 0, n_mesh = 0;
  if (valid && finite) sphere_tests(d, px, py, pz, best, n_sph);
  if (d.collision >= 2 && d.ot.n > 0) {
    team_point_query(d.ot, 0, valid && finite, q, stack, [&](int e) {
      const int4 t = d.ot.prim[e];
      if (may_be_inside_at(d.OX, pf, t) && strictly_inside_call(d.OX, px, py, pz, t)) ++n_mesh;
    });
#pragma unroll
    for (int o = TEAM_LANES / 2; o > 0; o >>= 1) n_mesh += __shfl_xor_sync(0xffffffffu, n_mesh, o);
  }
  if (valid && tl == 0) {
    n_obs = n_sph + n_mesh;
    d.obs_sphere[qi] = best;
    if (d.obs_mesh) d.obs_mesh[qi] = n_mesh;
  }
  const int s = block_sum_int(n_obs, shi);
  if (threadIdx.x == 0 && s) atomicAdd(&(d.hist + (d.ctrl->iter % d.hist_cap))->n_obstacle_pairs, s);
}

// ---- spring update ----
struct V3 {
  double x, y, z;
};
__device__ __forceinline__ V3 sub(V3 a, V3 b) { return {a.x - b.x, a.y - b.y, a.z - b.z}; }
__device__ __forceinline__ V3 add(V3 a, V3 b) { return {a.x + b.x, a.y + b.y, a.z + b.z}; }
__device__ __forceinline__ V3 scl(double s, V3 a) { return {s * a.x, s * a.y, s * a.z}; }
__device__ __forceinline__ double dot(V3 a, V3 b) { return a.x * b.x + a.y * b.y + a.z * b.z; }
__device__ __forceinline__ V3 cross(V3 a, V3 b) {
  return {a.y * b.z - a.z * b.y, a.z * b.x - a.x * b.z, a.x * b.y - a.y * b.x};
}
__device__ __forceinline__ double norm(V3 a) { return sqrt(dot(a, a)); }

template <typename T>
__device__ __forceinline__ V3 pos(const Dev<T>& d, int v) {
  const R4<T> a = d.X[v];
  return {(double)a.x, (double)a.y, (double)a.z};
}

// Moller-Trumbore with inclusive barycentrics and t > 0.
__device__ __forceinline__ bool ray_tri(V3 o, V3 dir, V3 q0, V3 q1, V3 q2, double& t, double& b1,
                                        double& b2) {
  const V3 e1 = sub(q1, q0), e2 = sub(q2, q0);
  const V3 pv = cross(dir, e2);
  const double det = dot(e1, pv);
  if (det == 0.0) return false;
  const double inv = 1.0 / det;
  const V3 tv = sub(o, q0);
  b1 = dot(tv, pv) * inv;
  const V3 qv = cross(tv, e1);
  b2 = dot(dir, qv) * inv;
  t = dot(e2, qv) * inv;
  return b1 >= 0.0 && b2 >= 0.0 && b1 + b2 <= 1.0 && t > 0.0;
}

// Closest point of a triangle: plane projection when inside, else the nearest
// edge projection.  Returns the barycentric weights of q1, q2.
__device__ __forceinline__ V3 closest_tri(V3 p, V3 q0, V3 q1, V3 q2, double& b1, double& b2) {
  const V3 e1 = sub(q1, q0), e2 = sub(q2, q0);
  const V3 n = cross(e1, e2);
  const double nn = dot(n, n);
  if (nn > 0.0) {
    const V3 x = sub(p, scl(dot(sub(p, q0), n) / nn, n));
    const double d11 = dot(e1, e1), d12 = dot(e1, e2), d22 = dot(e2, e2);
    const V3 r = sub(x, q0);
    const double r1 = dot(r, e1), r2 = dot(r, e2);
    const double den = d11 * d22 - d12 * d12;
    const double c1 = (d22 * r1 - d12 * r2) / den, c2 = (d11 * r2 - d12 * r1) / den;
    if (c1 >= 0.0 && c2 >= 0.0 && c1 + c2 <= 1.0) {
      b1 = c1;
      b2 = c2;
      return x;
    }
  }
  double bestd = 0.0;
  V3 best = q0;
  const V3 A[3] = {q0, q1, q2};
  const V3 B[3] = {q1, q2, q0};
  for (int k = 0; k < 3; ++k) {
    const V3 ab = sub(B[k], A[k]);
    const double den = dot(ab, ab);
    const double s = den == 0.0 ? 0.0 : fmin(1.0, fmax(0.0, dot(sub(p, A[k]), ab) / den));
    const V3 c = add(A[k], scl(s, ab));
    const V3 dd = sub(p, c);
    const double d2 = dot(dd, dd);
    if (k == 0 || d2 < bestd) {
      bestd = d2;
      best = c;
      if (k == 0) { b1 = s; b2 = 0.0; }
      else if (k == 1) { b1 = 1.0 - s; b2 = s; }
      else { b1 = 0.0; b2 = 1.0 - s; }
    }
  }
  return best;
}

template <typename T>
__device__ void face_verts(const Dev<T>& d, int f, V3& q0, V3& q1, V3& q2, int4& fv) {
  fv = chk_face(d.ctrl, d.faces[chk_idx(d.ctrl, f, d.n_f)], d.n_v);
  q0 = pos(d, fv.x);
  q1 = pos(d, fv.y);
  q2 = pos(d, fv.z);
}

// Warp argmin of (key, face id) over the lanes (face id < 0: no candidate);
// every lane ends with the minimum and its barycentrics.  The order is total,
// so the result does not depend on which lane held which face.
// Keys are non-negative doubles (ray parameters t > 0, squared distances), so
// their bit patterns order like their values and the comparisons run on the
// integer pipes: every lane of the warp takes part, and FP64 instructions
// with 32 active lanes are what the narrow FP64 pipe of this part is slowest
// at.
__device__ __forceinline__ unsigned long long key_bits(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ void warp_argmin(int& f, double& key, double& b1, double& b2) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const int of = __shfl_xor_sync(0xffffffffu, f, o);
    const double ok = __shfl_xor_sync(0xffffffffu, key, o);
    const double o1 = __shfl_xor_sync(0xffffffffu, b1, o);
    const double o2 = __shfl_xor_sync(0xffffffffu, b2, o);
    const unsigned long long kb = key_bits(key), okb = key_bits(ok);
    if (of >= 0 && (f < 0 || okb < kb || (okb == kb && of < f))) {
      f = of;
      key = ok;
      b1 = o1;
      b2 = o2;
    }
  }
}

// The same over the eight lanes of a team (all lanes of the warp take part).
__device__ __forceinline__ void team_argmin(int& f, double& key, double& b1, double& b2) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
    const int of = __shfl_xor_sync(0xffffffffu, f, o);
    const double ok = __shfl_xor_sync(0xffffffffu, key, o);
    const double o1 = __shfl_xor_sync(0xffffffffu, b1, o);
    const double o2 = __shfl_xor_sync(0xffffffffu, b2, o);
    const unsigned long long kb = key_bits(key), okb = key_bits(ok);
    if (of >= 0 && (f < 0 || okb < kb || (okb == kb && of < f))) {
      f = of;
      key = ok;
      b1 = o1;
      b2 = o2;
    }
  }
}

// FP32 bounds of the squared distance from a point to a triangle, its corners
// given as differences from the point (dl bounds the error that rounded FP64
// positions add to one).  The upper one is the distance of some point of the
// triangle, the lower one that of its support plane across the way there
// (no corner lies nearer along that direction), so neither depends on how good
// that point is; each has a margin for the rounding of its own evaluation, which
// is below 32 u times the corners' largest 1-norm (u = 2^-24).
__device__ __forceinline__ void triangle_d2_bounds(const float (&a)[3], const float (&b)[3], const float (&c)[3], float dl,
                                                   float& lb, float& ub) {
  float w[3] = {0.0f, 0.0f, 0.0f}, best = INFINITY;  // nearest point found
  auto at = [&](float x, float y, float z) {
    const float m = x * x + y * y + z * z;
    if (m < best) {
      best = m;
      w[0] = x;
      w[1] = y;
      w[2] = z;
    }
  };
  auto edge = [&](const float (&p)[3], const float (&q)[3]) {
    const float ex = q[0] - p[0], ey = q[1] - p[1], ez = q[2] - p[2];
    const float ee = ex * ex + ey * ey + ez * ez;
    const float t = ee > 0.0f ? fminf(fmaxf(-(p[0] * ex + p[1] * ey + p[2] * ez) / ee, 0.0f), 1.0f) : 0.0f;
    at(p[0] + t * ex, p[1] + t * ey, p[2] + t * ez);
  };
  edge(a, b);
  edge(b, c);
  edge(c, a);
  {
    // projection onto the plane, if it falls inside
    const float ux = b[0] - a[0], uy = b[1] - a[1], uz = b[2] - a[2], vx = c[0] - a[0], vy = c[1] - a[1], vz = c[2] - a[2];
    const float nx = uy * vz - uz * vy, ny = uz * vx - ux * vz, nz = ux * vy - uy * vx;
    const float nn = nx * nx + ny * ny + nz * nz;
    const float wb = nx * (vy * a[2] - vz * a[1]) + ny * (vz * a[0] - vx * a[2]) + nz * (vx * a[1] - vy * a[0]);
    const float wc = nx * (a[1] * uz - a[2] * uy) + ny * (a[2] * ux - a[0] * uz) + nz * (a[0] * uy - a[1] * ux);
    if (wb >= 0.0f && wc >= 0.0f && wb + wc <= nn && nn > 0.0f) {
      const float s = wb / nn, t = wc / nn;
      at(a[0] + s * ux + t * vx, a[1] + s * uy + t * vy, a[2] + s * uz + t * vz);
    }
  }
  const float size = fmaxf(l1(a), fmaxf(l1(b), l1(c)));
  const float margin = 2e-6f * size + dl;
  const float len = sqrtf(best);
  const float far = len * 1.000001f + margin;
  ub = far * far * 1.000001f + 1e-37f;
  const float da = w[0] * a[0] + w[1] * a[1] + w[2] * a[2], db = w[0] * b[0] + w[1] * b[1] + w[2] * b[2],
              dc = w[0] * c[0] + w[1] * c[1] + w[2] * c[2];
  const float near = len > 1e-15f ? fminf(da, fminf(db, dc)) / len * 0.999999f - margin : 0.0f;
  lb = near > 0.0f ? near * near * 0.999999f : 0.0f;
}
template <typename T>
__device__ __forceinline__ void triangle_bounds_at(const R4<T>& q0, const R4<T>& q1, const R4<T>& q2, const R4<T>& x,
                                                   float& lb, float& ub) {
  const float p[3] = {(float)x.x, (float)x.y, (float)x.z};
  float q[3][3] = {{(float)q0.x, (float)q0.y, (float)q0.z}, {(float)q1.x, (float)q1.y, (float)q1.z},
                   {(float)q2.x, (float)q2.y, (float)q2.z}};
  float dl = 0.0f;
  if constexpr (!std::is_same<T, float>::value) dl = 0x1p-22f * (l1(p) + l1(q[0]) + l1(q[1]) + l1(q[2]));
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int j = 0; j < 3; ++j) q[k][j] -= p[j];
  triangle_d2_bounds(q[0], q[1], q[2], dl, lb, ub);
}

// Closest-point candidate of face f for point o (lane-local running minimum).
template <typename T>
__device__ __forceinline__ void closest_candidate(const Dev<T>& d, int v, int rv, int f, V3 o, int& lf, double& ld,
                                                  double& l1, double& l2) {
  if (d.robot_of_face && d.robot_of_face[f] != rv) return;
  V3 q0, q1, q2;
  int4 fv;
  face_verts(d, f, q0, q1, q2, fv);
  if (fv.x == v || fv.y == v || fv.z == v) return;
  double b1, b2;
  const V3 x = closest_tri(o, q0, q1, q2, b1, b2);
  const V3 dd = sub(o, x);
  const double d2 = dot(dd, dd);
  if (lf < 0 || d2 < ld || (d2 == ld && f < lf)) {
    lf = f;
    ld = d2;
    l1 = b1;
    l2 = b2;
  }
}

// Closest boundary face, among those not containing vertex v, to point o of v
// (robot rv) by one warp, and the closest point's barycentrics.
// Found by scanning cubic shells of cells around v's cell.  After shell k every
// face with a point within k cells has been seen, so the search stops once the
// best distance is at most k cell edges (after the first neighbours at the
// earliest).  The shell's faces are spread over the lanes whatever their cells,
// FP32 bounds of their distances sort out the ones that cannot be closest, and
// what is left waits in a queue for the FP64 test.  (With a cell to a lane and
// FP64 throughout, one lane tested the ten faces of v's own cell one by one, 40 us
// for any launch with such a vertex.)
struct FaceQueue {
  int face[64];
  float low[64];  // lower bound of the squared distance
};
template <typename T>
__device__ int closest_face_warp(const Dev<T>& d, FaceQueue& queue, int v, int rv, V3 o, double& rb1, double& rb2) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const R4<T> x = {(T)o.x, (T)o.y, (T)o.z, T(0)};
  int best_f = -1, n = 0;
  rb1 = rb2 = 0.0;
  const int c0[3] = {cell_coord(o.x, d.inv_cell), cell_coord(o.y, d.inv_cell), cell_coord(o.z, d.inv_cell)};
  double bestd = 0.0;
  float limit = INFINITY;
  auto test = [&]() {  // the last of the queued faces, one to a lane
    __syncwarp();
    const int take = min(n, 32);
    int lf = -1;
    double ld = 0.0, l1 = 0.0, l2 = 0.0;
    if (lane < take && !(queue.low[n - 1 - lane] > limit))
      closest_candidate(d, v, rv, queue.face[n - 1 - lane], o, lf, ld, l1, l2);
    __syncwarp();
    n -= take;
    warp_argmin(lf, ld, l1, l2);
    if (lf >= 0 && (best_f < 0 || ld < bestd || (ld == bestd && lf < best_f))) {
      best_f = lf;
      bestd = ld;
      rb1 = l1;
      rb2 = l2;
      limit = fminf(limit, __double2float_ru(bestd));
    }
  };
  for (int k = 0; k <= 64; ++k) {
    const int side = 2 * k + 1;
    const int ncell = side * side * side;
    for (int base = 0; base < ncell; base += 32) {
      // this lane's cell, and the entries of the 32 cells in one sequence
      const int idx = base + lane;
      const int dx = idx % side - k, dy = (idx / side) % side - k, dz = idx / (side * side) - k;
      int first = 0, upto = 0;
      if (idx < ncell && max(abs(dx), max(abs(dy), abs(dz))) == k) {
        const int2 r = d.cell_range[hash_cell(c0[0] + dx, c0[1] + dy, c0[2] + dz, rv) & (d.H_f - 1u)];
        first = r.x;
        upto = max(min(r.y, d.cap_items) - r.x, 0);
      }
#pragma unroll
      for (int m = 1; m < 32; m <<= 1) {
        const int u = __shfl_up_sync(FULL, upto, m);
        if (lane >= m) upto += u;
      }
      const int total = __shfl_sync(FULL, upto, 31);
      for (int e0 = 0; e0 < total; e0 += 32) {
        // the cell of entry e: the number of cells whose sequences end at or before it
        const int e = e0 + lane;
        int cell = 0;
#pragma unroll
        for (int m = 16; m > 0; m >>= 1)
          if (__shfl_sync(FULL, upto, cell + m - 1) <= e) cell += m;
        cell = min(cell, 31);
        const int before = __shfl_sync(FULL, upto, max(cell - 1, 0)), start = __shfl_sync(FULL, first, cell);
        int f = -1;
        float lb = 0.0f, ub = INFINITY;
        if (e < total) {
          f = d.items[start + e - (cell ? before : 0)];
          const int4 fv = chk_face(d.ctrl, d.faces[chk_idx(d.ctrl, f, d.n_f)], d.n_v);
          if ((d.robot_of_face && d.robot_of_face[f] != rv) || fv.x == v || fv.y == v || fv.z == v) f = -1;
          else triangle_bounds_at(d.X[fv.x], d.X[fv.y], d.X[fv.z], x, lb, ub);
        }
        if (f < 0) ub = INFINITY;
#pragma unroll
        for (int m = 16; m > 0; m >>= 1) ub = fminf(ub, __shfl_xor_sync(FULL, ub, m));
        limit = fminf(limit, ub);
        const unsigned keep = __ballot_sync(FULL, f >= 0 && !(lb > limit));
        if (keep >> lane & 1u) {
          const int at = n + __popc(keep & ((1u << lane) - 1u));
          queue.face[at] = f;
          queue.low[at] = lb;
        }
        n += __popc(keep);
        if (n > 32) test();
      }
    }
    if (k == 0) continue;
    while (n > 0) test();
    if (best_f >= 0 && sqrt(bestd) <= k * d.cell) return best_f;
  }
  if (best_f >= 0) return best_f;
  // the shell search found nothing within 64 cells: every face (rare)
  int lf = -1;
  double ld = 0.0, l1 = 0.0, l2 = 0.0;
  for (int f = lane; f < d.n_f; f += 32) closest_candidate(d, v, rv, f, o, lf, ld, l1, l2);
  warp_argmin(lf, ld, l1, l2);
  rb1 = l1;
  rb2 = l2;
  return lf;
}

template <typename T>
__device__ __forceinline__ V3 face_point(const Dev<T>& d, int f, double b1, double b2, V3& nunit) {
  V3 q0, q1, q2;
  int4 fv;
  face_verts(d, f, q0, q1, q2, fv);
  V3 n = cross(sub(q1, q0), sub(q2, q0));
  nunit = scl(1.0 / norm(n), n);
  return add(add(scl(1.0 - b1 - b2, q0), scl(b1, q1)), scl(b2, q2));
}

// Point and unit outward normal of boundary face f of the tetrahedral
// obstacle at barycentrics (b1, b2).
template <typename T>
__device__ __forceinline__ V3 obstacle_face_point(const Dev<T>& d, int f, double b1, double b2, V3& nunit) {
  const int4 fv = d.oface[f];
  const R4<T> a = d.OX[fv.x], b = d.OX[fv.y], c = d.OX[fv.z];
  const V3 q0 = {(double)a.x, (double)a.y, (double)a.z}, q1 = {(double)b.x, (double)b.y, (double)b.z},
           q2 = {(double)c.x, (double)c.y, (double)c.z};
  const V3 n = cross(sub(q1, q0), sub(q2, q0));
  nunit = scl(1.0 / norm(n), n);
  return add(add(scl(1.0 - b1 - b2, q0), scl(b1, q1)), scl(b2, q2));
}

// Best primitive of a tree for each searching team of the warp; all lanes take
// part.  begin(lo, hi) is the FP32 key at which a box begins (INFINITY: never),
// may(f, lb, ub) an FP32 test of a primitive with bounds of its key, test(f, key,
// e1, e2) the FP64 one.  The smallest key wins, then the lowest id; what begins
// beyond limit_of(best key), or slack times an upper bound, holds nothing better.  The teams visit their nodes and
// collect the primitives that FP32 leaves open, and only then meet for the FP64
// test of all teams' (it costs its scheduler as much for one lane as for 32).
template <typename Begin, typename May, typename Test, typename Limit>
__device__ __forceinline__ void team_search(const BvhDev& b, int root, bool search, TeamStack& stack, int& bf, double& bt,
                                            double& b1, double& b2, Begin begin, May may, Test test, Limit limit_of,
                                            float slack = 1.0f) {
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, tl = lane & (TEAM_LANES - 1);
  const unsigned tmask = 0xFFu << (lane & 24), before = (1u << lane) - 1u;
  float limit = INFINITY;
  int n = 0, nc = 0;  // nodes and primitives waiting
  if (search && root != BVH_EMPTY) {
    if (root < 0) {
      nc = 1;
      if (tl == 0) {
        stack.cand[0] = ~root;
        stack.cand_key[0] = -INFINITY;
      }
    } else {
      const float key = begin(b.lo[root], b.hi[root]);
      n = key < INFINITY ? 1 : 0;
      if (tl == 0) {
        stack.node[0] = root;
        stack.key[0] = key;
      }
    }
  }
  __syncwarp();
  for (;;) {
    while (__any_sync(FULL, n > 0 && nc <= TEAM_LANES)) {
      // (the teams that wait for the others take nothing)
      const int take = nc <= TEAM_LANES ? team_take(n) : 0;
      int node = -1;
      if (tl < take && stack.key[n - 1 - tl] <= limit) node = stack.node[n - 1 - tl];
      __syncwarp();
      n -= take;
      int2 c = make_int2(0, 0);
      if (node >= 0) c = b.child[node];
      float key[2] = {INFINITY, INFINITY}, low[2] = {0.0f, 0.0f};
      bool open[2] = {false, false};
      float least = limit;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int ch = k ? c.y : c.x;
        if (node < 0) continue;
        if (ch >= 0) {
          key[k] = begin(b.lo[ch], b.hi[ch]);
        } else {
          float ub = INFINITY;
          open[k] = may(~ch, low[k], ub);
          if (open[k]) least = fminf(least, ub * slack);
        }
      }
#pragma unroll
      for (int o = TEAM_LANES / 2; o > 0; o >>= 1) least = fminf(least, __shfl_xor_sync(FULL, least, o));
      limit = least;
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const bool keep = open[k] && !(low[k] > limit);
        const unsigned who = __ballot_sync(FULL, keep) & tmask;
        const int at = nc + __popc(who & before);
        if (keep) {
          stack.cand[at] = ~(k ? c.y : c.x);
          stack.cand_key[at] = low[k];
        }
        nc += __popc(who);
      }
      // the farther child first, so that the nearer one is visited next
      const bool swap = key[1] > key[0];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const bool second = (k == 0) == swap;
        const float t = second ? key[1] : key[0];
        team_push(stack, n, t < INFINITY && t <= limit, second ? c.y : c.x, t);
      }
      __syncwarp();
    }
    if (!__any_sync(FULL, nc > 0)) break;
    const int take = min(nc, TEAM_LANES);
    int f = -1;
    if (tl < take && !(stack.cand_key[nc - 1 - tl] > limit)) f = stack.cand[nc - 1 - tl];
    __syncwarp();
    nc -= take;
    if (!__any_sync(FULL, f >= 0)) continue;
    int lf = -1;
    double lk = 0.0, e1 = 0.0, e2 = 0.0;
    if (f >= 0 && test(f, lk, e1, e2)) lf = f;
    if (!__any_sync(FULL, lf >= 0)) continue;
    team_argmin(lf, lk, e1, e2);
    if (lf >= 0 && (bf < 0 || key_bits(lk) < key_bits(bt) || (key_bits(lk) == key_bits(bt) && lf < bf))) {
      bf = lf;
      bt = lk;
      b1 = e1;
      b2 = e2;
      limit = fminf(limit, limit_of(bt));
    }
  }
}

// Closest boundary face of the tetrahedral obstacle to each team's point, and its
// barycentrics and squared distance.
template <typename T>
__device__ __forceinline__ int team_obstacle_closest(const Dev<T>& d, bool search, R4<T> xv, TeamStack& stack,
                                                     double& b1, double& b2, double& d2) {
  const V3 x = {(double)xv.x, (double)xv.y, (double)xv.z};
  int bf = -1;
  b1 = b2 = d2 = 0.0;
  const PtF pf = pt_f(x.x, x.y, x.z);
  const int root = d.of.n > 0 ? (d.of.root ? d.of.root[0] : 0) : BVH_EMPTY;
  team_search(
      d.of, root, search, stack, bf, d2, b1, b2, [&](float4 lo, float4 hi) { return box_d2(lo, hi, pf); },
      [&](int f, float& lb, float& ub) {
        const int4 fv = d.oface[f];
        triangle_bounds_at(d.OX[fv.x], d.OX[fv.y], d.OX[fv.z], xv, lb, ub);
        return true;
      },
      [&](int f, double& key, double& e1, double& e2) {
        const int4 fv = d.oface[f];
        const R4<T> a = d.OX[fv.x], b = d.OX[fv.y], c = d.OX[fv.z];
        const V3 dd = sub(x, closest_tri(x, V3{(double)a.x, (double)a.y, (double)a.z}, V3{(double)b.x, (double)b.y, (double)b.z},
                                         V3{(double)c.x, (double)c.y, (double)c.z}, e1, e2));
        key = dot(dd, dd);
        return true;
      },
      [](double best) { return __double2float_ru(best); });
  return bf;
}

// Spring update, one thread per query vertex.  A vertex in a self pair (and
// in no obstacle) needs a ray cast: it is appended to the cast list and finished
// by k_cast (or k_cast_bvh); every other vertex is finished by the update itself.
static constexpr int CAST_THREADS = 256;

// Signature term of one spring record (see sig_mix): query index and the
// decision code (0 a self spring kept from its record, 1 a sphere spring, 2 a
// tetrahedral-obstacle spring, 3 a self spring cast in this iteration) with
// the face, sphere or obstacle face id.
__device__ __forceinline__ unsigned long long spring_term(int qi, int code, int face) {
  return sig_mix((unsigned)qi, ((unsigned)code << 30) ^ (unsigned)(face + 1));
}

// Spring update of query vertex qi, by one thread, once its contacts of this
// iteration are known (pair_count, obs_sphere, and for a vertex inside the
// tetrahedral obstacle its closest face mf there with barycentrics m1, m2 and
// squared distance md2): creates, re-targets or releases its spring, or queues
// it for a ray cast.  Adds 1 to active_out for a finished active spring and its
// signature term to ssig.
template <typename T>
__device__ void spring_update_vertex(const Dev<T>& d, int qi, bool in_mesh, int mf, double m1, double m2, double md2,
                                     int& active_out, unsigned long long& ssig) {
  {
    const int v = d.q_verts[qi];
    // area-weighted unit vertex normal of the incident boundary faces, formed
    // only where it is used (a sphere spring whose vertex sits at the centre)
    auto normal = [&]() {
      V3 n = {0.0, 0.0, 0.0};
      for (int k = d.qf_ptr[qi]; k < d.qf_ptr[qi + 1]; ++k) {
        V3 q0, q1, q2;
        int4 fv;
        face_verts(d, d.qf[k], q0, q1, q2, fv);
        n = add(n, cross(sub(q1, q0), sub(q2, q0)));
      }
      const double nl = norm(n);
      return nl > 0.0 ? scl(1.0 / nl, n) : V3{0.0, 0.0, 0.0};
    };
    int active = d.sp.active[qi];
    int kind = d.sp.kind[qi];
    int face = d.sp.face[qi];
    double b1 = d.sp.bary[2 * qi], b2 = d.sp.bary[2 * qi + 1];
    V3 tgt = {0.0, 0.0, 0.0};
    int js = d.obs_sphere[qi];
    const double eps = d.eps;
    bool deferred = false;
    // the position in FP64, read only by a vertex with an obstacle contact or
    // a spring to re-target (the conversions are FP64 instructions)
    V3 x = {0.0, 0.0, 0.0};
    if (in_mesh || js >= 0 || active) x = pos(d, v);
    // inside the tetrahedral obstacle: its closest boundary point, unless a
    // containing sphere's surface is at least as near (signed distances
    // |x - c| - r and minus the distance to the obstacle's boundary)
    if (js >= 0 && mf >= 0) {
      const V3 c = {d.spheres[4 * js], d.spheres[4 * js + 1], d.spheres[4 * js + 2]};
      if (!(norm(sub(x, c)) - d.spheres[4 * js + 3] <= -sqrt(md2))) js = -1;
      else mf = -1;
    }
    if (js >= 0) {
      const V3 c = {d.spheres[4 * js], d.spheres[4 * js + 1], d.spheres[4 * js + 2]};
      const double r = d.spheres[4 * js + 3];
      V3 u = sub(x, c);
      const double nu = norm(u);
      u = nu == 0.0 ? scl(-1.0, normal()) : scl(1.0 / nu, u);
      active = 1;
      kind = 1;
      face = js;
      b1 = b2 = 0.0;
      tgt = add(c, scl(r + eps, u));
    } else if (mf >= 0) {
      V3 nf;
      const V3 bp = obstacle_face_point(d, mf, m1, m2, nf);
      active = 1;
      kind = 2;
      face = mf;
      b1 = m1;
      b2 = m2;
      tgt = add(bp, scl(eps, nf));
    } else if (d.pair_count[qi] > 0) {
      deferred = true;
      const int slot = atomicAdd(&d.ctrl->n_cast, 1);  // < n_q: each vertex enters once
      if (slot < d.n_q) d.cast_list[slot] = qi;
    } else if (active) {
      if (kind == 1) {
        const V3 c = {d.spheres[4 * face], d.spheres[4 * face + 1], d.spheres[4 * face + 2]};
        const double r = d.spheres[4 * face + 3];
        V3 u = sub(x, c);
        const double nu = norm(u);
        if (nu - r > eps) {
          active = 0;
        } else {
          u = nu == 0.0 ? scl(-1.0, normal()) : scl(1.0 / nu, u);
          tgt = add(c, scl(r + eps, u));
        }
      } else if (kind == 2) {
        V3 nf;
        const V3 bp = obstacle_face_point(d, face, b1, b2, nf);
        if (dot(nf, sub(x, bp)) > eps) {
          active = 0;
        } else {
          tgt = add(bp, scl(eps, nf));
        }
      } else {
        V3 nf;
        const V3 bp = face_point(d, face, b1, b2, nf);
        if (dot(nf, sub(x, bp)) > eps) {
          active = 0;
        } else {
          tgt = add(bp, scl(eps, nf));
        }
      }
    }
    if (!deferred) {
      if (!active) {
        kind = 0;
        face = -1;
        b1 = b2 = 0.0;
        tgt = {0.0, 0.0, 0.0};
      }
      d.sp.active[qi] = active;
      d.sp.fallback[qi] = 0;
      d.sp.kind[qi] = kind;
      d.sp.face[qi] = face;
      d.sp.bary[2 * qi] = b1;
      d.sp.bary[2 * qi + 1] = b2;
      d.sp.target[3 * qi] = tgt.x;
      d.sp.target[3 * qi + 1] = tgt.y;
      d.sp.target[3 * qi + 2] = tgt.z;
      d.spring_c[v] = R4<double>{tgt.x, tgt.y, tgt.z, active ? 1.0 : 0.0};
      active_out += active;
      if (active) {
        ssig += spring_term(qi, kind, face);
        if (d.tm_springs) atomicAdd(&d.tm_springs[d.robot_of_vert ? d.robot_of_vert[v] : 0], 1);
      }
    }
  }
}

// Spring update of every query vertex, one thread each, and the contact counts
// of the narrow phase.
template <typename T>
__global__ void __launch_bounds__(128) k_springs(Dev<T> d) {
  __shared__ int shi[32];
  const int qi = blockIdx.x * blockDim.x + threadIdx.x;
  int n_self = 0, n_spr = 0;
  unsigned long long ssig = 0;
  if (qi < d.n_q) {
    n_self = d.pair_count[qi];
    if (n_self > d.max_pairs) d.pair_count[qi] = n_self = d.max_pairs;
    // (vertices inside the tetrahedral obstacle: k_mesh_springs)
    if (!(d.obs_mesh && d.obs_mesh[qi] > 0)) spring_update_vertex(d, qi, false, -1, 0.0, 0.0, 0.0, n_spr, ssig);
  }
  spring_block_totals(d, n_self, n_spr, ssig, shi);
}

// Spring update of the vertices inside the tetrahedral obstacle, a team per query
// vertex (most teams leave at once).
template <typename T>
__global__ void __launch_bounds__(NARROW_BVH_THREADS, 3) k_mesh_springs(Dev<T> d) {
  __shared__ int shi[32];
  __shared__ TeamStack s_stack[NARROW_BVH_THREADS / TEAM_LANES];
  const int qi = (blockIdx.x * NARROW_BVH_THREADS + threadIdx.x) / TEAM_LANES;
  const bool in_mesh = qi < d.n_q && d.obs_mesh[qi] > 0;
  int n_spr = 0;
  unsigned long long ssig = 0;
  if (__any_sync(0xffffffffu, in_mesh)) {
    R4<T> x{};
    if (in_mesh) x = d.X[d.q_verts[qi]];
    double m1, m2, md2;
    const int mf = team_obstacle_closest(d, in_mesh, x, s_stack[threadIdx.x / TEAM_LANES], m1, m2, md2);
    if (in_mesh && (threadIdx.x & (TEAM_LANES - 1)) == 0) spring_update_vertex(d, qi, true, mf, m1, m2, md2, n_spr, ssig);
  }
  spring_block_totals(d, 0, n_spr, ssig, shi);
}

// FP32 test of a face against a ray from o along the unit direction dir, which
// may only reject what the FP64 test (exit face, then ray_tri) rejects.  The
// signs of five triple products decide: dir.(e1 x e2) > 0 (exit face), the two
// barycentrics and their sum, the ray parameter.  Each is formed in FP32 from
// coordinate differences; with |dir| = 1 its rounding errors are below 8 u times
// the product of the factors' 1-norms (u = 2^-24; two differences, dir, the
// products and the sums), and 1e-6 = 16.8 u is used.  FP64 positions enter
// rounded to FP32, which adds dl = 2^-22 times the coordinates' sizes to every
// difference.  The constant covers underflow, differences above 1e9 (products
// that could overflow) and NaN pass, like every value within its bound.  A face
// that is certainly hit gives an upper bound t_max of its ray parameter (INFINITY
// otherwise).
template <typename T>
__device__ __forceinline__ bool face_may_hit(const R4<T>& q0, const R4<T>& q1, const R4<T>& q2, const float (&o)[3],
                                             const float (&dir)[3], float& t_max) {
  const float a[3] = {(float)q0.x, (float)q0.y, (float)q0.z}, b[3] = {(float)q1.x, (float)q1.y, (float)q1.z},
              c[3] = {(float)q2.x, (float)q2.y, (float)q2.z};
  float e1[3], e2[3], tv[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    e1[k] = b[k] - a[k];
    e2[k] = c[k] - a[k];
    tv[k] = o[k] - a[k];
  }
  const float dl = std::is_same<T, float>::value ? 0.0f : 0x1p-22f * (l1(a) + l1(b) + l1(c) + l1(o));
  const float n1 = l1(e1) + dl, n2 = l1(e2) + dl, n0 = l1(tv) + dl;
  t_max = INFINITY;
  if (!(n0 + n1 + n2 < 1e9f)) return true;
  const float tiny = 1e-25f, k = 1e-6f;
  const float det = triple(dir, e1, e2);          // > 0 for an exit face
  const float v1 = triple(tv, dir, e2);           // -b1 det
  const float v2 = triple(dir, tv, e1);           // -b2 det
  const float vt = triple(e2, tv, e1);            // -t det
  const float bd = k * n1 * n2 + dl * (n1 + n2) + tiny, b1 = k * n0 * n2 + dl * (n0 + n2) + tiny,
              b2 = k * n0 * n1 + dl * (n0 + n1) + tiny,
              bt = k * n0 * n1 * n2 + dl * (n0 * n1 + n1 * n2 + n0 * n2) + tiny;
  if (det > 2.0f * bd && v1 < -b1 && v2 < -b2 && v1 + v2 + det > bd + b1 + b2 && vt < -bt)
    t_max = (bt - vt) / (det - bd) * 1.00001f;
  return !(det < -bd || v1 > b1 || v2 > b2 || -(v1 + v2) - det > bd + b1 + b2 || vt > bt);
}

// Ray direction of query vertex qi (unit, against the area-weighted normal of its
// incident boundary faces, which are summed in their listed order), by a team of
// eight lanes; all lanes of the warp take part.
template <typename T>
__device__ __forceinline__ V3 cast_direction(const Dev<T>& d, int qi) {
  constexpr unsigned FULL = 0xffffffffu;
  const int tl = threadIdx.x & 7;
  V3 n = {0.0, 0.0, 0.0};
  const int f0 = d.qf_ptr[qi], nf = d.qf_ptr[qi + 1] - f0, most = __reduce_max_sync(FULL, nf);
  for (int k = 0; k < most; k += 8) {
    V3 c = {0.0, 0.0, 0.0};
    if (k + tl < nf) {
      V3 q0, q1, q2;
      int4 fv;
      face_verts(d, d.qf[f0 + k + tl], q0, q1, q2, fv);
      c = cross(sub(q1, q0), sub(q2, q0));
    }
    for (int s = 0; s < min(8, most - k); ++s)
      n = add(n, V3{__shfl_sync(FULL, c.x, s, 8), __shfl_sync(FULL, c.y, s, 8), __shfl_sync(FULL, c.z, s, 8)});
  }
  const double nl = norm(n);
  return nl > 0.0 ? scl(-1.0 / nl, n) : V3{0.0, 0.0, 0.0};
}

// Records the spring of query vertex qi (internal vertex v, robot rv) from its
// correspondence: face (or -1) and barycentrics; 1 if it is active.
template <typename T>
__device__ __forceinline__ int finish_cast(const Dev<T>& d, int qi, int v, int rv, int face, bool missed, double b1,
                                           double b2) {
  V3 tgt = {0.0, 0.0, 0.0};
  if (face >= 0) {
    V3 nh;
    const V3 bp = face_point(d, face, b1, b2, nh);
    tgt = add(bp, scl(d.eps, nh));
  } else {
    b1 = b2 = 0.0;
  }
  const int active = face >= 0;
  d.sp.active[qi] = active;
  d.sp.fallback[qi] = missed;
  d.sp.kind[qi] = 0;
  d.sp.face[qi] = face;
  d.sp.bary[2 * qi] = b1;
  d.sp.bary[2 * qi + 1] = b2;
  d.sp.target[3 * qi] = tgt.x;
  d.sp.target[3 * qi + 1] = tgt.y;
  d.sp.target[3 * qi + 2] = tgt.z;
  d.spring_c[v] = R4<double>{tgt.x, tgt.y, tgt.z, active ? 1.0 : 0.0};
  if (active && d.tm_springs) atomicAdd(&d.tm_springs[rv], 1);
  if (active && d.stats)
    atomicAdd(&(d.hist + (d.ctrl->iter % d.hist_cap))->spring_sig, spring_term(qi, 3, face));
  return active;
}

// Self springs of the listed vertices: eight lanes per vertex (persistent grid,
// the warps stride over the list four vertices at a time); v_c = hit point + eps
// n_f.  The correspondence is the first exit-face hit of the ray from the vertex
// along its negative area-weighted normal (3D-DDA over the face hash), the hit
// with the smallest (t, face id); without one, the closest point.
//
// What bounds it is FP64: an FP64 instruction costs its scheduler 64 cycles in
// one lane as in thirty-two, and the normal, the walk's set-up, a ray-triangle
// test and the target are about 300 of them.  So four vertices share each of
// those phases: a vertex's lanes take its incident faces, then its axes; the
// teams walk their cells with the FP32 test alone, which also bounds the first
// hit from above and so ends most walks, and then meet for the FP64 test of all
// teams' candidates.
// Measured, one warp per vertex with the FP64 test on every face, and this: 370 and
// 121 us for the 22,400 casts of a 983,040-tet finger, 67 and 43 us for the 4,300
// of the gripper.  (Meeting for FP64 at every cell with a face that passed: 48 us
// there; reading eight cells' ranges of the walk ahead: 50 us.)
template <typename T>
__global__ void __launch_bounds__(CAST_THREADS) k_cast(Dev<T> d) {
  __shared__ int shi[32];
  __shared__ FaceQueue s_queue[CAST_THREADS / 32];
  __shared__ int s_cand[CAST_THREADS / TEAM_LANES][3 * TEAM_LANES];
  int* const queue = s_cand[threadIdx.x / TEAM_LANES];
  constexpr unsigned FULL = 0xffffffffu;
  const int lane = threadIdx.x & 31, tl = lane & 7;
  const unsigned tmask = 0xFFu << (lane & 24);
  const int n_warps = gridDim.x * (CAST_THREADS / 32);
  const int n_cast = min(d.ctrl->n_cast, d.n_q);
  int active_out = 0;
  for (int j0 = 4 * (int)((blockIdx.x * (unsigned)CAST_THREADS + threadIdx.x) >> 5); j0 < n_cast; j0 += 4 * n_warps) {
    const int j = j0 + (lane >> 3);
    const bool valid = j < n_cast;
    const int qi = valid ? chk_idx(d.ctrl, d.cast_list[j], d.n_q) : 0;
    const int v = d.q_verts[qi];
    const int rv = d.robot_of_vert ? d.robot_of_vert[v] : 0;
    const R4<T> xv = d.X[v];
    const V3 o = {(double)xv.x, (double)xv.y, (double)xv.z};
    const V3 dir = cast_direction(d, qi);
    const float of[3] = {(float)xv.x, (float)xv.y, (float)xv.z};
    const float df[3] = {(float)dir.x, (float)dir.y, (float)dir.z};
    // DDA set-up: lane a < 3 of the team forms axis a's start cell, step, first
    // boundary parameter and increment, and its bound on the ray parameter from
    // the bounding box of this iteration's boundary faces (the ray can meet no
    // face beyond it)
    int cell[3], step[3];
    double tmax[3], tdel[3], tbox;
    {
      const double dva = tl == 0 ? dir.x : tl == 1 ? dir.y : dir.z;
      const double ova = tl == 0 ? o.x : tl == 1 ? o.y : o.z;
      int c_a = 0, st_a = 0;
      double tm_a = INFINITY, td_a = INFINITY, tb_a = INFINITY;
      if (tl < 3) {
        c_a = cell_coord(ova, d.inv_cell);
        if (dva > 0.0 || dva < 0.0) {
          const bool up = dva > 0.0;
          const double bound = up ? order_decode(d.ctrl->box_hi[tl]) + d.cell : order_decode(d.ctrl->box_lo[tl]) - d.cell;
          st_a = up ? 1 : -1;
          tm_a = ((up ? c_a + 1 : c_a) * d.cell - ova) / dva;
          td_a = (up ? d.cell : -d.cell) / dva;
          tb_a = (bound - ova) / dva;
        }
        // ray parameters of the walk are compared by their bit patterns below,
        // so they are made non-negative: a start within rounding of a cell face
        // can give -0.0 or a tiny negative first boundary (either way the walk
        // first steps across it), and the walk starts inside the faces' box
        tm_a = tm_a > 0.0 ? tm_a : 0.0;
        tb_a = tb_a > 0.0 ? tb_a : 0.0;
      }
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        cell[k] = __shfl_sync(FULL, c_a, k, 8);
        step[k] = __shfl_sync(FULL, st_a, k, 8);
        tmax[k] = __shfl_sync(FULL, tm_a, k, 8);
        tdel[k] = __shfl_sync(FULL, td_a, k, 8);
      }
      const unsigned long long t0 = key_bits(__shfl_sync(FULL, tb_a, 0, 8)), t1 = key_bits(__shfl_sync(FULL, tb_a, 1, 8)),
                               t2 = key_bits(__shfl_sync(FULL, tb_a, 2, 8));
      tbox = __longlong_as_double((long long)min(t0, min(t1, t2)));
    }
    int best_f = -1;
    double best_t = 0.0, b1 = 0.0, b2 = 0.0;
    unsigned long long stop = key_bits(INFINITY);  // bits of a ray parameter beyond which no hit is the first
    bool walking = valid;             // team-uniform, like the walk's whole state
    int steps = 0, kk = 0, k1 = 0;    // cells left behind; the next entry of this cell and its end
    int nc = 0;                       // faces in the team's queue
    auto enter = [&]() {
      const int2 r = d.cell_range[hash_cell(cell[0], cell[1], cell[2], rv) & (d.H_f - 1u)];
      kk = r.x;
      k1 = min(r.y, d.cap_items);
    };
    if (walking) enter();
    for (;;) {
      // FP32 only, until each team is at the end of its walk or its queue is
      // full; the four go round together, so that their reads are in flight
      // together
      while (__any_sync(FULL, walking && nc <= 2 * TEAM_LANES)) {
        const bool on = walking && nc <= 2 * TEAM_LANES;
        int cand = -1;
        float t_max = INFINITY;
        if (on && kk < k1) {
          const int k = kk + tl;
          if (k < k1) {
            const int f = d.items[k];
            if (!d.robot_of_face || d.robot_of_face[f] == rv) {
              const int4 fv = chk_face(d.ctrl, d.faces[chk_idx(d.ctrl, f, d.n_f)], d.n_v);
              if (fv.x != v && fv.y != v && fv.z != v &&
                  face_may_hit(d.X[fv.x], d.X[fv.y], d.X[fv.z], of, df, t_max))
                cand = f;
            }
          }
          kk += 8;
        }
        const unsigned who = __ballot_sync(FULL, cand >= 0) & tmask;
        if (cand >= 0) queue[nc + __popc(who & ((1u << lane) - 1u))] = cand;
        nc += __popc(who);
        if (__any_sync(FULL, who != 0)) {
          if (cand < 0) t_max = INFINITY;
#pragma unroll
          for (int m = 4; m > 0; m >>= 1) t_max = fminf(t_max, __shfl_xor_sync(FULL, t_max, m));
          if (t_max < INFINITY) stop = min(stop, key_bits((double)t_max));
        }
        if (!on || kk < k1) continue;
        // the cell is done
        const unsigned long long m0 = key_bits(tmax[0]), m1 = key_bits(tmax[1]), m2 = key_bits(tmax[2]);
        const unsigned long long texit = m0 < m1 ? (m0 < m2 ? m0 : m2) : (m1 < m2 ? m1 : m2);
        if (stop < texit || texit >= key_bits(INFINITY) || texit > key_bits(tbox) || ++steps >= MAX_DDA_STEPS) {
          walking = false;
          continue;
        }
        if (m0 <= m1 && m0 <= m2) {
          cell[0] += step[0];
          tmax[0] += tdel[0];
        } else if (m1 <= m2) {
          cell[1] += step[1];
          tmax[1] += tdel[1];
        } else {
          cell[2] += step[2];
          tmax[2] += tdel[2];
        }
        enter();
      }
      __syncwarp();
      if (!__any_sync(FULL, nc > 0)) break;
      // all teams' queued faces, FP64
      const int take = min(nc, TEAM_LANES);
      const int f = tl < take ? queue[nc - 1 - tl] : -1;
      __syncwarp();
      nc -= take;
      int lf = -1;
      double lt = 0.0, l1 = 0.0, l2 = 0.0;
      if (f >= 0) {
        V3 q0, q1, q2;
        int4 fv;
        face_verts(d, f, q0, q1, q2, fv);
        if (dot(dir, cross(sub(q1, q0), sub(q2, q0))) > 0.0 && ray_tri(o, dir, q0, q1, q2, lt, l1, l2)) lf = f;
      }
      if (__any_sync(FULL, lf >= 0)) {
        team_argmin(lf, lt, l1, l2);
        if (lf >= 0 && (best_f < 0 || key_bits(lt) < key_bits(best_t) || (lt == best_t && lf < best_f))) {
          best_f = lf;
          best_t = lt;
          b1 = l1;
          b2 = l2;
          stop = min(stop, key_bits(best_t * (1.0 + 1e-9)));
        }
      }
    }
    // vertices without a hit, one after the other by the whole warp
    const bool missed = valid && best_f < 0;
    unsigned todo = __ballot_sync(FULL, missed && tl == 0);
    while (todo) {
      const int src = __ffs(todo) - 1;
      todo &= todo - 1;
      const V3 os = {__shfl_sync(FULL, o.x, src), __shfl_sync(FULL, o.y, src), __shfl_sync(FULL, o.z, src)};
      double c1, c2;
      const int f = closest_face_warp(d, s_queue[threadIdx.x >> 5], __shfl_sync(FULL, v, src), __shfl_sync(FULL, rv, src), os, c1, c2);
      if ((lane & 24) == (src & 24)) {
        best_f = f;
        b1 = c1;
        b2 = c2;
      }
    }
    if (valid && tl == 0) active_out += finish_cast(d, qi, v, rv, best_f, missed, b1, b2);
  }
  const int ns = block_sum_int(active_out, shi);
  if (threadIdx.x == 0 && ns) atomicAdd(&(d.hist + (d.ctrl->iter % d.hist_cap))->n_springs, ns);
}

// Self springs of the listed vertices with the robot's face tree (broad phase 1),
// eight lanes per vertex and the same results as k_cast: the first exit-face hit
// (smallest t, then the lowest face id); without one, the closest point of the
// faces not containing v (smallest squared distance, then the lowest face id).
template <typename T>
__global__ void __launch_bounds__(NARROW_BVH_THREADS, 3) k_cast_bvh(Dev<T> d) {
  constexpr unsigned FULL = 0xffffffffu;
  __shared__ int shi[32];
  __shared__ TeamStack s_stack[NARROW_BVH_THREADS / TEAM_LANES];
  const int lane = threadIdx.x & 31, tl = lane & (TEAM_LANES - 1);
  TeamStack& stack = s_stack[threadIdx.x / TEAM_LANES];
  const int n_warps = gridDim.x * (NARROW_BVH_THREADS / 32);
  const int n_cast = min(d.ctrl->n_cast, d.n_q);
  const BvhDev& b = d.bf;
  int active_out = 0;
  for (int j0 = 4 * (int)((blockIdx.x * (unsigned)NARROW_BVH_THREADS + threadIdx.x) >> 5); j0 < n_cast;
       j0 += 4 * n_warps) {
    const int j = j0 + (lane >> 3);
    const bool valid = j < n_cast;
    const int qi = valid ? chk_idx(d.ctrl, d.cast_list[j], d.n_q) : 0;
    const int v = d.q_verts[qi];
    const int rv = d.robot_of_vert ? d.robot_of_vert[v] : 0;
    const R4<T> xv = d.X[v];
    const V3 x = {(double)xv.x, (double)xv.y, (double)xv.z};
    const V3 dir = cast_direction(d, qi);
    const float of[3] = {(float)xv.x, (float)xv.y, (float)xv.z};
    const float df[3] = {(float)dir.x, (float)dir.y, (float)dir.z};
    RayF ray;
    ray.o = pt_f(x.x, x.y, x.z);
#pragma unroll
    for (int a = 0; a < 3; ++a) ray.inv[a] = df[a] != 0.0f ? 1.0f / df[a] : INFINITY;
    const int root = b.n > 0 ? (b.root ? b.root[rv] : 0) : BVH_EMPTY;
    int bf = -1;
    double bt = 0.0, b1 = 0.0, b2 = 0.0;
    auto other = [&](int f, int4& fv) {  // a face of this robot without v
      if (d.robot_of_face && d.robot_of_face[f] != rv) return false;
      fv = chk_face(d.ctrl, d.faces[f], d.n_v);
      return fv.x != v && fv.y != v && fv.z != v;
    };
    team_search(
        b, root, valid, stack, bf, bt, b1, b2, [&](float4 lo, float4 hi) { return ray_box_t(lo, hi, ray); },
        [&](int f, float&, float& ub) {
          int4 fv;
          return other(f, fv) && face_may_hit(d.X[fv.x], d.X[fv.y], d.X[fv.z], of, df, ub);
        },
        [&](int f, double& key, double& e1, double& e2) {
          V3 q0, q1, q2;
          int4 fv;
          face_verts(d, f, q0, q1, q2, fv);
          return dot(dir, cross(sub(q1, q0), sub(q2, q0))) > 0.0 && ray_tri(x, dir, q0, q1, q2, key, e1, e2);
        },
        // (the box tests of the ray are accurate to a margin)
        [](double best) { return __double2float_ru(best * (1.0 + 1e-6) + 1e-9); }, 1.0001f);
    const bool missed = valid && bf < 0;
    if (__any_sync(FULL, missed))
      team_search(
          b, root, missed, stack, bf, bt, b1, b2, [&](float4 lo, float4 hi) { return box_d2(lo, hi, ray.o); },
          [&](int f, float& lb, float& ub) {
            int4 fv;
            if (!other(f, fv)) return false;
            triangle_bounds_at(d.X[fv.x], d.X[fv.y], d.X[fv.z], xv, lb, ub);
            return true;
          },
          [&](int f, double& key, double& e1, double& e2) {
            V3 q0, q1, q2;
            int4 fv;
            face_verts(d, f, q0, q1, q2, fv);
            const V3 dd = sub(x, closest_tri(x, q0, q1, q2, e1, e2));
            key = dot(dd, dd);
            return true;
          },
          [](double best) { return __double2float_ru(best); });
    if (valid && tl == 0) active_out += finish_cast(d, qi, v, rv, bf, missed, b1, b2);
  }
  const int ns = block_sum_int(active_out, shi);
  if (threadIdx.x == 0 && ns) atomicAdd(&(d.hist + (d.ctrl->iter % d.hist_cap))->n_springs, ns);
}

// ---- launchers ----
template <typename T>
void launch_bvh_refit(const BvhDev& b, const R4<T>* X, cudaStream_t st) {
  if (b.n < 2 || !b.flag) return;
  cudaMemsetAsync(b.flag, 0, sizeof(int) * (size_t)(b.n - 1), st);
  k_bvh_refit<T><<<(b.n + 255) / 256, 256, 0, st>>>(b, X);
}

// First of the broad phase; both sides below follow it.
template <typename T>
void launch_broad_clear(const Dev<T>& d, const CollisionScratch& cs, cudaStream_t st) {
  if (d.broad != 1) cudaMemsetAsync(cs.zero, 0, cs.zero_bytes, st);
}

// Face side, read by the ray casts alone.
template <typename T>
void launch_faces(const Dev<T>& d, cudaStream_t st) {
  if (d.broad == 1) {
    launch_bvh_refit<T>(d.bf, d.X, st);
    return;
  }
  if (d.n_f <= 0) return;
  const int nb = (d.n_f + FACE_THREADS - 1) / FACE_THREADS;
  k_faces<T, false><<<nb, FACE_THREADS, 0, st>>>(d);
  k_place_cells<T><<<((int)d.H_f + SCAN_TILE - 1) / SCAN_TILE, SCAN_THREADS, 0, st>>>(d);
  k_faces<T, true><<<nb, FACE_THREADS, 0, st>>>(d);
}

// Narrow phase over the tets once the query vertices are in their lists.
template <typename T>
void launch_tets(const Dev<T>& d, bool check, cudaStream_t st) {
  // a warp works off what its tets' boxes hold in rounds, so a mesh that would
  // leave the device half empty gets warps with fewer tets: 8 or 16 as long as all
  // warps run at once (32 of them on each of about 150 processors).  32 tets to a
  // warp and this: 15.1 and 10.9 us for 1,920 tets (22.2 and 15.6 in the
  // allocation-free check), 37.4 and 32.2 us for 51,840 in FP64; at 193,920 and
  // above it is the same.
  constexpr int ONE_WAVE = 4800;
  int per = 8;
  while (per < 32 && d.n_t > per * ONE_WAVE) per *= 2;
  const int bs = d.narrow_threads > 0 ? std::min(d.narrow_threads, TETS_MAX_THREADS) : TETS_MAX_THREADS;
  const int tets = bs / 32 * per, nb = (d.n_t + tets - 1) / tets;
  if (check)
    k_tets<T, true><<<nb, bs, 0, st>>>(d, per);
  else
    k_tets<T, false><<<nb, bs, 0, st>>>(d, per);
}

// A caller's positions into the kernels' layout, and its query vertices, whose
// ids are tested first, into their lists.
__global__ void __launch_bounds__(QUERY_THREADS) k_pack_queries(Dev<float> d, const float* __restrict__ xyz,
                                                                R4<float>* __restrict__ X) {
  const int i = blockIdx.x * QUERY_THREADS + threadIdx.x;
  if (i < d.n_v) X[i] = R4<float>{xyz[3 * i], xyz[3 * i + 1], xyz[3 * i + 2], 0.0f};
  if (i < d.n_q) {
    const int v = d.q_verts[i];
    if (v < 0 || v >= d.n_v) set_status(d.ctrl, ST_BAD_INPUT);
    else bin_query(d, i, v, 0, R4<float>{xyz[3 * v], xyz[3 * v + 1], xyz[3 * v + 2], 0.0f});
  }
}

void launch_pack_queries(const Dev<float>& d, const float* xyz, R4<float>* X, cudaStream_t st) {
  k_pack_queries<<<(std::max(d.n_v, d.n_q) + QUERY_THREADS - 1) / QUERY_THREADS, QUERY_THREADS, 0, st>>>(d, xyz, X);
}

// Pairs and obstacle contacts.
template <typename T>
void launch_collision(const Dev<T>& d, cudaStream_t st) {
  if (d.broad == 1) {
    // AABB tree: refit the tet tree to this iteration's positions
    launch_bvh_refit<T>(d.bt, d.X, st);
    const int per_block = NARROW_BVH_THREADS / TEAM_LANES;
    k_narrow_bvh<T><<<(d.n_q + per_block - 1) / per_block, NARROW_BVH_THREADS, 0, st>>>(d);
    return;
  }
  k_queries<T><<<(d.n_q + QUERY_THREADS - 1) / QUERY_THREADS, QUERY_THREADS, 0, st>>>(d);
  launch_tets<T>(d, false, st);
}

// The spring update, then the ray casts of the vertices it queued.
// These wait for faces_ready (unless null): the face side may be on a branch of
// its own.
template <typename T>
void launch_springs(const Dev<T>& d, cudaStream_t st, cudaEvent_t faces_ready) {
  if (d.n_q <= 0) return;
  k_springs<T><<<(d.n_q + 127) / 128, 128, 0, st>>>(d);
  const int teams = NARROW_BVH_THREADS / TEAM_LANES;
  if (d.obs_mesh && d.ot.n > 0) k_mesh_springs<T><<<(d.n_q + teams - 1) / teams, NARROW_BVH_THREADS, 0, st>>>(d);
  if (faces_ready) cudaStreamWaitEvent(st, faces_ready, 0);
  if (d.broad == 1) {
    k_cast_bvh<T><<<std::min((d.n_q + teams - 1) / teams, 1024), NARROW_BVH_THREADS, 0, st>>>(d);
    return;
  }
  // enough teams for one pass over a list of up to 32,768 casts
  const int per_block = CAST_THREADS / 8;
  const int blocks = std::min((d.n_q + per_block - 1) / per_block, 1024);
  k_cast<T><<<blocks, CAST_THREADS, 0, st>>>(d);
}
int scan_tiles(int n) { return (n + SCAN_TILE - 1) / SCAN_TILE; }

void launch_scan_exclusive(const int* in, int* out, int n, int* tile_sums, int* total, cudaStream_t st) {
  if (n <= 0) return;
  const int n_tiles = scan_tiles(n);
  k_scan_tiles<<<n_tiles, SCAN_THREADS, 0, st>>>(in, out, tile_sums, n);
  k_scan_top<<<1, 1024, 0, st>>>(tile_sums, n_tiles, total);
  k_scan_add<<<(n + 255) / 256, 256, 0, st>>>(out, tile_sums, n);
}

template void launch_bvh_refit<float>(const BvhDev&, const R4<float>*, cudaStream_t);
template void launch_bvh_refit<double>(const BvhDev&, const R4<double>*, cudaStream_t);
template void launch_broad_clear<float>(const Dev<float>&, const CollisionScratch&, cudaStream_t);
template void launch_broad_clear<double>(const Dev<double>&, const CollisionScratch&, cudaStream_t);
template void launch_collision<float>(const Dev<float>&, cudaStream_t);
template void launch_collision<double>(const Dev<double>&, cudaStream_t);
template void launch_tets<float>(const Dev<float>&, bool, cudaStream_t);
template void launch_faces<float>(const Dev<float>&, cudaStream_t);
template void launch_faces<double>(const Dev<double>&, cudaStream_t);
template void launch_springs<float>(const Dev<float>&, cudaStream_t, cudaEvent_t);
template void launch_springs<double>(const Dev<double>&, cudaStream_t, cudaEvent_t);

}  // namespace casim
