// CUDA kernels of the PIT/PIDT particle step for sm_103a (arXiv:1508.02435).
//
// Step structure (Section 3 PIC cycle + Section 5 re-binning):
//   deposit   k_leaf_partials -> k_vertex_charge -> k_sum_blocks        (item 1)
//   solve     k_rhs -> sweeps of uniform_solve / adaptive_solve / row_solve / resident_solve (auxiliary, item 2)
//   field     k_efield_uniform / k_efield_adaptive                      (item 3)
//   push      k_push64 / k_push32: gather E_i = R^T(x_i) E, leapfrog kick
//             and drift, wrap, re-location (descent / split resolve), new
//             key, moved flag (warp ballot), mover ranks                 (items 3-4)
//   re-bin    rebin.cuh: scans of the ballot words and of the keys -> k_place ->
//             k_sort_medium/large -> k_gather_* (stable: stayers first, then
//             movers in storage order)
//
// Determinism: no floating-point atomics.  Every sum has a fixed order (bucket
// order within a leaf, ascending leaf-corner order per vertex); integer atomics
// only count, and the one order they decide (mover ranks) is put right.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <utility>

#include "dev.cuh"
#include "launch.hpp"
#include "segsort.cuh"

namespace pic {

// Entry of the reference element's matrix for two corners that differ on k axes.
// Of the dimension alone: handles of both dimensions may be alive together.
template <int D>
__host__ __device__ constexpr double kref(int k) {
  return D == 2 ? (k == 0 ? 4.0 / 6.0 : k == 1 ? -1.0 / 6.0 : -2.0 / 6.0)
                : (k == 0 ? 4.0 / 12.0 : k == 1 ? 0.0 : -1.0 / 12.0);
}

__constant__ double c_width64[19];  // 3^-level
__constant__ float c_width32[19];

constexpr int kBlock = 256;
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 8;
constexpr int kScanTile = kScanThreads * kScanItems;
static_assert(kScanTile == kScanTileElems, "scan tile size disagrees with launch.hpp");

static std::atomic<int64_t> g_launches{0};
int64_t launches() { return g_launches.load(); }
void count_launches(int64_t k) { g_launches.fetch_add(k); }
#define COUNT(k) g_launches.fetch_add(k)

static inline int bsz(int32_t b) { return b > 0 ? b : kBlock; }

static inline unsigned grid_for(int64_t n, int block = kBlock) {
  int64_t g = (n + block - 1) / block;
  if (g < 1) g = 1;
  return (unsigned)g;
}

// ---------------------------------------------------------------------------
// tree view helpers
// ---------------------------------------------------------------------------

__device__ __forceinline__ void leaf_info(const DevTree &t, int32_t L, int *lev, int32_t *c) {
  *lev = t.leaf_level[L];
  for (int a = 0; a < t.d; ++a) c[a] = t.leaf_coords[(int64_t)L * t.d + a];
}

__device__ __forceinline__ const InstInfo &inst_of_leaf(const DevTree &t, int32_t L) {
  return t.inst[t.n_inst > 1 ? t.inst_of_leaf[L] : 0];
}
__device__ __forceinline__ const InstInfo &inst_of_vertex(const DevTree &t, int64_t v) {
  return t.inst[t.n_inst > 1 ? t.inst_of_vert[v] : 0];
}

// Global vertex ids of the corners of uniform-grid cell c of instance I.
template <typename Grid>
__device__ __forceinline__ void corner_vertices(const Grid &I, const int32_t *c, int d, int32_t *vid) {
  uniform_corner_vertices(c, d, I.M, vid);
  for (int e = 0; e < (1 << d); ++e) vid[e] += I.vert_off;
}

// PIDT owner vertex of corner a of leaf L (uniform grids: the FE vertex).
__device__ __forceinline__ int32_t pidt_vertex(const DevTree &t, int32_t L, int a) {
  if (t.uniform) {
    int32_t c[3] = {0, 0, 0};
    for (int k = 0; k < t.d; ++k) c[k] = t.leaf_coords[(int64_t)L * t.d + k];
    int32_t vid[8];
    corner_vertices(inst_of_leaf(t, L), c, t.d, vid);
    return vid[a];
  }
  return t.corner_pv[(int64_t)L * t.nc + a];
}

// Sort key of a particle in leaf L owned through corner a: PIT = leaf; PIDT =
// owner vertex * 2^d + quadrant of the leaf seen from the vertex.
__device__ __forceinline__ int32_t key_of(const DevTree &t, int32_t L, int a) {
  if (t.scheme == 0) return L;
  return pidt_vertex(t, L, a) * t.nc + (t.nc - 1 - a);
}

// Value of a vertex field at corner e of leaf L (hanging corners interpolated
// from their masters, in ascending master order).
__device__ __forceinline__ double corner_value(const DevTree &t, int32_t L, const int32_t *c, int e,
                                               const double *F) {
  if (t.uniform) return F[inst_of_leaf(t, L).vert_off + uniform_corner_vertex(c, e, t.d, inst_of_leaf(t, L).M)];
  int64_t i = (int64_t)L * t.nc + e;
  double s = 0.0;
  for (int32_t j = t.cexp_ptr[i]; j < t.cexp_ptr[i + 1]; ++j) s = s + t.cexp_w64[j] * F[t.cexp_vid[j]];
  return s;
}

__device__ __forceinline__ float corner_value(const DevTree &t, int32_t L, const int32_t *c, int e,
                                              const float *F) {
  if (t.uniform) return F[inst_of_leaf(t, L).vert_off + uniform_corner_vertex(c, e, t.d, inst_of_leaf(t, L).M)];
  int64_t i = (int64_t)L * t.nc + e;
  float s = 0.0f;
  for (int32_t j = t.cexp_ptr[i]; j < t.cexp_ptr[i + 1]; ++j) s = s + t.cexp_w32[j] * F[t.cexp_vid[j]];
  return s;
}

__device__ __forceinline__ const double *inc_weights(const DevTree &t, double) { return t.inc_w64; }
__device__ __forceinline__ const float *inc_weights(const DevTree &t, float) { return t.inc_w32; }
__device__ __forceinline__ double ion_load(const DevTree &t, int64_t v, double) {
  return t.uniform ? inst_of_vertex(t, v).ion_load : t.ion64[v];
}
__device__ __forceinline__ float ion_load(const DevTree &t, int64_t v, float) {
  return t.uniform ? inst_of_vertex(t, v).ion_load32 : t.ion32[v];
}
__device__ __forceinline__ double diag_val(const DevTree &t, int64_t v, double) {
  return t.uniform ? inst_of_vertex(t, v).diag : t.diag64[v];
}
__device__ __forceinline__ float diag_val(const DevTree &t, int64_t v, float) {
  return t.uniform ? inst_of_vertex(t, v).diag32 : t.diag32[v];
}

// Block partial FP64 sums (fixed reduction tree) for deterministic totals.
__device__ __forceinline__ void block_sum_store(double v, double *block_out) {
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    int nw = blockDim.x >> 5;
    v = lane < nw ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) block_out[blockIdx.x] = v;
  }
}

__global__ void k_sum_blocks(const double *in, int64_t n, double *out) {
  double v = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) v += in[i];
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    v = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) *out = v;
  }
}

__device__ __forceinline__ void local_coords(const double *x, int64_t n, int64_t p, int lev, const int32_t *c,
                                             int d, double *tl) {
  double s = (double)c_pow3[lev];
  for (int a = 0; a < d; ++a) {
    double u = x[a * n + p] * s - (double)c[a];
    tl[a] = u < 0.0 ? 0.0 : (u > 1.0 ? 1.0 : u);
  }
}

// ---------------------------------------------------------------------------
// a8 solve (auxiliary): b = Q - (sum Q) integral(phi); damped Jacobi
// ---------------------------------------------------------------------------

// With scale, also omega / diag per vertex; with raw (FP64, uniform trees), b itself
// there and b times omega / diag, rounded once, in b: a rounded factor would shift
// the whole potential (field of 2D batches against plain 64-bit values, with the
// leaf width's rounding in k_efield_uniform: 2.8e-16 relative, 2.1e-16 so).
template <typename T>
__global__ void k_rhs(DevTree t, const T *Q, const double *total, T *b, T omega, T *scale, T *raw) {
  int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= t.n_vert) return;
  T tot = (T)(t.n_inst > 1 ? total[1 + t.inst_of_vert[v]] : *total);
  const T r = Q[v] - tot * ion_load(t, v, (T)0);
  if (raw) {
    const InstInfo &I = inst_of_vertex(t, v);
    b[v] = (T)fma((double)r, I.rhs, (double)r * I.rhs_lo);
  } else {
    b[v] = r;
  }
  if (raw) raw[v] = r;
  if (scale) scale[v] = omega / diag_val(t, v, (T)0);
}

}  // namespace pic

#include "uniform_solve.cuh"
#include "adaptive_solve.cuh"
#include "resident_solve.cuh"
#include "row_solve.cuh"
#include "relocate.cuh"

namespace pic {

// ---------------------------------------------------------------------------
// a1/a2 initial keys and split conversion
// ---------------------------------------------------------------------------

// Upper half of the leaf C of level lev that holds Q, per axis.
__device__ __forceinline__ int pidt_corner_q(const uint32_t *Q, const uint32_t *C, int lev, int d) {
  const uint32_t s = c_pow3[18 - lev];
  int a_idx = 0;
  for (int a = 0; a < d; ++a)
    if (Q[a] - C[a] * (2u * s) >= s) a_idx |= 1 << a;
  return a_idx;
}

__device__ __forceinline__ int pidt_corner_o(const float *o, int d) {
  int a_idx = 0;
  for (int a = 0; a < d; ++a)
    if (o[a] >= 0.5f) a_idx |= 1 << a;
  return a_idx;
}

// Instance of input particle p (binary search over the first particles).
__device__ __forceinline__ int inst_of_particle(const DevTree &t, int64_t p) {
  int lo = 0, hi = t.n_inst;
  while (hi - lo > 1) {
    int mid = (lo + hi) >> 1;
    if (t.inst[mid].poff <= p) lo = mid; else hi = mid;
  }
  return lo;
}

// FP64: wrap x in place, covering leaf and key.
__global__ void k_init64(DevTree t, double *x, int64_t n, int32_t *leaf, int32_t *key, int32_t *err) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int root = t.inst[inst_of_particle(t, p)].tab_root;
  uint32_t Q[3] = {0u, 0u, 0u};
  for (int a = 0; a < t.d; ++a) {
    double xa = x[a * n + p];
    if (!isfinite(xa)) { atomicOr(err, 1); xa = 0.0; }
    double y = wrap01(xa);
    x[a * n + p] = y;
    Q[a] = quantise(y);
  }
  int lev;
  uint32_t C[3] = {0u, 0u, 0u};
  const int32_t L = t.d == 3 ? locate_q<3>(t, Q, root, &lev, C) : locate_q<2>(t, Q, root, &lev, C);
  leaf[p] = L;
  key[p] = key_of(t, L, pidt_corner_q(Q, C, lev, t.d));
}

// Split: leaf by the FP64 owner, o = RN32(clamp(RN64(x 3^l) - c)), v = RN32(v).
__global__ void k_init32(DevTree t, const double *x, const double *v, int64_t n, int32_t *leaf, float *o,
                         float *vf, int32_t *key, int32_t *err) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int root = t.inst[inst_of_particle(t, p)].tab_root;
  uint32_t Q[3] = {0u, 0u, 0u};
  double y[3] = {0.0, 0.0, 0.0};
  for (int a = 0; a < t.d; ++a) {
    double xa = x[a * n + p];
    if (!isfinite(xa) || !isfinite(v[a * n + p])) { atomicOr(err, 1); xa = 0.0; }
    y[a] = wrap01(xa);
    Q[a] = quantise(y[a]);
  }
  int lev;
  uint32_t C[3] = {0u, 0u, 0u};
  const int32_t L = t.d == 3 ? locate_q<3>(t, Q, root, &lev, C) : locate_q<2>(t, Q, root, &lev, C);
  leaf[p] = L;
  double s = (double)c_pow3[lev];
  float oo[3] = {0.f, 0.f, 0.f};
  for (int a = 0; a < t.d; ++a) {
    double u = y[a] * s - (double)t.leaf_coords[(int64_t)L * t.d + a];
    if (u < 0.0) u = 0.0;
    oo[a] = clamp_off((float)u);
    o[a * n + p] = oo[a];
    vf[a * n + p] = (float)v[a * n + p];
  }
  key[p] = key_of(t, L, pidt_corner_o(oo, t.d));
}

// ---------------------------------------------------------------------------
// a6 stable counting sort
// ---------------------------------------------------------------------------

constexpr int kMedSeg = 1024;        // longest segment one warp sorts in shared memory
constexpr int kMedThreads = 256;
constexpr unsigned kMedBlocks = 7 * 152;  // as many as fit the SMs' shared memory
constexpr int kLargeSeg = 16384;     // chunk of a long segment sorted in shared memory
constexpr int kLargeThreads = 1024;

}  // namespace pic

#include "rebin.cuh"

namespace pic {

// ---------------------------------------------------------------------------
// a3 + a4 + a1/a2 + a5: fused gather, push, re-location, key, moved flag
// ---------------------------------------------------------------------------

// Adds to count[key] the length of every run of equal keys in adjacent
// active lanes, one atomic per run (particles in bucket order mostly share
// their new bucket with their neighbours; equal keys apart count as separate
// runs).  Active lanes are a prefix of the warp or all of it.
__device__ __forceinline__ void add_runs(int32_t *count, int32_t key, bool act) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int32_t prev = __shfl_up_sync(full, key, 1);
  const unsigned acts = __ballot_sync(full, act);
  const bool head = act && (lane == 0 || prev != key);
  const unsigned heads = __ballot_sync(full, head);
  if (head) {
    const unsigned after = ~((2u << lane) - 1u);  // lanes above this one (none for lane 31)
    const unsigned stop = (heads | ~acts) & after;
    const int end = stop ? __ffs(stop) - 1 : 32;
    atomicAdd(&count[key], end - lane);
  }
}

}  // namespace pic

#include "push.cuh"
#include "deposit.cuh"

namespace pic {

// ---------------------------------------------------------------------------
// misc
// ---------------------------------------------------------------------------

__global__ void k_absolute_split(DevTree t, const int32_t *leaf, const float *o, int64_t n, double *x) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  int32_t L = leaf[p];
  int lev = t.leaf_level[L];
  double s = (double)c_pow3[lev];
  for (int a = 0; a < t.d; ++a)
    x[a * n + p] = ((double)t.leaf_coords[(int64_t)L * t.d + a] + (double)o[a * n + p]) / s;
}

__global__ void k_widen(const float *in, int64_t n, double *out) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = (double)in[i];
}

__global__ void k_half_kick64(const double *Ep, int64_t n, double c, double *v) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) v[i] = v[i] - c * Ep[i];
}

__global__ void k_half_kick32(const float *Ep, int64_t n, float c, float *v) {
  int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) v[i] = v[i] - c * Ep[i];
}

// Gather only (leapfrog start): E at the particles, [d][n].
__global__ void k_gather_only64(DevTree t, const double *x, const int32_t *leaf, int64_t n, const double *Ev,
                                double *Ep) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  int32_t L = leaf[p];
  int lev;
  int32_t c[3] = {0, 0, 0};
  leaf_info(t, L, &lev, c);
  double tl[3];
  local_coords(x, n, p, lev, c, t.d, tl);
  double E[3] = {0.0, 0.0, 0.0};
  for (int e = 0; e < t.nc; ++e) {
    double w = shape<double>(tl, e, t.d);
    for (int ax = 0; ax < t.d; ++ax) E[ax] = E[ax] + w * corner_value(t, L, c, e, Ev + ax * t.n_vert);
  }
  for (int ax = 0; ax < t.d; ++ax) Ep[ax * n + p] = E[ax];
}

__global__ void k_gather_only32(DevTree t, const float *o, const int32_t *leaf, int64_t n, const float *Ev,
                                float *Ep) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  int32_t L = leaf[p];
  int lev;
  int32_t c[3] = {0, 0, 0};
  leaf_info(t, L, &lev, c);
  float tl[3] = {0.f, 0.f, 0.f};
  for (int a = 0; a < t.d; ++a) tl[a] = o[a * n + p];
  float E[3] = {0.f, 0.f, 0.f};
  for (int e = 0; e < t.nc; ++e) {
    float w = shape<float>(tl, e, t.d);
    for (int ax = 0; ax < t.d; ++ax) E[ax] = E[ax] + w * corner_value(t, L, c, e, Ev + ax * t.n_vert);
  }
  for (int ax = 0; ax < t.d; ++ax) Ep[ax * n + p] = E[ax];
}

// ---------------------------------------------------------------------------
// a9 re-refinement: depth-first cell index on the finest admissible level
// ---------------------------------------------------------------------------

// Counts of level m at count + coff[m].
struct AdaptCheck {
  int32_t *count;
  int64_t coff[11];
  int dmin, dmax;
  int64_t ppc;
};

// Particles per cell of level m (depth-first cell index): the cell of the
// quantised position (FP64), or of leaf + offset, whose digits below the leaf
// follow the drop rule of the split re-location.
template <int D>
__global__ void k_level_count64(const double *x, int64_t n, int m, int32_t *count) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = p < n;
  int32_t cell = -1;
  if (act) {
    uint32_t c[D];
#pragma unroll
    for (int a = 0; a < D; ++a) c[a] = div_pow3(quantise(x[a * n + p]) >> 1, 18 - m);
    cell = subtree_index<D>(c, m);
  }
  add_runs(count, cell, act);
}

template <int D>
__global__ void k_level_count32(DevTree t, const int32_t *leaf, const float *o, int64_t n, int m, int32_t *count) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = p < n;
  int32_t cell = -1;
  if (act) {
    const int32_t L = leaf[p];
    const int lev = t.leaf_level[L];
    uint32_t c[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      uint32_t I = (uint32_t)t.leaf_coords[(int64_t)L * D + a];
      if (lev >= m) {
        I = div_pow3(I, lev - m);
      } else {
        float f = o[a * n + p];
        for (int l = lev; l < m; ++l) {
          const float u = 3.0f * f;
          int dg = (int)floorf(u);
          dg = dg > 2 ? 2 : dg;
          f = clamp_off(u - (float)dg);
          I = 3u * I + (uint32_t)dg;
        }
      }
      c[a] = I;
    }
    cell = subtree_index<D>(c, m);
  }
  add_runs(count, cell, act);
}

// The same from the buckets, for the cells of the installed tree: every leaf's
// particles go to its cell on level min(its level, top).  (Cells below a leaf
// stay empty.)
template <int D>
__global__ void k_bucket_count(DevTree t, const int32_t *start, AdaptCheck ac, int top) {
  const int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (L >= t.n_leaves) return;
  int l;
  int32_t c[3] = {0, 0, 0};
  leaf_info(t, (int32_t)L, &l, c);
  const int m = l < top ? l : top;
  if (m < ac.dmin) return;
  int32_t cnt = 0;
  for (int a = 0; a < (t.scheme == 0 ? 1 : t.nc); ++a) {
    const int32_t k = key_of(t, (int32_t)L, a);
    cnt += start[k + 1] - start[k];
  }
  uint32_t C[D];
#pragma unroll
  for (int a = 0; a < D; ++a) C[a] = div_pow3((uint32_t)c[a], l - m);
  if (cnt) atomicAdd(&ac.count[ac.coff[m] + subtree_index<D>(C, m)], cnt);
}

__global__ void k_threshold_bits(const int32_t *count, int64_t ncells, int64_t ppc, uint32_t *bits) {
  int64_t wd = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (wd * 32 >= ncells) return;
  uint32_t b = 0;
  for (int i = 0; i < 32; ++i) {
    int64_t c = wd * 32 + i;
    if (c < ncells && count[c] > ppc) b |= 1u << i;
  }
  bits[wd] = b;
}

// Cell counts of one level from those of the level below: the sum over the
// 3^d children (child ch of cell c is cell c 3^d + ch).
// With `add`, to what the cell holds itself (a leaf on the coarser level).
__global__ void k_count_parent(const int32_t *fine, int64_t ncoarse, int nch, int32_t *coarse, bool add) {
  int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= ncoarse) return;
  int32_t t = add ? coarse[c] : 0;
  for (int ch = 0; ch < nch; ++ch) t += fine[c * nch + ch];
  coarse[c] = t;
}

// Whether the particles-per-cell criterion keeps the installed tree: every
// leaf on level l needs dmin <= l <= dmax and (l == dmax or its count <= ppc),
// every ancestor on levels dmin .. l-1 a count > ppc.  Any leaf that fails
// sets *changed.

__global__ void k_adapt_check(DevTree t, AdaptCheck ac, int32_t *changed) {
  const int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (L >= t.n_leaves) return;
  int l;
  int32_t c[3] = {0, 0, 0};
  leaf_info(t, (int32_t)L, &l, c);
  bool bad = l < ac.dmin || l > ac.dmax;
  for (int m = ac.dmin; !bad && m <= l && m < ac.dmax; ++m) {
    const uint32_t sh = c_pow3[l - m];
    const int32_t idx = local_index((uint32_t)c[0] / sh, (uint32_t)c[1] / sh, t.d == 3 ? (uint32_t)c[2] / sh : 0u,
                                    t.d, m);
    const int32_t cnt = ac.count[ac.coff[m] + idx];
    bad = m < l ? cnt <= ac.ppc : cnt > ac.ppc;
  }
  if (bad) *changed = 1;
}

// The same on a uniform tree of one instance, PIT: the leaves below any cell are
// contiguous, so its count is a difference of bucket offsets.
__global__ void k_adapt_check_uniform(DevTree t, const int32_t *__restrict__ start, AdaptCheck ac, int32_t *changed) {
  const int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (L >= t.n_leaves) return;
  const int l = t.depth;
  bool bad = l < ac.dmin || l > ac.dmax;
  int64_t width = 1;
  for (int m = l; !bad && m >= ac.dmin; --m) {
    if (m < ac.dmax) {
      const int64_t b = L / width * width;
      const int32_t cnt = start[b + width] - start[b];
      bad = m < l ? cnt <= ac.ppc : cnt > ac.ppc;
    }
    width *= t.nch;
  }
  if (bad) *changed = 1;
}

// Split particles of tree `from` re-located in tree `to` (same positions):
// the resolver of the split push with zero displacement.
__global__ void k_relocate32(DevTree from, DevTree to, const int32_t *leaf, const float *o, const float *v,
                             int64_t n, int32_t *leaf2, float *o2, float *v2) {
  int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int32_t L = leaf[p];
  const int lev = from.leaf_level[L];
  uint32_t I[3] = {0u, 0u, 0u};
  float f[3] = {0.f, 0.f, 0.f};
  for (int a = 0; a < from.d; ++a) {
    I[a] = (uint32_t)from.leaf_coords[(int64_t)L * from.d + a];
    f[a] = o[a * n + p];
  }
  float on[3] = {0.f, 0.f, 0.f};
  leaf2[p] = to.d == 3 ? locate_split<3>(to, lev, I, f, on, 0) : locate_split<2>(to, lev, I, f, on, 0);
  for (int a = 0; a < from.d; ++a) {
    o2[a * n + p] = on[a];
    v2[a * n + p] = v[a * n + p];
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------

cudaError_t set_constants(cudaStream_t s) {
  uint32_t p3[21];
  p3[0] = 1;
  for (int i = 1; i < 21; ++i) p3[i] = p3[i - 1] * 3u;
  double w64[19];
  float w32[19];
  for (int i = 0; i < 19; ++i) {
    w64[i] = 1.0 / (double)p3[i];
    w32[i] = (float)w64[i];
  }
  uint2 dv[19];
  double p64[19];
  for (int i = 0; i < 19; ++i) {
    uint32_t sh = 0;
    while ((p3[i] >> (sh + 1)) != 0u) ++sh;
    dv[i] = make_uint2((uint32_t)(((1ull << (31 + sh)) + p3[i] - 1) / p3[i]), sh);
    p64[i] = (double)p3[i];
  }
  cudaError_t ed = cudaMemcpyToSymbolAsync(c_div3, dv, sizeof(dv), 0, cudaMemcpyHostToDevice, s);
  if (ed == cudaSuccess) ed = cudaMemcpyToSymbolAsync(c_pow3_64, p64, sizeof(p64), 0, cudaMemcpyHostToDevice, s);
  if (ed != cudaSuccess) return ed;
  cudaError_t ew = cudaMemcpyToSymbolAsync(c_width64, w64, sizeof(w64), 0, cudaMemcpyHostToDevice, s);
  if (ew == cudaSuccess) ew = cudaMemcpyToSymbolAsync(c_width32, w32, sizeof(w32), 0, cudaMemcpyHostToDevice, s);
  if (ew != cudaSuccess) return ew;
  cudaError_t e = cudaFuncSetAttribute(k_sort_large, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)(sizeof(int32_t) * kLargeSeg));
  if (e != cudaSuccess) return e;
  e = cudaFuncSetAttribute(k_sort_medium, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)(sizeof(int32_t) * kMedSeg * (kMedThreads / 32)));
  if (e != cudaSuccess) return e;
  return cudaMemcpyToSymbolAsync(c_pow3, p3, sizeof(p3), 0, cudaMemcpyHostToDevice, s);
}

void launch_init64(const DevTree &t, double *x, int64_t n, int32_t *leaf, int32_t *key, int32_t *err,
                   cudaStream_t s) {
  if (n > 0) { COUNT(1); k_init64<<<grid_for(n), kBlock, 0, s>>>(t, x, n, leaf, key, err); }
}

void launch_init32(const DevTree &t, const double *x, const double *v, int64_t n, int32_t *leaf, float *o,
                   float *vf, int32_t *key, int32_t *err, cudaStream_t s) {
  if (n > 0) { COUNT(1); k_init32<<<grid_for(n), kBlock, 0, s>>>(t, x, v, n, leaf, o, vf, key, err); }
}

// Flag = 1 if keys are not in ascending order.
__global__ void k_check_sorted(const int32_t *key, int64_t n, int32_t *flag) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool bad = i + 1 < n && key[i] > key[i + 1];
  if (__syncthreads_or(bad) && threadIdx.x == 0) atomicOr(flag, 1);
}

void launch_check_sorted(const int32_t *key, int64_t n, int32_t *flag, cudaStream_t s) {
  if (n > 1) { COUNT(1); k_check_sorted<<<grid_for(n), kBlock, 0, s>>>(key, n, flag); }
}

void launch_adapt_bits(const DevTree &t, bool split, const void *pos, const int32_t *leaf, int64_t n, int dmin, int dmax,
                       int64_t ppc, int32_t *count, const int64_t *cnt_off, uint32_t *bits, const int64_t *bit_off,
                       cudaStream_t s) {
  if (dmax <= dmin) return;
  const int m0 = dmax - 1;
  int64_t ncells = 1;
  for (int m = 0; m < m0; ++m) ncells *= t.nch;
  int32_t *fine = count + cnt_off[m0];
  cudaMemsetAsync(fine, 0, sizeof(int32_t) * ncells, s);
  if (n > 0) {
    COUNT(1);
    const unsigned g = grid_for(n);
    if (split) {
      if (t.d == 3) k_level_count32<3><<<g, kBlock, 0, s>>>(t, leaf, (const float *)pos, n, m0, fine);
      else k_level_count32<2><<<g, kBlock, 0, s>>>(t, leaf, (const float *)pos, n, m0, fine);
    } else if (t.d == 3) {
      k_level_count64<3><<<g, kBlock, 0, s>>>((const double *)pos, n, m0, fine);
    } else {
      k_level_count64<2><<<g, kBlock, 0, s>>>((const double *)pos, n, m0, fine);
    }
  }
  for (int m = m0; m >= dmin; --m) {
    if (m < m0) {
      COUNT(1);
      k_count_parent<<<grid_for(ncells), kBlock, 0, s>>>(count + cnt_off[m + 1], ncells, t.nch, count + cnt_off[m], false);
    }
    COUNT(1);
    k_threshold_bits<<<grid_for((ncells + 31) / 32), kBlock, 0, s>>>(count + cnt_off[m], ncells, ppc,
                                                                    bits + bit_off[m]);
    ncells /= t.nch;
  }
}

void launch_adapt_check(const DevTree &t, const int32_t *start, int32_t *count, const int64_t *coff, int dmin, int dmax,
                        int64_t ppc, int32_t *changed, cudaStream_t s) {
  AdaptCheck ac{};
  ac.count = count;
  for (int m = 0; m <= dmax && m < 11; ++m) ac.coff[m] = coff[m];
  ac.dmin = dmin;
  ac.dmax = dmax;
  ac.ppc = ppc;
  if (t.n_leaves <= 0) return;
  const unsigned g = grid_for(t.n_leaves);
  if (t.uniform && t.scheme == 0) {
    COUNT(1);
    k_adapt_check_uniform<<<g, kBlock, 0, s>>>(t, start, ac, changed);
    return;
  }
  const int top = std::min(t.depth, dmax - 1);
  if (top >= dmin) {
    int64_t ncells = 1;
    for (int m = 0; m < top; ++m) ncells *= t.nch;
    cudaMemsetAsync(count + coff[dmin], 0, sizeof(int32_t) * (coff[top] + ncells - coff[dmin]), s);
    COUNT(1);
    if (t.d == 3) k_bucket_count<3><<<g, kBlock, 0, s>>>(t, start, ac, top);
    else k_bucket_count<2><<<g, kBlock, 0, s>>>(t, start, ac, top);
    for (int m = top - 1; m >= dmin; --m) {
      ncells /= t.nch;
      COUNT(1);
      k_count_parent<<<grid_for(ncells), kBlock, 0, s>>>(count + coff[m + 1], ncells, t.nch, count + coff[m], true);
    }
  }
  COUNT(1);
  k_adapt_check<<<g, kBlock, 0, s>>>(t, ac, changed);
}

void launch_relocate32(const DevTree &from, const DevTree &to, const int32_t *leaf, const float *o, const float *v,
                       int64_t n, int32_t *leaf2, float *o2, float *v2, cudaStream_t s) {
  if (n <= 0) return;
  COUNT(1);
  k_relocate32<<<grid_for(n), kBlock, 0, s>>>(from, to, leaf, o, v, n, leaf2, o2, v2);
}

// Sweeps on a uniform tree between V and Vtmp, then the residual's block sums from
// `raw` (FP64; FP32: b again); returns their number.
template <typename T, int D>
static int64_t sweep_uniform(const DevTree &t, const T *b, const T *raw, T *V, T *Vtmp, int sweeps, T omega, double *r2,
                             cudaStream_t s) {
  T *in = V, *out = Vtmp;
  for (int it = 0; it < sweeps; ++it) {
    launch_jacobi_uniform<T, D, false>(t, b, in, out, omega, nullptr, s);
    std::swap(in, out);
  }
  if (in != V) cudaMemcpyAsync(V, in, sizeof(T) * t.n_vert, cudaMemcpyDeviceToDevice, s);
  return launch_jacobi_uniform<T, D, true>(t, raw, V, nullptr, omega, r2, s);
}

// The same on an adaptive tree, V in place; part: one value per leaf corner.
template <typename T, int D>
static int64_t sweep_adaptive(const DevTree &t, const T *b, T *V, T *part, const T *scale, int sweeps, T omega,
                              double *r2, cudaStream_t s) {
  const dim3 gc(grid_for(t.n_leaves * t.nc)), gv(grid_for(t.n_vert)), block(kBlock);
  for (int it = 0; it <= sweeps; ++it) {
    COUNT(2);
    launch_pdl(k_corner_pass<T, D, true>, gc, block, s, t, V, part);
    if (it < sweeps) launch_pdl(k_vertex_pass<T, false>, gv, block, s, t, b, part, scale, V, omega, r2);
    else launch_pdl(k_vertex_pass<T, true>, gv, block, s, t, b, part, scale, V, omega, r2);
  }
  return gv.x;
}

template <typename T>
static void solve(const DevTree &t, const RowMatrix &A, const T *Q, const double *total, T *b, T *V, T *Vtmp, T *part,
                  int sweeps, T omega, double *block_sum, double *resid2, cudaStream_t s) {
  if (t.resident) {
    resident_solve<T>(false, t, Q, total, V, sweeps, omega, resid2, s);
    return;
  }
  // the FP64 two-pass solve of an adaptive tree leaves Vtmp free: it holds omega / diag
  T *scale = sizeof(T) == 8 && !t.uniform && !A.val ? Vtmp : nullptr;
  // FP64 sweeps of a uniform tree take b times omega / diag; the leaf corners' scratch keeps b for the residual
  T *raw = sizeof(T) == 8 && t.uniform ? part : nullptr;
  { COUNT(1); k_rhs<T><<<grid_for(t.n_vert), kBlock, 0, s>>>(t, Q, total, b, omega, scale, raw); }
  int64_t nb;
  if constexpr (sizeof(T) == 8) {
    if (A.val) {
      nb = t.d == 3 ? sweep_rows<3>(t, A, b, V, Vtmp, sweeps, block_sum, s)
                    : sweep_rows<2>(t, A, b, V, Vtmp, sweeps, block_sum, s);
      { COUNT(1); k_sum_blocks<<<1, 1024, 0, s>>>(block_sum, nb, resid2); }
      return;
    }
  }
  if (t.uniform)
    nb = t.d == 3 ? sweep_uniform<T, 3>(t, b, raw ? raw : b, V, Vtmp, sweeps, omega, block_sum, s)
                  : sweep_uniform<T, 2>(t, b, raw ? raw : b, V, Vtmp, sweeps, omega, block_sum, s);
  else
    nb = t.d == 3 ? sweep_adaptive<T, 3>(t, b, V, part, scale, sweeps, omega, block_sum, s)
                  : sweep_adaptive<T, 2>(t, b, V, part, scale, sweeps, omega, block_sum, s);
  { COUNT(1); k_sum_blocks<<<1, 1024, 0, s>>>(block_sum, nb, resid2); }
}

bool resident_solve_fits(const DevTree &t, bool split) {
  if (!t.uniform || t.n_inst > 1) return false;
  return split ? resident_solve<float>(true, t, nullptr, nullptr, nullptr, 0, 0.0f, nullptr, nullptr)
               : resident_solve<double>(true, t, nullptr, nullptr, nullptr, 0, 0.0, nullptr, nullptr);
}

void launch_solve(const DevTree &t, const RowMatrix &A, bool split, const void *Q, const double *total, void *b, void *V,
                  void *Vtmp, void *part, int sweeps, double omega, double *block_sum, double *resid2, cudaStream_t s) {
  if (split)
    solve<float>(t, A, (const float *)Q, total, (float *)b, (float *)V, (float *)Vtmp, (float *)part, sweeps,
                 (float)omega, block_sum, resid2, s);
  else
    solve<double>(t, A, (const double *)Q, total, (double *)b, (double *)V, (double *)Vtmp, (double *)part, sweeps,
                  omega, block_sum, resid2, s);
}

template <typename T>
static void efield(const DevTree &t, const T *V, T *E, T *part, cudaStream_t s) {
  const unsigned g = grid_for(t.n_vert), gc = grid_for(t.n_leaves * t.nc);
  COUNT(t.uniform ? 1 : 2);
  if (t.uniform) {
    if (t.d == 3) k_efield_uniform<3><<<g, kBlock, 0, s>>>(t, V, E);
    else k_efield_uniform<2><<<g, kBlock, 0, s>>>(t, V, E);
  } else if (t.d == 3) {
    k_corner_pass<T, 3, false><<<gc, kBlock, 0, s>>>(t, V, part);
    k_efield_adaptive<T, 3><<<g, kBlock, 0, s>>>(t, part, E);
  } else {
    k_corner_pass<T, 2, false><<<gc, kBlock, 0, s>>>(t, V, part);
    k_efield_adaptive<T, 2><<<g, kBlock, 0, s>>>(t, part, E);
  }
}

void launch_efield(const DevTree &t, bool split, const void *V, void *E, void *part, cudaStream_t s) {
  if (split) efield<float>(t, (const float *)V, (float *)E, (float *)part, s);
  else efield<double>(t, (const double *)V, (double *)E, (double *)part, s);
}

// Field at every leaf corner ([leaf][corner][axis]), expanded once per field
// instead of once per particle.
template <typename T, int D>
__global__ void k_corner_field(DevTree t, const T *__restrict__ E, T *__restrict__ Ec) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= t.n_leaves * t.nc) return;
  const T *w = corner_weights(t, (T)0);
  T q[D];
#pragma unroll
  for (int k = 0; k < D; ++k) q[k] = (T)0;
  for (int32_t j = t.cexp_ptr[i]; j < t.cexp_ptr[i + 1]; ++j) {
    const T wj = w[j];
    const T *e = E + t.cexp_vid[j];
#pragma unroll
    for (int k = 0; k < D; ++k) q[k] = q[k] + wj * e[k * t.n_vert];
  }
#pragma unroll
  for (int k = 0; k < D; ++k) Ec[i * D + k] = q[k];
}

size_t corner_field_bytes(const DevTree &t, bool split) {
  return (size_t)t.n_leaves * t.nc * t.d * (split ? sizeof(float) : sizeof(double));
}

void launch_corner_field(const DevTree &t, bool split, const void *E, void *Ec, cudaStream_t s) {
  const unsigned g = grid_for(t.n_leaves * t.nc);
  COUNT(1);
  if (split) {
    if (t.d == 3) k_corner_field<float, 3><<<g, kBlock, 0, s>>>(t, (const float *)E, (float *)Ec);
    else k_corner_field<float, 2><<<g, kBlock, 0, s>>>(t, (const float *)E, (float *)Ec);
  } else if (t.d == 3) {
    k_corner_field<double, 3><<<g, kBlock, 0, s>>>(t, (const double *)E, (double *)Ec);
  } else {
    k_corner_field<double, 2><<<g, kBlock, 0, s>>>(t, (const double *)E, (double *)Ec);
  }
}

// Coordinates and level of every leaf in one 16-byte record.
__global__ void k_leaf_records(DevTree t, int4 *rec) {
  const int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (L >= t.n_leaves) return;
  int lev;
  int32_t c[3] = {0, 0, 0};
  leaf_info(t, (int32_t)L, &lev, c);
  rec[L] = make_int4(c[0], c[1], c[2], lev);
}

void launch_leaf_records(const DevTree &t, int4 *rec, cudaStream_t s) {
  COUNT(1);
  k_leaf_records<<<grid_for(t.n_leaves), kBlock, 0, s>>>(t, rec);
}

void launch_push32(const DevTree &t, const Push32Args &a, cudaStream_t s) {
  COUNT(1);
  const unsigned b = bsz(t.block_push), g = grid_for(a.n, b);
  if (t.d == 3) {
    if (t.n_inst > 1) k_push32<3, true, true><<<g, b, 0, s>>>(t, a);
    else if (t.uniform) k_push32<3, true, false><<<g, b, 0, s>>>(t, a);
    else k_push32<3, false, false><<<g, b, 0, s>>>(t, a);
  } else {
    if (t.n_inst > 1) k_push32<2, true, true><<<g, b, 0, s>>>(t, a);
    else if (t.uniform) k_push32<2, true, false><<<g, b, 0, s>>>(t, a);
    else k_push32<2, false, false><<<g, b, 0, s>>>(t, a);
  }
}

void launch_push64(const DevTree &t, const Push64Args &a, cudaStream_t s) {
  COUNT(1);
  const unsigned b = bsz(t.block_push), g = grid_for(a.n, b);
  if (t.d == 3) {
    if (t.n_inst > 1) k_push64<3, true, true><<<g, b, 0, s>>>(t, a);
    else if (t.uniform) k_push64<3, true, false><<<g, b, 0, s>>>(t, a);
    else k_push64<3, false, false><<<g, b, 0, s>>>(t, a);
  } else {
    if (t.n_inst > 1) k_push64<2, true, true><<<g, b, 0, s>>>(t, a);
    else if (t.uniform) k_push64<2, true, false><<<g, b, 0, s>>>(t, a);
    else k_push64<2, false, false><<<g, b, 0, s>>>(t, a);
  }
}

void launch_jump_table(const DevTree &t, TabEntry *jump, cudaStream_t s) {
  COUNT(1);
  int64_t n = 1;
  for (int a = 0; a < t.d; ++a) n *= t.jump_cells;
  if (t.d == 3) k_jump_table<3><<<grid_for(n), kBlock, 0, s>>>(t.tab, t.jump_level, t.jump_cells, jump);
  else k_jump_table<2><<<grid_for(n), kBlock, 0, s>>>(t.tab, t.jump_level, t.jump_cells, jump);
}

// A given split state (leaf + offsets) as fresh particles, one pass: keys, ranks,
// whether the keys ascend, and what the gather reads -- in 3D the records, in 2D
// the rows (`given`: the state is in them already).  It is the only pass over the
// given arrays, which may be the caller's.  Flags leaves outside the tree and
// offsets outside [0,1), and stores them as 0: later passes index by both.
template <int D>
__global__ void k_fresh32(DevTree t, const int32_t *leaf, const float *o, const float *__restrict__ v,
                          int64_t n, int32_t *key /* may be leaf */, float4 *__restrict__ rec, StateRows r,
                          bool given, int32_t *count, uint32_t *words, int32_t *rank, int32_t *unsorted, int32_t *err) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = p < n;
  auto key_at = [&](int64_t q, float *oo, int32_t *L, bool *bad) {
    *L = leaf[q];
    if (*L < 0 || *L >= t.n_leaves) { *bad = true; *L = 0; }
#pragma unroll
    for (int a = 0; a < D; ++a) {
      oo[a] = o[a * n + q];
      if (!(oo[a] >= 0.0f && oo[a] < 1.0f)) { *bad = true; oo[a] = 0.0f; }
    }
    return key_of(t, *L, pidt_corner_o(oo, D));
  };
  int32_t k = 0, L = 0;
  bool bad = false;
  float oo[D];
  if (act) {
    k = key_at(p, oo, &L, &bad);
    key[p] = k;
    if (bad) atomicOr(err, 2);
    if (D == 3) {
      const float q[8] = {oo[0],    oo[1],    oo[D - 1], v[p], v[n + p], v[(D - 1) * n + p], __int_as_float(L),
                          __int_as_float(k)};
      store32((float *)(rec + 2 * p), q);
    }
    if ((D == 2 && !given) || bad) {
#pragma unroll
      for (int a = 0; a < D; ++a) r.o[a * n + p] = oo[a];
      if (r.leaf != key) r.leaf[p] = L;  // PIT keys are the leaves
    }
    if (D == 2 && !given) {
#pragma unroll
      for (int a = 0; a < D; ++a) r.v[a * n + p] = v[a * n + p];
    }
  }
  int32_t prev = __shfl_up_sync(0xffffffffu, k, 1);
  if ((threadIdx.x & 31) == 0 && act && p > 0) {
    float po[D];
    int32_t pl;
    bool pb = false;
    prev = key_at(p - 1, po, &pl, &pb);
  }
  const bool down = act && p > 0 && prev > k;
  if (__syncthreads_or(down) && threadIdx.x == 0) atomicOr(unsorted, 1);
  rank_movers<false>(p, act, k, count, words, rank);
}

void launch_fresh32(const DevTree &t, const int32_t *leaf, const float *o, const float *v, int64_t n, int32_t *key,
                    void *rec, const StateRows &r, bool given, int32_t *count, uint32_t *words, int32_t *rank,
                    int32_t *unsorted, int32_t *err, cudaStream_t s) {
  if (n <= 0) return;
  COUNT(1);
  if (t.d == 3)
    k_fresh32<3><<<grid_for(n), kBlock, 0, s>>>(t, leaf, o, v, n, key, (float4 *)rec, r, given, count, words, rank,
                                                  unsorted, err);
  else
    k_fresh32<2><<<grid_for(n), kBlock, 0, s>>>(t, leaf, o, v, n, key, (float4 *)rec, r, given, count, words, rank,
                                                  unsorted, err);
}

// Two offsets and two velocities of a 2D particle side by side.
__global__ void k_pack_rows(int64_t n, const float *__restrict__ o, const float *__restrict__ v,
                            float4 *__restrict__ quad) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p < n) quad[p] = make_float4(o[p], o[n + p], v[p], v[n + p]);
}

void launch_pack_rows(int64_t n, const float *o, const float *v, void *quad, cudaStream_t s) {
  if (n > 0) { COUNT(1); k_pack_rows<<<grid_for(n), kBlock, 0, s>>>(n, o, v, (float4 *)quad); }
}

// The rows of a state in records (3D, split).
__global__ void k_record_rows(int64_t n, const float *__restrict__ rec, StateRows r) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  float q[8];
  load32(rec + 8 * p, q);
#pragma unroll
  for (int k = 0; k < 3; ++k) r.o[k * n + p] = q[k];
#pragma unroll
  for (int k = 0; k < 3; ++k) r.v[k * n + p] = q[3 + k];
  r.leaf[p] = __float_as_int(q[6]);
}

void launch_record_rows(int64_t n, const void *rec, const StateRows &r, cudaStream_t s) {
  if (n > 0) { COUNT(1); k_record_rows<<<grid_for(n), kBlock, 0, s>>>(n, (const float *)rec, r); }
}

// Records of a fresh 3D state in rows: the gather then reads one 32- or 64-byte
// record per particle instead of seven or eight scattered values.
template <typename V, typename T>
__global__ void k_make_records(int64_t n, const T *x, const T *v, const int32_t *leaf, const int32_t *key, V *rec);
template <>
__global__ void k_make_records(int64_t n, const float *x, const float *v, const int32_t *leaf, const int32_t *key,
                               float4 *rec) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const float r[8] = {x[p],     x[n + p],     x[2 * n + p],           v[p],
                      v[n + p], v[2 * n + p], __int_as_float(leaf[p]), __int_as_float(key[p])};
  store32((float *)(rec + 2 * p), r);
}
template <>
__global__ void k_make_records(int64_t n, const double *x, const double *v, const int32_t *leaf, const int32_t *key,
                               double2 *rec) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const double r[8] = {x[p],     x[n + p],     x[2 * n + p], v[p],
                       v[n + p], v[2 * n + p], __longlong_as_double((long long)(((uint64_t)(uint32_t)key[p] << 32) |
                                                                                (uint32_t)leaf[p])),
                       0.0};
  store32((double *)(rec + 4 * p), r);
  store32((double *)(rec + 4 * p + 2), r + 4);
}

void launch_make_records(bool split, int64_t n, const void *x, const void *v, const int32_t *leaf, const int32_t *key,
                         void *rec, cudaStream_t s) {
  if (n <= 0) return;
  COUNT(1);
  if (split)
    k_make_records<float4, float><<<grid_for(n), kBlock, 0, s>>>(n, (const float *)x, (const float *)v, leaf, key,
                                                                 (float4 *)rec);
  else
    k_make_records<double2, double><<<grid_for(n), kBlock, 0, s>>>(n, (const double *)x, (const double *)v, leaf, key,
                                                                   (double2 *)rec);
}

void launch_absolute_split(const DevTree &t, const int32_t *leaf, const float *o, int64_t n, double *x,
                           cudaStream_t s) {
  if (n > 0) { COUNT(1); k_absolute_split<<<grid_for(n), kBlock, 0, s>>>(t, leaf, o, n, x); }
}

void launch_widen(const float *in, int64_t n, double *out, cudaStream_t s) {
  if (n > 0) { COUNT(1); k_widen<<<grid_for(n), kBlock, 0, s>>>(in, n, out); }
}

void launch_gather_only(const DevTree &t, bool split, const void *pos, const int32_t *leaf, int64_t n,
                        const void *Ev, void *Ep, cudaStream_t s) {
  if (n <= 0) return;
  if (split)
    { COUNT(1); k_gather_only32<<<grid_for(n), kBlock, 0, s>>>(t, (const float *)pos, leaf, n, (const float *)Ev, (float *)Ep); }
  else
    { COUNT(1); k_gather_only64<<<grid_for(n), kBlock, 0, s>>>(t, (const double *)pos, leaf, n, (const double *)Ev,
                                                   (double *)Ep); }
}

// ---------------------------------------------------------------------------
// Lift and drop counts of Algorithm 1 (diagnostic, PIT)
// ---------------------------------------------------------------------------

// The leaf of every particle before a step, by particle id.
__global__ void k_scatter_by_id(const int32_t *ids, const int32_t *leaf, int64_t n, int32_t *by_id) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (p >= n) return;
  const int32_t id = ids[p];
  if (id >= 0 && id < n) by_id[id] = leaf[p];
}

// True when the closed boxes of leaves L1 and L2 share a point (periodic),
// compared on the finer of the two levels.
__device__ __forceinline__ bool leaves_touch(const DevTree &t, int32_t L1, int32_t L2) {
  const int l1 = t.leaf_level[L1], l2 = t.leaf_level[L2];
  const int lm = l1 > l2 ? l1 : l2;
  const int64_t s1 = c_pow3[lm - l1], s2 = c_pow3[lm - l2], P = c_pow3[lm];
  for (int a = 0; a < t.d; ++a) {
    const int64_t lo1 = (int64_t)t.leaf_coords[(int64_t)L1 * t.d + a] * s1;
    const int64_t lo2 = (int64_t)t.leaf_coords[(int64_t)L2 * t.d + a] * s2;
    int64_t d12 = (lo2 - lo1) % P, d21 = (lo1 - lo2) % P;
    if (d12 < 0) d12 += P;
    if (d21 < 0) d21 += P;
    if (d12 > s1 && d21 > s2) return false;
  }
  return true;
}

// Warp sums of (lifts, drops, tunnellers) into counts[0..2].
__device__ __forceinline__ void add_counts(unsigned lifts, unsigned drops, unsigned tun, unsigned long long *counts) {
  for (int off = 16; off > 0; off >>= 1) {
    lifts += __shfl_down_sync(0xffffffffu, lifts, off);
    drops += __shfl_down_sync(0xffffffffu, drops, off);
    tun += __shfl_down_sync(0xffffffffu, tun, off);
  }
  if ((threadIdx.x & 31) == 0) {
    if (lifts) atomicAdd(&counts[0], (unsigned long long)lifts);
    if (drops) atomicAdd(&counts[1], (unsigned long long)drops);
    if (tun) atomicAdd(&counts[2], (unsigned long long)tun);
  }
}

// A particle that went from leaf L1 (level l1, coordinates c1) to leaf L2 is
// lifted out of every cell from L1 up to the deepest ancestor that contains
// L2, then dropped down to L2: lifts = l1 - m, drops = l2 - m with m the level
// of that ancestor (levels and coordinates of one instance's tree).  It
// tunnelled when L2 does not touch L1.  Warp sums go to counts[0] (lifts),
// counts[1] (drops) and counts[2] (tunnellers).
__global__ void k_lift_drop(DevTree t, const int32_t *ids, const int32_t *leaf, const int32_t *old_by_id, int64_t n,
                            unsigned long long *counts) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned lifts = 0, drops = 0, tun = 0;
  if (p < n) {
    const int32_t id = ids[p];
    const int32_t L2 = leaf[p];
    const int32_t L1 = (id >= 0 && id < n) ? old_by_id[id] : -1;
    if (L1 >= 0 && L1 < t.n_leaves && L2 >= 0 && L2 < t.n_leaves) {
      const int l1 = t.leaf_level[L1], l2 = t.leaf_level[L2];
      int m = l1 < l2 ? l1 : l2;
      uint32_t a1[3] = {0u, 0u, 0u}, a2[3] = {0u, 0u, 0u};
      for (int a = 0; a < t.d; ++a) {
        a1[a] = (uint32_t)t.leaf_coords[(int64_t)L1 * t.d + a] / c_pow3[l1 - m];
        a2[a] = (uint32_t)t.leaf_coords[(int64_t)L2 * t.d + a] / c_pow3[l2 - m];
      }
      while (m > 0 && (a1[0] != a2[0] || a1[1] != a2[1] || a1[2] != a2[2])) {
        for (int a = 0; a < 3; ++a) {
          a1[a] /= 3u;
          a2[a] /= 3u;
        }
        --m;
      }
      lifts = (unsigned)(l1 - m);
      drops = (unsigned)(l2 - m);
      tun = leaves_touch(t, L1, L2) ? 0u : 1u;
    }
  }
  add_counts(lifts, drops, tun, counts);
}

// Owner vertex (level, j) of PIDT key k (owner vertex id = k / 2^d): the
// finite-element vertex of a uniform tree (row-major on the finest level),
// else the owner-vertex table.
__device__ __forceinline__ int pidt_owner(const DevTree &t, const int32_t *pv_level, const int32_t *pv_j, int32_t k,
                                          int64_t *j) {
  const int32_t pv = k / t.nc;
  if (t.uniform) {
    int64_t v = pv;
    for (int a = 0; a < t.d; ++a) {
      j[a] = v % t.M;
      v /= t.M;
    }
    return t.depth;
  }
  for (int a = 0; a < t.d; ++a) j[a] = pv_j[(int64_t)pv * t.d + a];
  return pv_level[pv];
}

// Lifts and drops of PIDT (reading of Algorithms 2-3 as a count): a particle
// whose new owner is a vertex of its old leaf on that leaf's level is handed
// over inside the cell (none); any other is lifted from its old vertex to the
// deepest dual ancestor whose dual cell holds both owners' dual cells and
// dropped to the new owner, the dual parent of (l, j) being
// (l - 1, (j + 1) div 3).  Tunnellers as for PIT, from the leaves.
__global__ void k_lift_drop_pidt(DevTree t, const int32_t *pv_level, const int32_t *pv_j, const int32_t *ids,
                                 const int32_t *leaf, const int32_t *key, const int32_t *old_leaf_by_id,
                                 const int32_t *old_key_by_id, int64_t n, unsigned long long *counts) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  unsigned lifts = 0, drops = 0, tun = 0;
  if (p < n) {
    const int32_t id = ids[p];
    const int32_t L2 = leaf[p], k2 = key[p];
    const bool ok = id >= 0 && id < n;
    const int32_t L1 = ok ? old_leaf_by_id[id] : -1, k1 = ok ? old_key_by_id[id] : -1;
    if (L1 >= 0 && L1 < t.n_leaves && L2 >= 0 && L2 < t.n_leaves && k1 >= 0 && k1 < t.n_keys && k2 >= 0 &&
        k2 < t.n_keys) {
      tun = leaves_touch(t, L1, L2) ? 0u : 1u;
      if (k1 / t.nc != k2 / t.nc) {
        int64_t j1[3] = {0, 0, 0}, j2[3] = {0, 0, 0};
        const int l1 = pidt_owner(t, pv_level, pv_j, k1, j1);
        const int l2 = pidt_owner(t, pv_level, pv_j, k2, j2);
        const int ll = t.leaf_level[L1];
        const int64_t per = c_pow3[ll];
        bool handed = l2 == ll;
        for (int a = 0; a < t.d && handed; ++a) {
          int64_t r = (j2[a] - t.leaf_coords[(int64_t)L1 * t.d + a]) % per;
          if (r < 0) r += per;
          handed = r <= 1;
        }
        if (!handed) {
          int m = l1 < l2 ? l1 : l2;
          for (int l = l1; l > m; --l)
            for (int a = 0; a < t.d; ++a) j1[a] = ((j1[a] + 1) / 3) % (int64_t)c_pow3[l - 1];
          for (int l = l2; l > m; --l)
            for (int a = 0; a < t.d; ++a) j2[a] = ((j2[a] + 1) / 3) % (int64_t)c_pow3[l - 1];
          while (m > 0 && (j1[0] != j2[0] || j1[1] != j2[1] || j1[2] != j2[2])) {
            for (int a = 0; a < t.d; ++a) {
              j1[a] = ((j1[a] + 1) / 3) % (int64_t)c_pow3[m - 1];
              j2[a] = ((j2[a] + 1) / 3) % (int64_t)c_pow3[m - 1];
            }
            --m;
          }
          lifts = (unsigned)(l1 - m);
          drops = (unsigned)(l2 - m);
        }
      }
    }
  }
  add_counts(lifts, drops, tun, counts);
}

void launch_scatter_by_id(const int32_t *ids, const int32_t *leaf, int64_t n, int32_t *by_id, cudaStream_t s) {
  if (n > 0) { COUNT(1); k_scatter_by_id<<<grid_for(n), kBlock, 0, s>>>(ids, leaf, n, by_id); }
}

void launch_lift_drop(const DevTree &t, const int32_t *ids, const int32_t *leaf, const int32_t *old_by_id, int64_t n,
                      unsigned long long *counts, cudaStream_t s) {
  if (n > 0) { COUNT(1); k_lift_drop<<<grid_for(n), kBlock, 0, s>>>(t, ids, leaf, old_by_id, n, counts); }
}

void launch_lift_drop_pidt(const DevTree &t, const int32_t *pv_level, const int32_t *pv_j, const int32_t *ids,
                           const int32_t *leaf, const int32_t *key, const int32_t *old_leaf_by_id,
                           const int32_t *old_key_by_id, int64_t n, unsigned long long *counts, cudaStream_t s) {
  if (n > 0) {
    COUNT(1);
    k_lift_drop_pidt<<<grid_for(n), kBlock, 0, s>>>(t, pv_level, pv_j, ids, leaf, key, old_leaf_by_id, old_key_by_id,
                                                    n, counts);
  }
}

// ---------------------------------------------------------------------------
// raPIDT tree attribute v_max (Section 5.4)
// ---------------------------------------------------------------------------

// Per leaf: the largest velocity component magnitude of its particles -- PIT:
// the leaf's bucket; PIDT: the buckets of the leaf's 2^d vertices, i.e. every
// dual cell intersecting the leaf (the paper's definition).
template <typename T>
__global__ void k_leaf_vmax(DevTree t, const int32_t *__restrict__ start, const T *__restrict__ v, int64_t n,
                            double *leaf_vmax) {
  const int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (L >= t.n_leaves) return;
  double m = 0.0;
  const int na = t.scheme == 0 ? 1 : t.nc;
  for (int a = 0; a < na; ++a) {
    int32_t k0, k1;
    if (t.scheme == 0) {
      k0 = (int32_t)L;
      k1 = k0 + 1;
    } else {
      k0 = pidt_vertex(t, (int32_t)L, a) * t.nc;
      k1 = k0 + t.nc;
    }
    for (int32_t p = start[k0]; p < start[k1]; ++p)
      for (int ax = 0; ax < t.d; ++ax) {
        const double x = fabs((double)v[ax * n + p]);
        m = x > m ? x : m;
      }
  }
  leaf_vmax[L] = m;
}

// Per tree node of one level (level order): a leaf takes its leaf's value,
// a refined node the largest of its 3^d children's (Eq. v_max).
__global__ void k_node_vmax(const int32_t *child0, const int32_t *leaf_of_node, int64_t b, int64_t e, int nch,
                            const double *leaf_vmax, double *node_vmax) {
  const int64_t i = b + (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= e) return;
  if (leaf_of_node[i] >= 0) {
    node_vmax[i] = leaf_vmax[leaf_of_node[i]];
    return;
  }
  double m = 0.0;
  for (int k = 0; k < nch; ++k) {
    const double x = node_vmax[child0[i] + k];
    m = x > m ? x : m;
  }
  node_vmax[i] = m;
}

void launch_vmax(const DevTree &t, bool split, const int32_t *start, const void *v, int64_t n, const int32_t *child0,
                 const int32_t *leaf_of_node, const int64_t *level_begin, int depth, double *leaf_vmax,
                 double *node_vmax, cudaStream_t s) {
  COUNT(1);
  if (split)
    k_leaf_vmax<float><<<grid_for(t.n_leaves), kBlock, 0, s>>>(t, start, (const float *)v, n, leaf_vmax);
  else
    k_leaf_vmax<double><<<grid_for(t.n_leaves), kBlock, 0, s>>>(t, start, (const double *)v, n, leaf_vmax);
  for (int l = depth; l >= 0; --l) {
    const int64_t b = level_begin[l], e = level_begin[l + 1];
    if (e <= b) continue;
    COUNT(1);
    k_node_vmax<<<grid_for(e - b), kBlock, 0, s>>>(child0, leaf_of_node, b, e, t.nch, leaf_vmax, node_vmax);
  }
}

void launch_half_kick(bool split, const void *Ep, int64_t n_total, double c, void *v, cudaStream_t s) {
  if (n_total <= 0) return;
  if (split)
    { COUNT(1); k_half_kick32<<<grid_for(n_total), kBlock, 0, s>>>((const float *)Ep, n_total, (float)c, (float *)v); }
  else
    { COUNT(1); k_half_kick64<<<grid_for(n_total), kBlock, 0, s>>>((const double *)Ep, n_total, c, (double *)v); }
}

}  // namespace pic
