// Device view of a tabulated spacetree and the per-particle primitives of
// the PIT/PIDT step (arXiv:1508.02435): quantisation, descent of the
// flattened level-ordered table (the end state of the lifts and drops of
// Algorithm 1 / Theorem 1), the split-precision re-location, d-linear shape
// functions (Section 3) and leaf-corner to vertex maps.
//
// Device code is compiled with --fmad=false: every + - * / below is one IEEE
// round-to-nearest operation in program order.
#pragma once
#include <cstdint>

#include "tree.hpp"

namespace pic {

__constant__ uint32_t c_pow3[21];

// One plasma instance of a batch: its tree occupies the leaves, vertices and
// sort keys [*_off, *_off + count) of the concatenated arrays.  A single
// handle is a batch of one with every offset zero.
struct InstInfo {
  int32_t depth, M;            // uniform trees: level of every leaf, 3^depth
  int32_t leaf_off, vert_off, key_off, spread_off, tab_root, n_vert;
  int64_t poff;                // first particle of the instance in input order
  double q, ion, ion_load, diag;
  double h;                    // uniform trees: leaf width 3^-depth
  double jac[3];               // FP64 sweep: 1 - omega, -omega / diag times the face and edge / corner entries
  double rhs, rhs_lo;          // omega / diag in two doubles
  float q32, ion32, ion_load32, diag32, h32;
  float rdiag32, rdiag_lo32;   // 1 / diag32 in two floats
};

struct DevTree {
  int d, nch, nc, depth, uniform, scheme;
  int32_t n_inst;
  int32_t block_push, block_leaf, block_vert;  // threads per block (autotuned; 0 = 256)
  const InstInfo *inst;
  const int32_t *inst_of_leaf, *inst_of_vert;
  int64_t n_leaves, n_vert, n_pv, n_keys;
  int32_t M;  // 3^depth
  const TabEntry *tab;
  int32_t n_tab;
  // adaptive trees: the table entry of every cell of level jump_level (no leaf
  // is coarser), row-major; NULL where that level is the root
  const TabEntry *jump;
  int32_t jump_level, jump_cells;  // cells per axis: 3^jump_level
  int32_t resident;                // the solve runs as one cluster
  const int4 *leaf_rec;            // adaptive trees: leaf coordinates and level
  // uniform trees: spread[a * M + c] = base-3 digits of c interleaved on axis a,
  // so the depth-first leaf id of cell c is the sum over the axes
  const int32_t *spread;
  const uint8_t *leaf_level;
  const int32_t *leaf_coords;
  // adaptive grids
  const int32_t *cexp_ptr, *cexp_vid, *inc_ptr, *inc_lc, *dcnt, *corner_pv;
  const double *cexp_w64, *inc_w64, *ion64, *diag64;
  const float *cexp_w32, *inc_w32, *ion32, *diag32;
  // uniform grids
  double ion_u64, diag_u64;
  float ion_u32, diag_u32;
};

// 32 bytes in one store (eight floats, four doubles), to a 32-byte boundary: a
// whole sector, which two stores would write in two parts.
__device__ __forceinline__ void store32(float *p, const float *v) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
__device__ __forceinline__ void store32(double *p, const double *v) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(v[0]), "d"(v[1]), "d"(v[2]), "d"(v[3])
               : "memory");
}

// ---- quantisation ---------------------------------------------------------

__device__ __forceinline__ double wrap01(double x) {
  double y = x - floor(x);
  return y >= 1.0 ? 0.0 : y;
}

__device__ __forceinline__ uint32_t quantise(double y) {  // y already in [0,1)
  double s = y * 774840978.0;
  double f = floor(s);
  if (f < 0.0) f = 0.0;
  if (f > 774840977.0) f = 774840977.0;
  return (uint32_t)f;
}

// ---- descent ----------------------------------------------------------------

__device__ __forceinline__ int digit_q(const uint32_t Q[3], int d, int m) {
  uint32_t step = 2u * c_pow3[18 - m];
  int dg = (int)((Q[0] / step) % 3u) + 3 * (int)((Q[1] / step) % 3u);
  if (d == 3) dg += 9 * (int)((Q[2] / step) % 3u);
  return dg;
}

// Local depth-first index inside a complete subtree of depth k whose leaves
// have coordinates J (on the leaves' level): base-3^d digits, bottom-up.
__device__ __forceinline__ int32_t local_index(uint32_t J0, uint32_t J1, uint32_t J2, int d, int k) {
  int32_t local = 0, mul = 1, nch = d == 3 ? 27 : 9;
  for (int i = 0; i < k; ++i) {
    int dg = (int)(J0 % 3u) + 3 * (int)(J1 % 3u);
    if (d == 3) dg += 9 * (int)(J2 % 3u);
    J0 /= 3u; J1 /= 3u; J2 /= 3u;
    local += dg * mul;
    mul *= nch;
  }
  return local;
}

// Covering leaf of the quantised position Q (PIT owner, Theorem 1), from the
// table entry `root` of the instance's tree.
__device__ __forceinline__ int32_t descend_q(const TabEntry *tab, int d, const uint32_t Q[3], int *lev_out,
                                             int root = 0) {
  int ent = root, lev = 0;
  for (;;) {
    TabEntry e = tab[ent];
    if (e.a < 0) {
      int k = -e.a - 1;
      int L = lev + k;
      uint32_t step = 2u * c_pow3[18 - L];
      *lev_out = L;
      return e.b + local_index(Q[0] / step, Q[1] / step, d == 3 ? Q[2] / step : 0u, d, k);
    }
    ent = e.a + digit_q(Q, d, lev + 1);
    ++lev;
  }
}

__device__ __forceinline__ float clamp_off(float f) {
  const float one_minus = 0x1.fffffep-1f;
  return f < 0.0f ? 0.0f : (f > one_minus ? one_minus : f);
}

// ---- grid maps ---------------------------------------------------------------

// Row-major vertex ids of the 2^d corners of uniform-grid cell c (periodic).
__device__ __forceinline__ void uniform_corner_vertices(const int32_t *c, int d, int32_t M, int32_t *vid) {
  int32_t x0 = c[0], x1 = c[0] + 1 == M ? 0 : c[0] + 1;
  int32_t y0 = c[1] * M, y1 = (c[1] + 1 == M ? 0 : c[1] + 1) * M;
  vid[0] = x0 + y0; vid[1] = x1 + y0; vid[2] = x0 + y1; vid[3] = x1 + y1;
  if (d == 3) {
    int32_t z0 = c[2] * M * M, z1 = (c[2] + 1 == M ? 0 : c[2] + 1) * M * M;
    for (int e = 0; e < 4; ++e) { vid[e + 4] = vid[e] + z1; vid[e] += z0; }
  }
}

// Row-major vertex of corner e of the uniform-grid cell c (periodic).
__device__ __forceinline__ int32_t uniform_corner_vertex(const int32_t *c, int e, int d, int32_t M) {
  int64_t v = 0, mul = 1;
  for (int a = 0; a < d; ++a) {
    int32_t j = c[a] + ((e >> a) & 1);
    if (j >= M) j -= M;
    v += (int64_t)j * mul;
    mul *= M;
  }
  return (int32_t)v;
}

// Depth-first leaf id of cell c on a uniform tree (digit-interleave tables).
__device__ __forceinline__ int32_t uniform_leaf_of_cell(const int32_t *spread, int32_t M, const int32_t *c, int d) {
  int32_t l = __ldg(spread + c[0]) + __ldg(spread + M + c[1]);
  if (d == 3) l += __ldg(spread + 2 * M + c[2]);
  return l;
}

// d-linear shape function of corner e at local coordinates t.
template <typename T>
__device__ __forceinline__ T shape(const T *t, int e, int d) {
  T w = (T)1;
  for (int a = 0; a < d; ++a) {
    T f = ((e >> a) & 1) ? t[a] : (T)1 - t[a];
    w = w * f;
  }
  return w;
}

}  // namespace pic
