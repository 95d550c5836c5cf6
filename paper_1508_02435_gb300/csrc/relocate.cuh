// Re-location of a pushed particle: the covering leaf of its position (the end
// state of the lifts and drops of Algorithm 1 / Theorem 1) by a descent of the
// flattened table (included by kernels.cu).
//
// The descent starts at the jump table: the table entry of every cell of level
// t.jump_level, row-major, so that on an adaptive tree whose leaves differ by a
// level or two a particle reads one entry instead of one per level from the
// root.  Divisions by powers of three are multiplications by stored reciprocals
// (a division by a variable is some twenty instructions, three a level).
#pragma once

namespace pic {

__constant__ uint2 c_div3[19];       // x / 3^k = umulhi(2 x, c.x) >> c.y for x < 2^30
__constant__ double c_pow3_64[19];

__device__ __forceinline__ uint32_t div_pow3(uint32_t x, int k) {
  const uint2 m = c_div3[k];
  return __umulhi(2u * x, m.x) >> m.y;
}

// Depth-first index inside a complete subtree of depth k whose leaves have
// coordinates J on the leaves' level.
template <int D>
__device__ __forceinline__ int32_t subtree_index(const uint32_t *J, int k) {
  uint32_t r[D];
#pragma unroll
  for (int a = 0; a < D; ++a) r[a] = J[a];
  int32_t local = 0, mul = 1;
  for (int i = 0; i < k; ++i) {
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const uint32_t q = r[a] / 3u;
      local += (int32_t)(r[a] - 3u * q) * mul * (a == 0 ? 1 : a == 1 ? 3 : 9);
      r[a] = q;
    }
    mul *= D == 3 ? 27 : 9;
  }
  return local;
}

// The jump table's entry of cell J of its level.
template <int D>
__device__ __forceinline__ TabEntry jump_entry(const DevTree &t, const uint32_t *J) {
  const uint32_t g = (uint32_t)t.jump_cells;
  return t.jump[D == 3 ? J[0] + g * (J[1] + g * J[2]) : J[0] + g * J[1]];
}

// Covering leaf of the quantised position Q, from entry `root` of the
// instance's tree; C gets the leaf's coordinates.
template <int D>
__device__ __forceinline__ int32_t locate_q(const DevTree &t, const uint32_t *Q, int root, int *lev_out, uint32_t *C) {
  uint32_t H[D], J[D];
  int m = 0;
  TabEntry e;
#pragma unroll
  for (int a = 0; a < D; ++a) H[a] = Q[a] >> 1;
  if (t.jump) {
    m = t.jump_level;
#pragma unroll
    for (int a = 0; a < D; ++a) J[a] = div_pow3(H[a], 18 - m);
    e = jump_entry<D>(t, J);
  } else {
#pragma unroll
    for (int a = 0; a < D; ++a) J[a] = 0u;
    e = t.tab[root];
  }
  while (e.a >= 0) {
    ++m;
    int dg = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const uint32_t j = div_pow3(H[a], 18 - m);
      dg += (int)(j - 3u * J[a]) * (a == 0 ? 1 : a == 1 ? 3 : 9);
      J[a] = j;
    }
    e = t.tab[e.a + dg];
  }
  const int k = -e.a - 1, L = m + k;
  *lev_out = L;
#pragma unroll
  for (int a = 0; a < D; ++a) C[a] = div_pow3(H[a], 18 - L);
  return e.b + subtree_index<D>(C, k);
}

// One drop below the integer level: u = RN32(3 f), digit = min(floor u, 2),
// f = u - digit.
template <int D>
__device__ __forceinline__ int drop_digit(float *f) {
  int dg = 0;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const float u = 3.0f * f[a];
    int g = (int)floorf(u);
    g = g > 2 ? 2 : g;
    f[a] = clamp_off(u - (float)g);
    dg += g * (a == 0 ? 1 : a == 1 ? 3 : 9);
  }
  return dg;
}

// Split-precision re-location: the leaf covering integer cell I on level lev
// plus fraction f (used up).  Writes the leaf's offsets; returns the leaf.
template <int D>
__device__ __forceinline__ int32_t locate_split(const DevTree &t, int lev, const uint32_t *I, float *f, float *o_out,
                                                int root) {
  uint32_t J[D];
  int m = 0;
  TabEntry e;
  if (t.jump && lev >= t.jump_level) {
    m = t.jump_level;
#pragma unroll
    for (int a = 0; a < D; ++a) J[a] = div_pow3(I[a], lev - m);
    e = jump_entry<D>(t, J);
  } else {
#pragma unroll
    for (int a = 0; a < D; ++a) J[a] = 0u;
    e = t.tab[root];
  }
  auto digit = [&](int level) {  // of the cell on `level`; J moves there
    if (level > lev) return drop_digit<D>(f);
    int dg = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const uint32_t j = div_pow3(I[a], lev - level);
      dg += (int)(j - 3u * J[a]) * (a == 0 ? 1 : a == 1 ? 3 : 9);
      J[a] = j;
    }
    return dg;
  };
  while (e.a >= 0) {
    ++m;
    e = t.tab[e.a + digit(m)];
  }
  const int k = -e.a - 1, L = m + k;
  if (L == lev) {  // same level: the cell itself
#pragma unroll
    for (int a = 0; a < D; ++a) o_out[a] = clamp_off(f[a]);
    return e.b + subtree_index<D>(I, k);
  }
  if (L < lev) {  // lift
    const uint32_t sh = c_pow3[lev - L];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      J[a] = div_pow3(I[a], lev - L);
      o_out[a] = clamp_off(((float)(I[a] - J[a] * sh) + f[a]) / (float)sh);
    }
    return e.b + subtree_index<D>(J, k);
  }
  int32_t local = 0;  // digits from I down to lev, then drops from the fraction
  for (int level = m + 1; level <= L; ++level) local = local * (D == 3 ? 27 : 9) + digit(level);
#pragma unroll
  for (int a = 0; a < D; ++a) o_out[a] = clamp_off(f[a]);
  return e.b + local;
}

// The jump table: entry of every cell of level `level` (no leaf is coarser).
template <int D>
__global__ void k_jump_table(const TabEntry *tab, int level, int32_t cells, TabEntry *jump) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n = D == 3 ? (int64_t)cells * cells * cells : (int64_t)cells * cells;
  if (i >= n) return;
  uint32_t C[D], r = (uint32_t)i;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    C[a] = r % (uint32_t)cells;
    r /= (uint32_t)cells;
  }
  TabEntry e = tab[0];
  int m = 0;
  while (e.a >= 0 && m < level) {
    ++m;
    int dg = 0;
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const uint32_t j = div_pow3(C[a], level - m);
      dg += (int)(j % 3u) * (a == 0 ? 1 : a == 1 ? 3 : 9);
    }
    e = tab[e.a + dg];
  }
  if (e.a < 0) {  // inside a complete subtree: its part below this cell
    const int k = -e.a - 1 - (level - m);
    int32_t width = 1;
    for (int j = 0; j < k; ++j) width *= D == 3 ? 27 : 9;
    uint32_t J[D];
    const uint32_t sh = c_pow3[level - m];
#pragma unroll
    for (int a = 0; a < D; ++a) J[a] = C[a] % sh;
    e = TabEntry{-k - 1, e.b + subtree_index<D>(J, level - m) * width};
  }
  jump[i] = e;
}

}  // namespace pic
