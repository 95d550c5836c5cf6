// Jacobi sweeps and vertex field on adaptive trees (included by kernels.cu).
//
// A V is assembled in two passes: one thread per leaf corner expands the
// corner onto vertices once, and the 2^d lanes of a leaf exchange their values
// and form the leaf's product; one thread per vertex then adds the products of
// its incident leaf corners.  A single pass over the vertices would expand
// every corner once per corner of its leaf and incidence (4^d expansions a
// vertex instead of 2^d).  The order of every FP32 sum is that of the
// leaf-by-leaf assembly; FP64 uses fused multiply-adds.
//
// One sweep of the 1e6-particle bump (2D, 75,451 vertices, FP64): 64 -> 9.9 us, two
// dependent launches.  FP64 handles take assembled rows where row_solve.cuh has
// built them (3.8 us); FP32 sums must keep this order, so FP32 stays here.
#pragma once

namespace pic {

__device__ __forceinline__ double mul_add(double a, double b, double c) { return fma(a, b, c); }
__device__ __forceinline__ float mul_add(float a, float b, float c) { return c + a * b; }
__device__ __forceinline__ double cell_width(int lev, double) { return c_width64[lev]; }
__device__ __forceinline__ float cell_width(int lev, float) { return c_width32[lev]; }
__device__ __forceinline__ const double *corner_weights(const DevTree &t, double) { return t.cexp_w64; }
__device__ __forceinline__ const float *corner_weights(const DevTree &t, float) { return t.cexp_w32; }

// Per leaf corner i: the leaf's product sum_f K_ef h^(d-2) V(L, f) with
// kApply, else V itself expanded onto the corner.
template <typename T, int D, bool kApply>
__global__ void __launch_bounds__(256) k_corner_pass(DevTree t, const T *V, T *__restrict__ out) {
  constexpr int NC = 1 << D;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = i < t.n_leaves * NC;
  const int e = (int)threadIdx.x & (NC - 1);
  // the tables do not change: read, first entry included, while the pass before runs
  const T *w = corner_weights(t, (T)0);
  int32_t j0 = 0, j1 = 0, vid0 = 0;
  T c[NC], w0 = (T)0;
  if (act) {
    j0 = t.cexp_ptr[i];
    j1 = t.cexp_ptr[i + 1];
    vid0 = t.cexp_vid[j0];
    w0 = w[j0];
    if (kApply) {
      const T hs = D == 2 ? (T)1 : cell_width(t.leaf_level[i / NC], (T)0);
      const T k0 = (T)kref<D>(0) * hs, k1 = (T)kref<D>(1) * hs, k2 = (T)kref<D>(2) * hs, k3 = (T)kref<D>(3) * hs;
#pragma unroll
      for (int f = 0; f < NC; ++f) {
        const int df = __popc(e ^ f);
        c[f] = df == 0 ? k0 : df == 1 ? k1 : df == 2 ? k2 : k3;
      }
    }
  }
  pdl_wait();
  pdl_release();
  T s = act ? mul_add(w0, V[vid0], (T)0) : (T)0;
  for (int32_t j = j0 + 1; j < j1; ++j) s = mul_add(w[j], V[t.cexp_vid[j]], s);
  if (!kApply) {
    if (act) out[i] = s;
    return;
  }
  T y = (T)0;
#pragma unroll
  for (int f = 0; f < NC; ++f) {
    const T vf = __shfl_sync(0xffffffffu, s, f, NC);
    y = mul_add(c[f], vf, y);
  }
  if (act) out[i] = y;
}

// V + omega r / diag in place; FP64 multiplies by scale[v] = omega / diag
// (formed with the right-hand side), the FP64 quotient being several times
// the rest of the update.
__device__ __forceinline__ double updated(double v, double r, double, double, double scale) { return fma(scale, r, v); }
__device__ __forceinline__ float updated(float v, float r, float omega, float diag, float) { return v + omega * r / diag; }

// Per vertex: y = sum of w * product over its incident leaf corners, then the
// sweep's update of V (kRes: block sums of (b - y)^2 to r2 instead).
template <typename T, bool kRes>
__global__ void __launch_bounds__(256) k_vertex_pass(DevTree t, const T *b, const T *part, const T *scale, T *V,
                                                     T omega, double *r2) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = v < t.n_vert;
  const int32_t j0 = act ? t.inc_ptr[v] : 0, j1 = act ? t.inc_ptr[v + 1] : 0;
  const T *w = inc_weights(t, (T)0);
  const T diag = act && sizeof(T) == 4 ? diag_val(t, v, (T)0) : (T)1;
  double rr = 0.0;
  constexpr int kPre = 4;  // incidences known before the pass before ends
  int32_t lc[kPre];
  T wl[kPre];
#pragma unroll
  for (int k = 0; k < kPre; ++k) {
    const bool ok = j0 + k < j1;
    lc[k] = ok ? t.inc_lc[j0 + k] : -1;
    wl[k] = ok ? w[j0 + k] : (T)0;
  }
  pdl_wait();
  pdl_release();
  T y = (T)0, pv[kPre];
#pragma unroll
  for (int k = 0; k < kPre; ++k) pv[k] = lc[k] >= 0 ? part[lc[k]] : (T)0;
#pragma unroll
  for (int k = 0; k < kPre; ++k)
    if (lc[k] >= 0) y = mul_add(wl[k], pv[k], y);
  for (int32_t j = j0 + kPre; j < j1; ++j) y = mul_add(w[j], part[t.inc_lc[j]], y);
  if (act) {
    const T r = b[v] - y;
    if (kRes) rr = (double)r * (double)r;
    else V[v] = updated(V[v], r, omega, diag, sizeof(T) == 8 ? scale[v] : (T)0);
  }
  if (kRes) block_sum_store_at(rr, r2 + blockIdx.x);
}

// E = -grad V at the vertices from V at the leaf corners: minus the mean over
// the leaves that have v as an unconstrained corner of the edge differences.
__device__ __forceinline__ double over_width(double x, int lev) { return x * (double)c_pow3[lev]; }
__device__ __forceinline__ float over_width(float x, int lev) { return x / c_width32[lev]; }

template <typename T, int D>
__global__ void __launch_bounds__(256) k_efield_adaptive(DevTree t, const T *__restrict__ corner, T *__restrict__ E) {
  constexpr int NC = 1 << D;
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= t.n_vert) return;
  T acc[D];
#pragma unroll
  for (int a = 0; a < D; ++a) acc[a] = (T)0;
  for (int32_t j = t.inc_ptr[v]; j < t.inc_ptr[v + 1]; ++j) {
    const int32_t lc = t.inc_lc[j];
    const int32_t p = t.cexp_ptr[lc];
    if (t.cexp_ptr[lc + 1] - p != 1 || t.cexp_w64[p] != 1.0) continue;
    const int32_t L = lc / NC;
    const int e = lc - L * NC, lev = t.leaf_level[L];
    const T *c = corner + (int64_t)L * NC;
#pragma unroll
    for (int a = 0; a < D; ++a) acc[a] = acc[a] + over_width(c[e | (1 << a)] - c[e & ~(1 << a)], lev);
  }
  const T cn = (T)t.dcnt[v];
#pragma unroll
  for (int a = 0; a < D; ++a) E[a * t.n_vert + v] = -(acc[a] / cn);
}

}  // namespace pic
