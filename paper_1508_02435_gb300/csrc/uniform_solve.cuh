// Jacobi sweeps and vertex field on uniform trees (included by kernels.cu).
//
// On a uniform tree every vertex has its 2^d incident leaves on one level and
// no hanging corner, so a sweep is a 3^d-point stencil on the row-major vertex
// array instead of a walk over the leaf tables for each of the 4^d pairs of
// corners of a vertex's leaves.
//
// FP32 results are those of the leaf-by-leaf assembly bit for bit: per leaf
// corner the terms are added in ascending corner order, and the 2^d leaf
// contributions in ascending leaf order.  That order follows from the
// digit-interleaved leaf ids: the ids of two cells one step apart on axis a
// differ by delta_a = spread(j) - spread(j - 1), whatever the other axes, and
// the |delta| of a vertex, sorted, are super-increasing.  So the leaves are
// visited by nested loops over the axes, the largest |delta| outermost, the
// lower cell first on each axis (the upper one first at j = 0, where the lower
// cell is the wrapped last one).  A thread forms the contributions in a fixed
// order and transposes the axes by selects.  |delta_a| is 3^a wherever j is no
// multiple of 3 and at least 25 3^a (3D) elsewhere past a three-cell grid.
// FP64 sums the stencil by neighbour class: fewer operations (the FP64 pipe
// bounds these kernels), hence fewer roundings.
//
// One sweep, leaf walk -> here (GB300): 243^3 FP32 3,770 -> 68 us (172 MB of
// V, b and V' take 25 us; bound by latency and issue), 81^3 FP32 149 -> 5.4 us
// and FP64 277 -> 19.1 us, 27^3 FP32 22 -> 2.1 us and 27^2 FP64 11 -> 1.6 us
// (both the rate of dependent launches).
#pragma once

namespace pic {

__host__ __device__ constexpr int pop3(int x) { return (x & 1) + ((x >> 1) & 1) + ((x >> 2) & 1); }

// Programmatic dependent launch: a sweep's blocks are resident and have done
// their index arithmetic when the sweep before ends.  The release comes after
// the wait, so a block that runs sees every sweep but the last complete.  What
// the kernel before writes must not be read through the non-coherent path (it
// changes while the block is resident): those pointers are not __restrict__.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Constants of one uniform instance.  FP32: c0, c1, c2 = kref(0, 1, 2 axes differ)
// h^(d-2), the diagonal, and 1 / diagonal in two floats.  FP64: the weights of the
// value itself and of its neighbours that give the sweep's new value beside b omega /
// diag, or (res) the residual b - A V beside b -- from the matrix, so that it does
// not hang on omega, which may be zero.
template <typename T>
struct StencilC;
template <>
struct StencilC<float> {
  float c0, c1, c2, omega, diag, rhi, rlo;
};
template <>
struct StencilC<double> {
  double k0, k1, k2;
};

template <int D>
__device__ __forceinline__ void stencil_consts(const InstInfo &I, float omega, bool, StencilC<float> *s) {
  const float hs = D == 2 ? 1.0f : I.h32;
  s->c0 = (float)kref<D>(0) * hs;
  s->c1 = (float)kref<D>(1) * hs;
  s->c2 = (float)kref<D>(2) * hs;
  s->omega = omega;
  s->diag = I.diag32;
  s->rhi = I.rdiag32;
  s->rlo = I.rdiag_lo32;
}
template <int D>
__device__ __forceinline__ void stencil_consts(const InstInfo &I, double, bool res, StencilC<double> *s) {
  s->k0 = res ? -I.diag : I.jac[0];
  s->k1 = res ? 1.0 / 3.0 : I.jac[1];
  s->k2 = res ? (D == 3 ? I.h * (1.0 / 12.0) : 1.0 / 3.0) : I.jac[2];
}

// |spread(j) - spread(j - 1)| on one axis (0 on a one-cell axis).
__device__ __forceinline__ int32_t step_weight(const int32_t *sp, int32_t M, int32_t j) {
  const int32_t w = __ldg(sp + j) - __ldg(sp + (j == 0 ? M - 1 : j - 1));
  return w < 0 ? -w : w;
}

template <typename T>
__device__ __forceinline__ void order_swap(T &a, T &b, bool c) {
  const T x = a, y = b;
  a = c ? y : x;
  b = c ? x : y;
}

// Sum of the leaf contributions u[i] (bit a of i: 0 = lower cell on axis a) in
// ascending leaf order; w[a], flip[a]: step weight and j == 0 per axis.  kLow:
// axes 1.. are at no multiple of 3, so their weights are 3 (and 9) and only
// axis 0 can come out of order: outermost.
template <int D, bool kLow, typename T>
__device__ __forceinline__ T ordered_sum(T *u, const int32_t *w, const bool *flip) {
  constexpr int NC = 1 << D;
  bool any = false;
#pragma unroll
  for (int a = 0; a < (kLow ? 1 : D); ++a) any |= flip[a];
  if (any) {  // only the first plane, row or column of the periodic grid
#pragma unroll
    for (int a = 0; a < (kLow ? 1 : D); ++a)
#pragma unroll
      for (int i = 0; i < NC; ++i)
        if (!(i >> a & 1)) order_swap(u[i], u[i | 1 << a], flip[a]);
  }
  if (D == 2) {
    order_swap(u[1], u[2], w[0] > (kLow ? 3 : w[1]));
  } else if (kLow) {
    const bool c = w[0] > 9;
    const T v[8] = {u[0], u[1], u[2], u[3], u[4], u[5], u[6], u[7]};
    u[1] = c ? v[2] : v[1];
    u[2] = c ? v[4] : v[2];
    u[3] = c ? v[6] : v[3];
    u[4] = c ? v[1] : v[4];
    u[5] = c ? v[3] : v[5];
    u[6] = c ? v[5] : v[6];
  } else {
    const bool c01 = w[0] > w[1];
    const int32_t hi = c01 ? w[0] : w[1], lo = c01 ? w[1] : w[0];
    order_swap(u[1], u[2], c01);
    order_swap(u[5], u[6], c01);
    order_swap(u[2], u[4], hi > w[2]);
    order_swap(u[3], u[5], hi > w[2]);
    order_swap(u[1], u[2], lo > w[2]);
    order_swap(u[5], u[6], lo > w[2]);
  }
  T y = (T)0;
#pragma unroll
  for (int i = 0; i < NC; ++i) y = y + u[i];
  return y;
}

// FP32 (A V) at a vertex from its neighbours' terms: q(dx, dy, dz) is the
// matrix entry times V at that offset, m the centre's.  3D face neighbours
// have entry zero and are left out (face_terms below).
template <int D, bool kLow, typename Q>
__device__ __forceinline__ float stencil_row(Q q, float m, const int32_t *w, const bool *flip) {
  constexpr int NC = 1 << D;
  float u[NC];
#pragma unroll
  for (int f = 0; f < NC; ++f) {  // the leaf that has the vertex as its corner f
    float acc = 0.0f;
    bool first = true;
#pragma unroll
    for (int g = 0; g < NC; ++g) {
      const int df = pop3(f ^ g);
      if (D == 3 && df == 1) continue;
      const int dx = (g & 1) - (f & 1), dy = (g >> 1 & 1) - (f >> 1 & 1), dz = (g >> 2) - (f >> 2);
      const float term = df == 0 ? m : q(dx, dy, dz);
      acc = first ? term : acc + term;
      first = false;
    }
    u[NC - 1 - f] = acc;
  }
  return ordered_sum<D, kLow>(u, w, flip);
}

// The zero terms of the 3D face neighbours: they only pass on what is not finite.
template <typename Q>
__device__ __forceinline__ float face_terms(Q q) {
  float nf = fmaf(0.0f, q(-1, 0, 0), 0.0f);
  nf = fmaf(0.0f, q(1, 0, 0), nf);
  nf = fmaf(0.0f, q(0, -1, 0), nf);
  nf = fmaf(0.0f, q(0, 1, 0), nf);
  nf = fmaf(0.0f, q(0, 0, -1), nf);
  return fmaf(0.0f, q(0, 0, 1), nf);
}

__device__ __forceinline__ uint32_t high_word(double x) { return (uint32_t)__double2hiint(x) & 0x7fffffffu; }

// FP64, one sweep at a vertex with b times omega / diag, or the residual with b as it is: an edge neighbour shares
// two leaves with the vertex, a corner neighbour one (2D: a face neighbour two, of
// half the entry).  Three fused operations beside the neighbour sums.
__device__ __forceinline__ double sweep3(double c, double edges, double corners, const StencilC<double> &s, double b) {
  return fma(s.k2, fma(2.0, edges, corners), fma(s.k0, c, b));
}
__device__ __forceinline__ double sweep2(double c, double faces, double corners, const StencilC<double> &s, double b) {
  return fma(s.k2, corners, fma(s.k1, faces, fma(s.k0, c, b)));
}

// V + omega r / diag.  The FP32 quotient by the instance's constant diagonal
// is formed as fma(x, zh, x zl) with zh + zl = 1 / diag in two floats
// (Brisebarre, Muller and Raina, IEEE Trans. Computers 53(8), 2004): correctly
// rounded for every x at every diagonal a uniform tree can have (2D: 8/3; 3D:
// 8/3 3^-depth, depth 0 to 7; tests/test_quotient.py tries all 2^23 significands),
// as long as nothing underflows or overflows, which the range check sees to.
constexpr float kQuotLo = 0x1p-60f, kQuotHi = 0x1p60f;

template <int N>
__device__ __forceinline__ void jacobi_update(const float *y, const float *b, const float *vc, const StencilC<float> &s,
                                              float *out) {
  float x[N], lo = kQuotHi, hi = kQuotLo;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    x[j] = s.omega * (b[j] - y[j]);
    lo = fminf(lo, fabsf(x[j]));
    hi = fmaxf(hi, fabsf(x[j]));
  }
  if (lo > kQuotLo && hi < kQuotHi) {
#pragma unroll
    for (int j = 0; j < N; ++j) out[j] = vc[j] + fmaf(x[j], s.rhi, x[j] * s.rlo);
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) out[j] = vc[j] + x[j] / s.diag;
  }
}

// FP64 rows give the new value itself.
template <int N>
__device__ __forceinline__ void jacobi_update(const double *y, const double *, const double *, const StencilC<double> &,
                                              double *out) {
#pragma unroll
  for (int j = 0; j < N; ++j) out[j] = y[j];
}

// Squared residuals of N vertices, in order.
template <int N>
__device__ __forceinline__ double residual2(const float *y, const float *b) {
  double rr = 0.0;
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const double r = (double)(b[j] - y[j]);
    rr = rr + r * r;
  }
  return rr;
}
template <int N>
__device__ __forceinline__ double residual2(const double *y, const double *) {  // rows give the residual itself
  double rr = 0.0;
#pragma unroll
  for (int j = 0; j < N; ++j) rr = rr + y[j] * y[j];
  return rr;
}

// ---- one thread per vertex: small grids and batches ---------------------------

// A V at vertex j of an instance (base: its first vertex), and V there.
template <int D>
__device__ __forceinline__ float apply_at(const float *base, int32_t M, const int32_t *j,
                                          const int32_t *sp, const StencilC<float> &s, float, float *vc) {
  int32_t o[3][3], w[3] = {0, 0, 0}, stride = 1;
  bool flip[3];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    o[a][0] = (j[a] == 0 ? M - 1 : j[a] - 1) * stride;
    o[a][1] = j[a] * stride;
    o[a][2] = (j[a] + 1 == M ? 0 : j[a] + 1) * stride;
    stride *= M;
    flip[a] = j[a] == 0;
    w[a] = step_weight(sp + a * M, M, j[a]);
  }
  auto at = [&](int dx, int dy, int dz) {
    return base[o[0][dx + 1] + o[1][dy + 1] + (D == 3 ? o[2][dz + 1] : 0)];
  };
  *vc = at(0, 0, 0);
  float p[27];
#pragma unroll
  for (int k = 0; k < (D == 3 ? 27 : 9); ++k) {
    const int dx = k % 3 - 1, dy = k / 3 % 3 - 1, dz = D == 3 ? k / 9 - 1 : 0;
    if (dx == 0 && dy == 0 && dz == 0) continue;
    const bool face = (dx != 0) + (dy != 0) + (dz != 0) == 1;
    p[k] = (D == 2 && face ? s.c1 : s.c2) * at(dx, dy, dz);
  }
  auto q = [&](int dx, int dy, int dz) { return p[(D == 3 ? (dz + 1) * 9 : 0) + (dy + 1) * 3 + dx + 1]; };
  const float y = stencil_row<D, false>(q, s.c0 * *vc, w, flip);
  return D == 3 ? y + face_terms(q) : y;
}

template <int D>
__device__ __forceinline__ double apply_at(const double *base, int32_t M, const int32_t *j,
                                           const int32_t *, const StencilC<double> &s, double b, double *vc) {
  int32_t o[3][3], stride = 1;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    o[a][0] = (j[a] == 0 ? M - 1 : j[a] - 1) * stride;
    o[a][1] = j[a] * stride;
    o[a][2] = (j[a] + 1 == M ? 0 : j[a] + 1) * stride;
    stride *= M;
  }
  auto at = [&](int dx, int dy, int dz) {
    return base[o[0][dx + 1] + o[1][dy + 1] + (D == 3 ? o[2][dz + 1] : 0)];
  };
  *vc = at(0, 0, 0);
  if (D == 2)
    return sweep2(*vc, (at(-1, 0, 0) + at(1, 0, 0)) + (at(0, -1, 0) + at(0, 1, 0)),
                  (at(-1, -1, 0) + at(1, -1, 0)) + (at(-1, 1, 0) + at(1, 1, 0)), s, b);
  auto diag = [&](int dz) { return (at(-1, -1, dz) + at(1, -1, dz)) + (at(-1, 1, dz) + at(1, 1, dz)); };
  const double f[6] = {at(-1, 0, 0), at(1, 0, 0), at(0, -1, 0), at(0, 1, 0), at(0, 0, -1), at(0, 0, 1)};
  auto cross = [&](int dz) { return (at(-1, 0, dz) + at(1, 0, dz)) + (at(0, -1, dz) + at(0, 1, dz)); };
  double y = sweep3(*vc, diag(0) + (cross(-1) + cross(1)), diag(-1) + diag(1), s, b);
  uint32_t top = 0u;
#pragma unroll
  for (int k = 0; k < 6; ++k) top = max(top, high_word(f[k]));
  if (top >= 0x7ff00000u)  // the zero terms of the face neighbours pass on what is not finite
    for (int k = 0; k < 6; ++k) y = y + 0.0 * f[k];
  return y;
}

// Fixed-order block sum; every thread of a one-dimensional block calls it.
__device__ __forceinline__ void block_sum_store_at(double v, double *out) {
  __shared__ double sh[32];
  const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (lane == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x < 32) {
    v = lane < nw ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) *out = v;
  }
}

// One sweep V_out = V_in + omega (b - A V_in) / diag (kRes: block sums of
// (b - A V_in)^2 to r2 instead).
template <typename T, int D, bool kRes>
__global__ void __launch_bounds__(128) k_jacobi_vertex(DevTree t, const T *b, const T *Vin,
                                                       T *__restrict__ Vout, T omega, double *r2) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = v < t.n_vert;
  double rr = 0.0;
  const InstInfo &I = inst_of_vertex(t, act ? v : 0);
  const int32_t M = I.M;
  StencilC<T> s;
  stencil_consts<D>(I, omega, kRes, &s);
  int32_t j[3] = {0, 0, 0}, r = act ? (int32_t)(v - I.vert_off) : 0;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const int32_t q = r / M;
    j[a] = r - q * M;
    r = q;
  }
  pdl_wait();
  pdl_release();
  if (act) {
    const T bv = b[v];
    T vc;
    const T y = apply_at<D>(Vin + I.vert_off, M, j, t.spread + I.spread_off, s, bv, &vc);
    if (kRes) rr = residual2<1>(&y, &bv);
    else jacobi_update<1>(&y, &bv, &vc, s, Vout + v);
  }
  if (kRes) block_sum_store_at(rr, r2 + blockIdx.x);
}

// ---- three rows per thread: large grids ---------------------------------------
//
// A thread owns column x of the rows y0 .. y0 + 2, y0 a multiple of 3, and in
// 3D marches along z with the three newest planes of its 3 x 5 neighbourhood
// in registers: five loads a vertex, and in two of three rows (and planes) the
// order of the leaves depends on x alone.

template <typename T>
struct Slab3;  // one plane of the neighbourhood

template <>
struct Slab3<float> {
  float q[15], c[3];  // V times the matrix entry, row by row; the own vertices' V as it is
  __device__ __forceinline__ void set(const float *v, const StencilC<float> &s) {
#pragma unroll
    for (int k = 0; k < 15; ++k) q[k] = s.c2 * v[k];
#pragma unroll
    for (int j = 0; j < 3; ++j) c[j] = v[(j + 1) * 3 + 1];
  }
};

template <>
struct Slab3<double> {
  double c[3], cross[3], diag[3];  // sums over the in-plane neighbours on one and on two axes
  uint32_t top;                    // largest |high word| of the plane
  __device__ __forceinline__ void set(const double *v, const StencilC<double> &) {
    double a[5];
    top = 0u;
#pragma unroll
    for (int k = 0; k < 15; ++k) top = max(top, high_word(v[k]));
#pragma unroll
    for (int r = 0; r < 5; ++r) a[r] = v[r * 3] + v[r * 3 + 2];
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      c[j] = v[(j + 1) * 3 + 1];
      diag[j] = a[j] + a[j + 2];
      cross[j] = a[j + 1] + (v[j * 3 + 1] + v[(j + 2) * 3 + 1]);
    }
  }
};

// (A V) of the three rows at the middle plane.  kLow: z is no multiple of 3.
template <bool kLow>
__device__ __forceinline__ void strip_rows(const Slab3<float> &lo, const Slab3<float> &mid, const Slab3<float> &hi,
                                           const StencilC<float> &s, const int32_t *w, const bool *flip, float *y) {
  auto at = [&](int j, int dx, int dy, int dz) {
    return (dz < 0 ? lo : dz > 0 ? hi : mid).q[(j + 1 + dy) * 3 + dx + 1];
  };
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    auto q = [&](int dx, int dy, int dz) { return at(j, dx, dy, dz); };
    const float m = s.c0 * mid.c[j];
    if (j == 0) {
      y[j] = stencil_row<3, false>(q, m, w, flip);
    } else if (kLow) {
      y[j] = stencil_row<3, true>(q, m, w, flip);
    } else {
      const int32_t wj[3] = {w[0], 3, w[2]};
      const bool fj[3] = {flip[0], false, flip[2]};
      y[j] = stencil_row<3, false>(q, m, wj, fj);
    }
  }
  // A face neighbour that is not finite is the centre or an edge neighbour of
  // another row of the strip, except above and below the strip.
  const float seen = ((y[0] + y[1]) + y[2]) + fmaf(0.0f, mid.q[1], 0.0f * mid.q[13]);
  if (!(fabsf(seen) < __int_as_float(0x7f800000))) {
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      auto q = [&](int dx, int dy, int dz) { return at(j, dx, dy, dz); };
      y[j] = y[j] + face_terms(q);
    }
  }
}

__device__ __forceinline__ void strip_rows(const Slab3<double> &lo, const Slab3<double> &mid, const Slab3<double> &hi,
                                           const StencilC<double> &s, const double *b, double *y) {
#pragma unroll
  for (int j = 0; j < 3; ++j)
    y[j] = sweep3(mid.c[j], mid.diag[j] + (lo.cross[j] + hi.cross[j]), lo.diag[j] + hi.diag[j], s, b[j]);
  if (max(mid.top, max(lo.top, hi.top)) >= 0x7ff00000u) {
#pragma unroll
    for (int j = 0; j < 3; ++j) y[j] = y[j] + (0.0 * mid.cross[j] + 0.0 * (lo.c[j] + hi.c[j]));
  }
}

// The strip's part of one plane: rows y0 - 1 .. y0 + 3, columns x - 1 .. x + 1.
template <typename T>
__device__ __forceinline__ void strip_load(const T *p, const int32_t *row, const int32_t *col, T *v) {
#pragma unroll
  for (int r = 0; r < 5; ++r)
#pragma unroll
    for (int i = 0; i < 3; ++i) v[r * 3 + i] = p[row[r] + col[i]];
}

// FP64, straight from global memory: the FP64 pipe is the bound, and warps that
// need no barrier keep it busy.
template <bool kRes>
__global__ void __launch_bounds__(128) k_jacobi_strip3(DevTree t, const double *b, const double *Vin,
                                                       double *__restrict__ Vout, double omega, double *r2, int len) {
  const InstInfo &I = t.inst[0];
  const int32_t M = I.M, plane = M * M;
  StencilC<double> s;
  stencil_consts<3>(I, omega, kRes, &s);
  const int32_t i = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x), k = i / M, x = i - k * M;
  const bool act = 3 * k < M;
  const int32_t y0 = act ? 3 * k : 0;
  const int32_t col[3] = {x == 0 ? M - 1 : x - 1, x, x + 1 == M ? 0 : x + 1};
  const int32_t row[5] = {(y0 == 0 ? M - 1 : y0 - 1) * M, y0 * M, (y0 + 1) * M, (y0 + 2) * M,
                          (y0 + 3 == M ? 0 : y0 + 3) * M};
  double rr = 0.0;
  pdl_wait();
  pdl_release();
  if (act) {
    const int32_t z0 = (int32_t)blockIdx.y * len;
    Slab3<double> p0, p1, p2;
    auto load = [&](int32_t z, Slab3<double> &p) {
      double v[15];
      strip_load(Vin + (int64_t)z * plane, row, col, v);
      p.set(v, s);
    };
    auto put = [&](int32_t z, const Slab3<double> &lo, const Slab3<double> &mid, Slab3<double> &hi) {
      double bv[3], y[3];
      const int64_t at = (int64_t)z * plane + x;
#pragma unroll
      for (int j = 0; j < 3; ++j) bv[j] = b[at + row[j + 1]];
      load(z + 1 == M ? 0 : z + 1, hi);
      strip_rows(lo, mid, hi, s, bv, y);
      if (kRes) {
        rr = rr + residual2<3>(y, bv);
      } else {
#pragma unroll
        for (int j = 0; j < 3; ++j) Vout[at + row[j + 1]] = y[j];
      }
    };
    load(z0 == 0 ? M - 1 : z0 - 1, p0);
    load(z0, p1);
    for (int32_t z = z0; z < z0 + len; z += 3) {  // the three slabs take turns
      put(z, p0, p1, p2);
      put(z + 1, p1, p2, p0);
      put(z + 2, p2, p0, p1);
    }
  }
  if (kRes) block_sum_store_at(rr, r2 + (int64_t)blockIdx.y * gridDim.x + blockIdx.x);
}

// FP32: the planes are staged in shared memory by asynchronous copies, three at a
// time and three ahead, by blocks of 32 columns x 27 rows (nine strips); a thread
// reads its neighbourhood at fixed distances from one address.  One barrier for
// three planes, and a thread's nine b of them loaded ahead of it: with a barrier a
// plane the wait for the slowest warp took what the staging gave (243^3 80 us).
// Strips from global memory 82 us, this 70 (81^3: 5.9, 5.6).  Three blocks an SM
// leave too few registers (75 us, 81^3 8.2); 9 planes a block are the best march at
// 243^3 (27: 77 us, 81: 99), 3 at 81^3, whose 243 blocks are little more than one an
// SM.  Paired FP32 additions (two rows in one instruction) gave nothing: 71 us.
constexpr int kTileX = 32, kTileY = 27, kTileStrips = kTileY / 3;
constexpr int kTileRow = kTileX + 2, kTilePlane = kTileRow * (kTileY + 2);
constexpr int kTileThreads = kTileX * kTileStrips;
constexpr int kTileCopies = (kTilePlane + kTileThreads - 1) / kTileThreads;
template <bool kRes>
__global__ void __launch_bounds__(kTileThreads, 2) k_jacobi_tile3(DevTree t, const float *b, const float *Vin,
                                                                    float *__restrict__ Vout, float omega, double *r2,
                                                                    int len) {
  __shared__ float ring[2][3][kTilePlane];
  const InstInfo &I = t.inst[0];
  const int32_t M = I.M, plane = M * M;
  StencilC<float> s;
  stencil_consts<3>(I, omega, kRes, &s);
  const int tid = threadIdx.x, lane = tid & 31, strip = tid >> 5;
  const int32_t tiles = (M + kTileX - 1) / kTileX;
  const int32_t x0 = (int32_t)(blockIdx.x % tiles) * kTileX, yb = (int32_t)(blockIdx.x / tiles) * kTileY;
  const int32_t x = x0 + lane, y0 = yb + 3 * strip, z0 = (int32_t)blockIdx.y * len;
  const bool act = x < M;  // M is a multiple of 27: every row is a row of the grid
  int32_t src[kTileCopies];  // this thread's share of a plane's copies
#pragma unroll
  for (int k = 0; k < kTileCopies; ++k) {
    const int i = tid + k * kTileThreads, r = i / kTileRow, c = i - r * kTileRow;
    int32_t yy = yb + r - 1, xx = x0 + c - 1;
    yy = yy < 0 ? M - 1 : yy >= M ? 0 : yy;
    xx = xx < 0 ? M - 1 : xx >= M ? xx - M : xx;  // columns past the grid: any value
    src[k] = yy * M + xx;
  }
  const int32_t xc = act ? x : 0;
  int32_t w[3] = {step_weight(t.spread, M, xc), step_weight(t.spread + M, M, y0), 0};
  bool flip[3] = {xc == 0, y0 == 0, false};
  const int32_t at0 = y0 * M + xc;
  int32_t w2 = step_weight(t.spread + 2 * M, M, z0);
  double rr = 0.0;
  pdl_wait();
  pdl_release();
  auto fetch = [&](int32_t z, float *stage) {  // plane z (periodic)
    const float *p = Vin + (int64_t)(z < 0 ? z + M : z >= M ? z - M : z) * plane;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(stage + tid);
#pragma unroll
    for (int k = 0; k < kTileCopies; ++k)
      if (k + 1 < kTileCopies || tid + k * kTileThreads < kTilePlane)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + k * kTileThreads * 4), "l"(p + src[k])
                     : "memory");
  };
  auto commit = [&]() { asm volatile("cp.async.commit_group;" ::: "memory"); };
  Slab3<float> p0, p1, p2;
  auto take = [&](const float *stage, Slab3<float> &p) {
    const float *q = stage + 3 * strip * kTileRow + lane;
    float v[15];
#pragma unroll
    for (int r = 0; r < 5; ++r)
#pragma unroll
      for (int i = 0; i < 3; ++i) v[r * 3 + i] = q[r * kTileRow + i];
    p.set(v, s);
  };
  auto put = [&](int32_t z, bool low, const float *stage, const Slab3<float> &lo, const Slab3<float> &mid,
                 Slab3<float> &hi, const float *bv) {
    float y[3];
    take(stage, hi);
    flip[2] = false;
    w[2] = 9;
    if (!low) {
      flip[2] = z == 0;
      w[2] = w2;
      w2 = step_weight(t.spread + 2 * M, M, z + 3 < M ? z + 3 : 0);  // for the next such plane
      strip_rows<false>(lo, mid, hi, s, w, flip, y);
    } else {
      strip_rows<true>(lo, mid, hi, s, w, flip, y);
    }
    if (kRes) {
      if (act) rr = rr + residual2<3>(y, bv);
    } else {
      float out[3];
      jacobi_update<3>(y, bv, mid.c, s, out);
      if (act) {
#pragma unroll
        for (int j = 0; j < 3; ++j) Vout[(int64_t)z * plane + at0 + j * M] = out[j];
      }
    }
  };
  // planes z0 - 1, z0 by way of the second half of the ring
  fetch(z0 - 1, ring[1][0]);
  fetch(z0, ring[1][1]);
  commit();
#pragma unroll
  for (int k = 0; k < 3; ++k) fetch(z0 + 1 + k, ring[0][k]);
  commit();
  asm volatile("cp.async.wait_group 1;" ::: "memory");
  __syncthreads();
  take(ring[1][0], p0);
  take(ring[1][1], p1);
  int half = 0;
  for (int32_t z = z0; z < z0 + len; z += 3) {  // the three slabs take turns
    float bv[3][3];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int j = 0; j < 3; ++j) bv[k][j] = b[(int64_t)(z + k) * plane + at0 + j * M];
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // planes z + 1 .. z + 3 are there, and the other half has been read
    if (z + 3 < z0 + len) {
#pragma unroll
      for (int k = 0; k < 3; ++k) fetch(z + 4 + k, ring[half ^ 1][k]);
      commit();
    }
    put(z, false, ring[half][0], p0, p1, p2, bv[0]);
    put(z + 1, true, ring[half][1], p1, p2, p0, bv[1]);
    put(z + 2, true, ring[half][2], p2, p0, p1, bv[2]);
    half ^= 1;
  }
  if (kRes) block_sum_store_at(rr, r2 + (int64_t)blockIdx.y * gridDim.x + blockIdx.x);
}

__device__ __forceinline__ void strip_rows2(const float *v, const StencilC<float> &s, const int32_t *w,
                                            const bool *flip, const float *, float *y) {
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    auto q = [&](int dx, int dy, int) {
      return (dx != 0 && dy != 0 ? s.c2 : s.c1) * v[(j + 1 + dy) * 3 + dx + 1];
    };
    const float m = s.c0 * v[(j + 1) * 3 + 1];
    y[j] = j == 0 ? stencil_row<2, false>(q, m, w, flip) : stencil_row<2, true>(q, m, w, flip);
  }
}

__device__ __forceinline__ void strip_rows2(const double *v, const StencilC<double> &s, const int32_t *, const bool *,
                                            const double *b, double *y) {
  double a[5];
#pragma unroll
  for (int r = 0; r < 5; ++r) a[r] = v[r * 3] + v[r * 3 + 2];
#pragma unroll
  for (int j = 0; j < 3; ++j)
    y[j] = sweep2(v[(j + 1) * 3 + 1], a[j + 1] + (v[j * 3 + 1] + v[(j + 2) * 3 + 1]), a[j] + a[j + 2], s, b[j]);
}

template <typename T, bool kRes>
__global__ void __launch_bounds__(128) k_jacobi_strip2(DevTree t, const T *b, const T *Vin,
                                                       T *__restrict__ Vout, T omega, double *r2) {
  const InstInfo &I = t.inst[0];
  const int32_t M = I.M;
  StencilC<T> s;
  stencil_consts<2>(I, omega, kRes, &s);
  const int32_t i = (int32_t)(blockIdx.x * blockDim.x + threadIdx.x), k = i / M, x = i - k * M;
  const bool act = 3 * k < M;
  const int32_t y0 = act ? 3 * k : 0;
  const int32_t col[3] = {x == 0 ? M - 1 : x - 1, x, x + 1 == M ? 0 : x + 1};
  const int32_t row[5] = {(y0 == 0 ? M - 1 : y0 - 1) * M, y0 * M, (y0 + 1) * M, (y0 + 2) * M,
                          (y0 + 3 == M ? 0 : y0 + 3) * M};
  int32_t w[3] = {0, 0, 0};
  const bool flip[3] = {x == 0, y0 == 0, false};
  if (sizeof(T) == 4) {
    w[0] = step_weight(t.spread, M, x);
    w[1] = step_weight(t.spread + M, M, y0);
  }
  double rr = 0.0;
  pdl_wait();
  pdl_release();
  if (act) {
    T v[15], bv[3], y[3];
#pragma unroll
    for (int j = 0; j < 3; ++j) bv[j] = b[row[j + 1] + x];
    strip_load(Vin, row, col, v);
    strip_rows2(v, s, w, flip, bv, y);
    const T vc[3] = {v[4], v[7], v[10]};
    if (kRes) {
      rr = residual2<3>(y, bv);
    } else {
      T out[3];
      jacobi_update<3>(y, bv, vc, s, out);
#pragma unroll
      for (int j = 0; j < 3; ++j) Vout[row[j + 1] + x] = out[j];
    }
  }
  if (kRes) block_sum_store_at(rr, r2 + blockIdx.x);
}

// ---- launches -------------------------------------------------------------------

// Grids of this many vertices fill the chip with three vertices a thread; the
// sizes next to the line are 3^10 = 59,049 and 3^12 = 531,441 (81^3 FP32: 8.2 us a
// sweep with a thread per vertex, 5.6 us in tiles).
constexpr int64_t kStripVertices = 200000;
constexpr unsigned kJacobiThreads = 128;

// Planes per thread of k_jacobi_strip3 (M is a multiple of 27): a long march reads
// fewer planes twice, but leaves the FP64 pipes fewer warps.  3 / 9 / 27 / 81 planes:
// 81^3 21.8 / 20.6 / 46.3 / 127.7 us a sweep with its share of the solve, 243^3 393 /
// 344 / 349 / 413.
constexpr int kMarch = 9;

template <typename... P, typename... A>
inline void launch_pdl(void (*k)(P...), dim3 grid, dim3 block, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k, P(args)...);
}

// One sweep, or with kRes the residual's block sums: at most
// (n_vert + 127) / 128 of them.  FP64 sweeps take b omega / diag, the residual
// takes b.  Returns the number of blocks.
template <typename T, int D, bool kRes>
int64_t launch_jacobi_uniform(const DevTree &t, const T *b, const T *Vin, T *Vout, T omega, double *r2,
                              cudaStream_t s) {
  COUNT(1);
  if (t.n_inst > 1 || t.n_vert < kStripVertices) {
    const dim3 g(grid_for(t.n_vert, kJacobiThreads));
    launch_pdl(k_jacobi_vertex<T, D, kRes>, g, dim3(kJacobiThreads), s, t, b, Vin, Vout, omega, r2);
    return g.x;
  }
  const int64_t M = t.M;
  if constexpr (D == 2) {
    const dim3 g(grid_for(M * (M / 3), kJacobiThreads));
    launch_pdl(k_jacobi_strip2<T, kRes>, g, dim3(kJacobiThreads), s, t, b, Vin, Vout, omega, r2);
    return g.x;
  }
  if constexpr (D == 3 && sizeof(T) == 4) {
    const int len = M >= 243 ? 9 : 3;
    const dim3 g((unsigned)((M + kTileX - 1) / kTileX * (M / kTileY)), (unsigned)(M / len));
    launch_pdl(k_jacobi_tile3<kRes>, g, dim3(kTileThreads), s, t, b, Vin, Vout, omega, r2, len);
    return (int64_t)g.x * g.y;
  } else if constexpr (D == 3) {
    // one warp a block spreads the work evenly over the SMs' FP64 pipes (81^3: 486
    // blocks of 128 threads leave the pipes idle for half the time, 29.7 -> 23.5 us)
    const dim3 g(grid_for(M * (M / 3), 32), (unsigned)(M / kMarch));
    launch_pdl(k_jacobi_strip3<kRes>, g, dim3(32), s, t, b, Vin, Vout, omega, r2, kMarch);
    return (int64_t)g.x * g.y;
  }
}

// ---- vertex field -----------------------------------------------------------------

// E = -grad V, one thread per vertex: per axis the mean over the 2^d incident
// leaves of the edge difference, the lower or the upper edge of the axis.
// FP32 adds them in ascending leaf order as above.
template <int D>
__global__ void __launch_bounds__(256) k_efield_uniform(DevTree t, const float *__restrict__ V, float *__restrict__ E) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= t.n_vert) return;
  const InstInfo &I = inst_of_vertex(t, v);
  const int32_t M = I.M;
  const float *F = V + I.vert_off;
  int32_t r = (int32_t)(v - I.vert_off), stride = 1, w[3] = {0, 0, 0};
  const int32_t at = r;
  float d0[3], d1[3];  // edge difference of the leaves visited first and second on the axis
  const float vc = F[at], h = I.h32;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const int32_t q = r / M, j = r - q * M;
    r = q;
    w[a] = step_weight(t.spread + I.spread_off + a * M, M, j);
    const float lo = (vc - F[at + (j == 0 ? M - 1 : -1) * stride]) / h;
    const float hi = (F[at + (j + 1 == M ? 1 - M : 1) * stride] - vc) / h;
    d0[a] = j == 0 ? hi : lo;
    d1[a] = j == 0 ? lo : hi;
    stride *= M;
  }
  constexpr int NC = 1 << D;
#pragma unroll
  for (int a = 0; a < D; ++a) {
    int rank = 0;  // axes that change faster than a along the visit order
#pragma unroll
    for (int k = 0; k < D; ++k)
      if (k != a) rank += k < a ? w[k] <= w[a] : w[k] < w[a];
    float acc = 0.0f;
#pragma unroll
    for (int i = 0; i < NC; ++i) acc = acc + ((i >> rank) & 1 ? d1[a] : d0[a]);
    E[a * t.n_vert + v] = -(acc / (float)NC);
  }
}

template <int D>
__global__ void __launch_bounds__(256) k_efield_uniform(DevTree t, const double *__restrict__ V,
                                                        double *__restrict__ E) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (v >= t.n_vert) return;
  const InstInfo &I = inst_of_vertex(t, v);
  const int32_t M = I.M;
  const double *F = V + I.vert_off;
  int32_t r = (int32_t)(v - I.vert_off), stride = 1;
  const int32_t at = r;
  const double f = 0.5 / I.h;  // the rounded leaf width, as in the edge differences (not M / 2 at 243)
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const int32_t q = r / M, j = r - q * M;
    r = q;
    const double lo = F[at + (j == 0 ? M - 1 : -1) * stride], hi = F[at + (j + 1 == M ? 1 - M : 1) * stride];
    E[a * t.n_vert + v] = (lo - hi) * f;
    stride *= M;
  }
}

}  // namespace pic
