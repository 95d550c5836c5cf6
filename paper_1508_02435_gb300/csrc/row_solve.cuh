// Assembled rows of the FP64 solve on adaptive trees (included by kernels.cu).
//
// The two passes of adaptive_solve.cuh spend five FP64 operations per leaf corner
// and one per incidence, some 30 a vertex in 2D, and two launches a sweep.  The
// same operator assembled per vertex has 9 entries in most rows (27 in 3D): one
// launch, 9 fused adds.  Rows are stored in slices of 32, entry k of the slice's
// rows side by side, padded to the slice's longest row; a sweep is V' = V + scale
// (b - A V) with scale = omega / diag per vertex, tabulated beside them.
//
// A row of the exact matrix sums to zero; of the rounded entries it does not, and that
// acts on the potential like a term of its own in every sweep.  In 2D the missing part
// (rest, exact to a rounding of itself) is a tenth term of the sum.  3D rows, whose 27
// terms also round more, take differences to the vertex's own value, which cost a
// subtraction an entry on the FP64 pipe (in 2D 4.8 us a sweep of the bump below).
// Against sweeps in extended precision, 100 sweeps of 24,017 vertices in 2D: the
// potential is off by 1.7e-16, the field by 9.0e-16, without the rest 2.7e-15 and
// 2.4e-15, leaf by leaf 3.9e-16 and 8.6e-16; 833 vertices in 3D: 1.1e-16 and 2.4e-16, as
// plain sums 3.0e-16 and 4.0e-16, leaf by leaf 1.1e-16 and 2.2e-16.
//
// One sweep of the 2D bump (75,451 vertices): 9.9 -> 3.8 us.
#pragma once

namespace pic {

constexpr int kRowMax = 48;  // entries of a row; a tree with a longer one keeps the two passes

// The row of vertex v by one thread: columns and values (unscaled) in the order met;
// returns its length, or kRowMax + 1.
template <int D>
__device__ __forceinline__ int assemble_row(const DevTree &t, int64_t v, int32_t *col, double *val) {
  constexpr int NC = 1 << D;
  int len = 0;
  for (int32_t i = t.inc_ptr[v]; i < t.inc_ptr[v + 1]; ++i) {
    const int32_t lc = t.inc_lc[i], L = lc / NC;
    const int e = lc - L * NC;
    const double w = t.inc_w64[i] * (D == 2 ? 1.0 : c_width64[t.leaf_level[L]]);
    for (int f = 0; f < NC; ++f) {
      const double k = w * kref<D>(__popc(e ^ f));
      const int32_t c = L * NC + f;
      for (int32_t j = t.cexp_ptr[c]; j < t.cexp_ptr[c + 1]; ++j) {
        const int32_t u = t.cexp_vid[j];
        int at = 0;
        while (at < len && col[at] != u) ++at;
        if (at == len) {
          if (len == kRowMax) return kRowMax + 1;
          col[len] = u;
          val[len++] = 0.0;
        }
        val[at] = fma(k, t.cexp_w64[j], val[at]);
      }
    }
  }
  return len;
}

// The same by one warp: entry k in slot k / 32 of lane k % 32.  The terms of an
// incidence, its leaf's expansions, lie side by side: 32 are loaded at once, then
// added one by one, the warp comparing all columns with one ballot a slot.  In 3D a
// vertex has 64 terms, thousands between levels, and a thread takes some twenty steps
// for each: assembly of the 3D bump's 47,965 rows 4.4 ms by threads, 0.5 by warps; of
// the 2D bump's 75,451 (16 terms in most) 0.19 and 0.30.
template <int D, bool kValues>
__device__ __forceinline__ int assemble_row_warp(const DevTree &t, int64_t v, int32_t *col, double *val) {
  constexpr int NC = 1 << D;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  int len = 0;
  col[0] = col[1] = -1;
  val[0] = val[1] = 0.0;
  for (int32_t i = t.inc_ptr[v]; i < t.inc_ptr[v + 1]; ++i) {
    const int32_t lc = t.inc_lc[i], L = lc / NC;
    const int e = lc - L * NC;
    const double w = kValues ? t.inc_w64[i] * (D == 2 ? 1.0 : c_width64[t.leaf_level[L]]) : 0.0;
    const int32_t mine = t.cexp_ptr[L * NC + (lane <= NC ? lane : NC)];  // the corners' first terms, and the end
    const int32_t b = __shfl_sync(full, mine, 0), end = __shfl_sync(full, mine, NC);
    for (int32_t j0 = b; j0 < end; j0 += 32) {
      const int32_t j = j0 + lane;
      int f = 0;
#pragma unroll
      for (int g = 1; g < NC; ++g) f += j >= __shfl_sync(full, mine, g);
      const int32_t u = j < end ? t.cexp_vid[j] : -1;
      const double k = kValues ? w * kref<D>(__popc(e ^ f)) : 0.0, c = kValues && j < end ? t.cexp_w64[j] : 0.0;
      const int m = end - j0 < 32 ? end - j0 : 32;
      for (int q = 0; q < m; ++q) {
        const int32_t uq = __shfl_sync(full, u, q);
        const unsigned lo = __ballot_sync(full, col[0] == uq), hi = __ballot_sync(full, col[1] == uq);
        int at = lo ? __ffs(lo) - 1 : hi ? 31 + __ffs(hi) : len;
        if (at == len) {
          if (len == kRowMax) return kRowMax + 1;
          ++len;
          if (at == lane) col[0] = uq;
          if (at == lane + 32) col[1] = uq;
        }
        if (kValues) {
          const double kq = __shfl_sync(full, k, q), cq = __shfl_sync(full, c, q);
          if (at == lane) val[0] = fma(kq, cq, val[0]);
          if (at == lane + 32) val[1] = fma(kq, cq, val[1]);
        }
      }
    }
  }
  return len;
}

// A block takes a slice of 32 rows: a warp a row in 3D, a thread a row (one warp)
// in 2D.
template <int D>
__host__ __device__ constexpr int row_threads() { return D == 3 ? 256 : 32; }

// Entries of every slice; *too_long where a row does not fit.
template <int D>
__global__ void __launch_bounds__(row_threads<D>()) k_row_count(DevTree t, int32_t *slice, int32_t *too_long) {
  __shared__ int most;
  if (threadIdx.x == 0) most = 0;
  __syncthreads();
  for (int r = D == 3 ? threadIdx.x >> 5 : threadIdx.x; r < 32; r += row_threads<D>() / (D == 3 ? 32 : 1)) {
    const int64_t v = (int64_t)blockIdx.x * 32 + r;
    if (v >= t.n_vert) break;
    int32_t col[D == 3 ? 2 : kRowMax];
    double val[D == 3 ? 2 : kRowMax];
    const int len = D == 3 ? assemble_row_warp<D, false>(t, v, col, val) : assemble_row<D>(t, v, col, val);
    if (len > kRowMax) *too_long = 1;
    if (D == 2 || (threadIdx.x & 31) == 0) atomicMax(&most, len);
  }
  __syncthreads();
  if (threadIdx.x == 0) slice[blockIdx.x] = 32 * most;
}

// Adds x to hi + lo (Knuth's two-sum).
__device__ __forceinline__ void two_sum(double &hi, double &lo, double x) {
  const double s = hi + x, z = s - hi;
  lo += (hi - (s - z)) + (x - z);
  hi = s;
}

template <int D>
__global__ void __launch_bounds__(row_threads<D>()) k_row_fill(DevTree t, const int32_t *ptr, double omega, int32_t *cols,
                                                               double *vals, double *scale, double *rest) {
  const int32_t b = ptr[blockIdx.x], m = (ptr[blockIdx.x + 1] - b) >> 5;
  auto put = [&](int64_t v, int k, int len, int32_t col, double val) {  // entry k of the row, padded to m
    const int64_t at = b + 32 * k + (v & 31);
    cols[at] = k < len ? col : v < t.n_vert ? (int32_t)v : 0;
    vals[at] = k < len ? val : 0.0;
  };
  if constexpr (D == 3) {
    const int lane = threadIdx.x & 31;
    for (int r = threadIdx.x >> 5; r < 32; r += row_threads<D>() / 32) {
      const int64_t v = (int64_t)blockIdx.x * 32 + r;
      int32_t col[2];
      double val[2];
      const int len = v < t.n_vert ? assemble_row_warp<D, true>(t, v, col, val) : 0;
      if (v < t.n_vert && lane == 0) scale[v] = omega / t.diag64[v];
      if (lane < m) put(v, lane, len, col[0], val[0]);
      if (lane + 32 < m) put(v, lane + 32, len, col[1], val[1]);
    }
  } else {
    const int64_t v = (int64_t)blockIdx.x * 32 + threadIdx.x;
    int32_t col[kRowMax];
    double val[kRowMax];
    const int len = v < t.n_vert ? assemble_row<D>(t, v, col, val) : 0;
    double hi = 0.0, lo = 0.0;
    for (int k = 0; k < len; ++k) two_sum(hi, lo, val[k]);
    if (v < t.n_vert) {
      scale[v] = omega / t.diag64[v];
      rest[v] = -(hi + lo);
    }
    for (int k = 0; k < m; ++k) put(v, k, len, col[k], val[k]);
  }
}

// b and V as in k_vertex_pass; kRes: block sums of the squared residual.
template <int D, bool kRes>
__global__ void __launch_bounds__(128) k_row_sweep(DevTree t, RowMatrix A, const double *b, const double *Vin,
                                                   double *__restrict__ Vout, double *r2) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = v < t.n_vert;
  constexpr int kPre = 9;  // entries read while the sweep before runs
  int32_t col[kPre], p = 0, end = 0;
  double val[kPre];
  const double scale = !kRes && act ? A.scale[v] : 0.0, rest = D == 2 && act ? A.rest[v] : 0.0;
  if (act) {
    p = A.ptr[v >> 5];
    end = A.ptr[(v >> 5) + 1];
    p += (int32_t)(v & 31);
  }
#pragma unroll
  for (int k = 0; k < kPre; ++k) {
    const bool ok = p + 32 * k < end;
    col[k] = ok ? A.col[p + 32 * k] : -1;
    val[k] = ok ? A.val[p + 32 * k] : 0.0;
  }
  pdl_wait();
  pdl_release();
  double rr = 0.0;
  if (act) {
    double u[kPre], y = 0.0;
#pragma unroll
    for (int k = 0; k < kPre; ++k) u[k] = col[k] >= 0 ? Vin[col[k]] : 0.0;
    const double bv = b[v], vc = Vin[v];
    if (D == 2) y = rest * vc;
#pragma unroll
    for (int k = 0; k < kPre; ++k)
      if (col[k] >= 0) y = fma(val[k], D == 3 ? u[k] - vc : u[k], y);
    for (int32_t i = p + 32 * kPre; i < end; i += 32) y = fma(A.val[i], D == 3 ? Vin[A.col[i]] - vc : Vin[A.col[i]], y);
    const double r = bv - y;
    if (kRes) rr = r * r;
    else Vout[v] = fma(scale, r, vc);
  }
  if (kRes) block_sum_store_at(rr, r2 + blockIdx.x);
}

int64_t row_slices(const DevTree &t) { return (t.n_vert + 31) / 32; }

// Entries to hold: any rows in 3D and on small trees; in 2D most rows have 9 to 12
// entries, and 32 a vertex hold the padded slices of trees with several levels.
int64_t row_capacity(const DevTree &t) {
  return row_slices(t) * 32 * (t.d == 3 || t.n_vert < 65536 ? kRowMax : 32);
}

void launch_row_count(const DevTree &t, int32_t *slice, int32_t *too_long, cudaStream_t s) {
  COUNT(1);
  const unsigned g = (unsigned)row_slices(t);
  if (t.d == 3) k_row_count<3><<<g, row_threads<3>(), 0, s>>>(t, slice, too_long);
  else k_row_count<2><<<g, row_threads<2>(), 0, s>>>(t, slice, too_long);
}

void launch_row_fill(const DevTree &t, const int32_t *ptr, double omega, int32_t *cols, double *vals, double *scale,
                     double *rest, cudaStream_t s) {
  COUNT(1);
  const unsigned g = (unsigned)row_slices(t);
  if (t.d == 3) k_row_fill<3><<<g, row_threads<3>(), 0, s>>>(t, ptr, omega, cols, vals, scale, rest);
  else k_row_fill<2><<<g, row_threads<2>(), 0, s>>>(t, ptr, omega, cols, vals, scale, rest);
}

// Sweeps between V and Vtmp, then the residual's block sums; returns their number.
template <int D>
static int64_t sweep_rows(const DevTree &t, const RowMatrix &A, const double *b, double *V, double *Vtmp, int sweeps,
                          double *r2, cudaStream_t s) {
  const dim3 g(grid_for(t.n_vert, 128)), block(128);
  double *in = V, *out = Vtmp;
  for (int it = 0; it < sweeps; ++it) {
    COUNT(1);
    launch_pdl(k_row_sweep<D, false>, g, block, s, t, A, b, in, out, r2);
    std::swap(in, out);
  }
  if (in != V) cudaMemcpyAsync(V, in, sizeof(double) * t.n_vert, cudaMemcpyDeviceToDevice, s);
  COUNT(1);
  launch_pdl(k_row_sweep<D, true>, g, block, s, t, A, b, V, nullptr, r2);
  return g.x;
}

}  // namespace pic
