// Assembled rows of the FP64 solve on adaptive trees (included by kernels.cu).
//
// The two passes of adaptive_solve.cuh spend five FP64 operations per leaf corner
// and one per incidence, some 30 a vertex in 2D, and two launches a sweep.  The
// same operator assembled per vertex has 9 entries in most rows (27 in 3D): one
// launch, 9 fused adds.  Rows are stored in slices of 32, entry k of the slice's
// rows side by side, padded to the slice's longest row; a sweep is V' = V + scale
// (b - A V) with scale = omega / diag per vertex, tabulated beside them.
//
// One sweep of the 2D bump (75,451 vertices): 9.9 -> 4.0 us.
#pragma once

namespace pic {

constexpr int kRowMax = 48;  // entries of a row; a tree with a longer one keeps the two passes

// The row of vertex v: columns and values (unscaled) in the order met; returns
// its length, or kRowMax + 1.
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

// Entries of every slice of 32 rows; *too_long where a row does not fit.
template <int D>
__global__ void __launch_bounds__(128) k_row_count(DevTree t, int32_t *slice, int32_t *too_long) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int32_t col[kRowMax];
  double val[kRowMax];
  const int len = v < t.n_vert ? assemble_row<D>(t, v, col, val) : 0;
  if (len > kRowMax) *too_long = 1;
  const int m = __reduce_max_sync(0xffffffffu, len);
  if ((threadIdx.x & 31) == 0 && v < t.n_vert) slice[v >> 5] = 32 * m;
}

template <int D>
__global__ void __launch_bounds__(128) k_row_fill(DevTree t, const int32_t *ptr, double omega, int32_t *cols,
                                                  double *vals, double *scale) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if ((v & ~(int64_t)31) >= t.n_vert) return;
  int32_t col[kRowMax];
  double val[kRowMax];
  const int len = v < t.n_vert ? assemble_row<D>(t, v, col, val) : 0;
  if (v < t.n_vert) scale[v] = omega / t.diag64[v];
  const int32_t b = ptr[v >> 5], m = (ptr[(v >> 5) + 1] - b) >> 5;
  for (int k = 0; k < m; ++k) {
    const int64_t at = b + 32 * k + (v & 31);
    cols[at] = k < len ? col[k] : v < t.n_vert ? (int32_t)v : 0;
    vals[at] = k < len ? val[k] : 0.0;
  }
}

// b and V as in k_vertex_pass; kRes: block sums of the squared residual.
template <bool kRes>
__global__ void __launch_bounds__(128) k_row_sweep(DevTree t, RowMatrix A, const double *b, const double *Vin,
                                                   double *__restrict__ Vout, double *r2) {
  const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = v < t.n_vert;
  constexpr int kPre = 9;  // entries read while the sweep before runs
  int32_t col[kPre], p = 0, end = 0;
  double val[kPre];
  const double scale = !kRes && act ? A.scale[v] : 0.0;
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
#pragma unroll
    for (int k = 0; k < kPre; ++k)
      if (col[k] >= 0) y = fma(val[k], u[k], y);
    for (int32_t i = p + 32 * kPre; i < end; i += 32) y = fma(A.val[i], Vin[A.col[i]], y);
    const double r = bv - y;
    if (kRes) rr = r * r;
    else Vout[v] = fma(scale, r, vc);
  }
  if (kRes) block_sum_store_at(rr, r2 + blockIdx.x);
}

int64_t row_slices(const DevTree &t) { return (t.n_vert + 31) / 32; }

void launch_row_count(const DevTree &t, int32_t *slice, int32_t *too_long, cudaStream_t s) {
  COUNT(1);
  if (t.d == 3) k_row_count<3><<<grid_for(t.n_vert, 128), 128, 0, s>>>(t, slice, too_long);
  else k_row_count<2><<<grid_for(t.n_vert, 128), 128, 0, s>>>(t, slice, too_long);
}

void launch_row_fill(const DevTree &t, const int32_t *ptr, double omega, int32_t *cols, double *vals, double *scale,
                     cudaStream_t s) {
  COUNT(1);
  if (t.d == 3) k_row_fill<3><<<grid_for(t.n_vert, 128), 128, 0, s>>>(t, ptr, omega, cols, vals, scale);
  else k_row_fill<2><<<grid_for(t.n_vert, 128), 128, 0, s>>>(t, ptr, omega, cols, vals, scale);
}

// Sweeps between V and Vtmp, then the residual's block sums; returns their number.
static int64_t sweep_rows(const DevTree &t, const RowMatrix &A, const double *b, double *V, double *Vtmp, int sweeps,
                          double *r2, cudaStream_t s) {
  const dim3 g(grid_for(t.n_vert, 128)), block(128);
  double *in = V, *out = Vtmp;
  for (int it = 0; it < sweeps; ++it) {
    COUNT(1);
    launch_pdl(k_row_sweep<false>, g, block, s, t, A, b, in, out, r2);
    std::swap(in, out);
  }
  if (in != V) cudaMemcpyAsync(V, in, sizeof(double) * t.n_vert, cudaMemcpyDeviceToDevice, s);
  COUNT(1);
  launch_pdl(k_row_sweep<true>, g, block, s, t, A, b, V, nullptr, r2);
  return g.x;
}

}  // namespace pic
