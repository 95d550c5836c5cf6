// The whole solve of a small uniform tree in one launch (included by kernels.cu).
//
// A sweep over a few thousand vertices takes less than the two microseconds that
// dependent launches are apart.  Here one cluster of up to
// nine CTAs keeps the grid in shared memory: each holds a slab of rows (2D) or
// planes (3D) and a halo on both sides, writes its outer rows into its
// neighbours' halos as it updates them, and meets the others at a cluster
// barrier after every sweep.  The sums are those of uniform_solve.cuh.
//
// 100 sweeps of 27^2 cells, FP64: 188 us as launches, 88 us here; 81^2 FP32 188 ->
// 75 us.
#pragma once

namespace pic {

template <typename T, int D, int M>
struct Resident {
  static constexpr int kCtas = M < 9 ? M : 9;                // cluster size
  static constexpr int kSlab = M / kCtas;                    // rows or planes of a CTA
  static constexpr int kPlane = D == 3 ? M * M : M;          // vertices of one
  static constexpr int kItems = D == 3 ? kSlab : 1;          // vertices of a thread: a column (3D) or one
  static constexpr int kWork = D == 3 ? kPlane : kPlane * kSlab;
  static constexpr int kThreads = (kWork + 31) / 32 * 32;
  static constexpr int kBuf = (kSlab + 2) * kPlane;          // values of a slab with its halos
  static constexpr bool kScaled = D == 3 && sizeof(T) == 4;  // shared memory holds c2 V
};

__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_meet() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Shared address of `p` in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t peer_addr(const void *p, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void peer_store(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
__device__ __forceinline__ void peer_store(uint32_t a, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// A V of item `i` of a thread; s: the slab buffer, col: in-plane offsets of the
// nine columns (3D) or three (2D) around it, row: its slab row (2D).
template <int M>
__device__ __forceinline__ float resident_row3(const float *s, const int *col, int i, float v, const StencilC<float> &c,
                                               const int32_t *w, const bool *flip, bool bad, float) {
  constexpr int PL = M * M;
  float p[27];
#pragma unroll
  for (int k = 0; k < 27; ++k) {
    const int dx = k % 3 - 1, dy = k / 3 % 3 - 1, dz = k / 9 - 1;
    if ((dx != 0) + (dy != 0) + (dz != 0) >= 2) p[k] = s[(i + 1 + dz) * PL + col[k % 9]];
  }
  auto q = [&](int dx, int dy, int dz) { return p[(dz + 1) * 9 + (dy + 1) * 3 + dx + 1]; };
  float y = stencil_row<3, false>(q, c.c0 * v, w, flip);
  if (bad) {
    auto f = [&](int dx, int dy, int dz) { return s[(i + 1 + dz) * PL + col[(dy + 1) * 3 + dx + 1]]; };
    y = y + face_terms(f);
  }
  return y;
}

template <int M>
__device__ __forceinline__ double resident_row3(const double *s, const int *col, int i, double v,
                                                const StencilC<double> &c, const int32_t *, const bool *, bool bad, double b) {
  constexpr int PL = M * M;
  auto at = [&](int k, int dz) { return s[(i + 1 + dz) * PL + col[k]]; };
  auto diag = [&](int dz) { return (at(0, dz) + at(2, dz)) + (at(6, dz) + at(8, dz)); };
  auto cross = [&](int dz) { return (at(3, dz) + at(5, dz)) + (at(1, dz) + at(7, dz)); };
  double y = sweep3(v, diag(0) + (cross(-1) + cross(1)), diag(-1) + diag(1), c, b);
  if (bad) y = y + (0.0 * at(1, 0) + 0.0 * at(7, 0)) + (0.0 * at(3, 0) + 0.0 * at(5, 0)) + (0.0 * at(4, -1) + 0.0 * at(4, 1));
  return y;
}

template <int M>
__device__ __forceinline__ float resident_row2(const float *s, const int *col, int row, float v, const StencilC<float> &c,
                                               const int32_t *w, const bool *flip, float) {
  float p[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    const int dx = k % 3 - 1, dy = k / 3 - 1;
    if (k != 4) p[k] = (dx != 0 && dy != 0 ? c.c2 : c.c1) * s[(row + 1 + dy) * M + col[dx + 1]];
  }
  auto q = [&](int dx, int dy, int) { return p[(dy + 1) * 3 + dx + 1]; };
  return stencil_row<2, false>(q, c.c0 * v, w, flip);
}

template <int M>
__device__ __forceinline__ double resident_row2(const double *s, const int *col, int row, double v,
                                                const StencilC<double> &c, const int32_t *, const bool *, double b) {
  auto at = [&](int k, int dy) { return s[(row + 1 + dy) * M + col[k]]; };
  return sweep2(v, (at(0, 0) + at(2, 0)) + (at(1, -1) + at(1, 1)), (at(0, -1) + at(2, -1)) + (at(0, 1) + at(2, 1)), c,
                b);
}

__device__ __forceinline__ bool not_finite(float x) { return !(fabsf(x) < __int_as_float(0x7f800000)); }
__device__ __forceinline__ bool not_finite(double x) { return high_word(x) >= 0x7ff00000u; }

template <typename T, int D, int M>
__global__ void __launch_bounds__(Resident<T, D, M>::kThreads) k_solve_resident(DevTree t, const T *__restrict__ Q,
                                                                              const double *__restrict__ total, T *V,
                                                                              int sweeps, T omega, double *r2) {
  using R = Resident<T, D, M>;
  constexpr int PL = R::kPlane, N = R::kItems;
  __shared__ T buf[2][R::kBuf];
  __shared__ int bad;  // some V is not finite: the zero terms of the 3D face neighbours count
  const InstInfo &I = t.inst[0];
  StencilC<T> c;
  stencil_consts<D>(I, omega, false, &c);
  const int rank = (int)cluster_rank(), z0 = rank * R::kSlab, tid = threadIdx.x;
  const bool act = tid < R::kWork;
  const int row = D == 3 ? 0 : tid / M;
  const int x = tid % M, y = D == 3 ? tid / M % M : 0, own = D == 3 ? tid : x;
  const int xs[3] = {x == 0 ? M - 1 : x - 1, x, x + 1 == M ? 0 : x + 1};
  int col[9];
  if (D == 3) {
    const int ys[3] = {y == 0 ? M - 1 : y - 1, y, y + 1 == M ? 0 : y + 1};
#pragma unroll
    for (int k = 0; k < 9; ++k) col[k] = ys[k / 3] * M + xs[k % 3];
  } else {
#pragma unroll
    for (int k = 0; k < 9; ++k) col[k] = xs[k % 3];
  }
  int32_t w[3] = {0, 0, 0}, wl[N];
  bool flip[3] = {x == 0, y == 0, false};
  if (sizeof(T) == 4) {
    w[0] = step_weight(t.spread, M, x);
    if (D == 3) w[1] = step_weight(t.spread + M, M, y);
#pragma unroll
    for (int i = 0; i < N; ++i) wl[i] = step_weight(t.spread + (D - 1) * M, M, z0 + (D == 3 ? i : row < R::kSlab ? row : 0));
  }
  const uint32_t lo_peer = (uint32_t)((rank + R::kCtas - 1) % R::kCtas), hi_peer = (uint32_t)((rank + 1) % R::kCtas);
  const uint32_t lo_buf = peer_addr(&buf[0][0], lo_peer), hi_buf = peer_addr(&buf[0][0], hi_peer);
  const T tot = (T)*total;
  T v[N], b[N], raw[N];
  auto stored = [&](T u) {  // what shared memory holds of a value
    if constexpr (R::kScaled) return c.c2 * u;
    else return u;
  };
  if (tid == 0) bad = 0;
  __syncthreads();
  bool odd = false;
  for (int k = tid; k < R::kBuf; k += blockDim.x) {  // the slab and its halos
    const int z = (z0 + k / PL - 1 + M) % M;
    const T u = V[z * PL + k % PL];
    odd |= not_finite(u);
    buf[0][k] = stored(u);
  }
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const int at = act ? (z0 + (D == 3 ? i : row)) * PL + own : 0;
    v[i] = V[at];
    b[i] = raw[i] = Q[at] - tot * ion_load(t, 0, (T)0);
    if constexpr (sizeof(T) == 8) b[i] = fma(b[i], I.rhs, b[i] * I.rhs_lo);
  }
  auto apply = [&](const T *s, int i, bool any) {
    if (sizeof(T) == 4) w[D - 1] = wl[i];
    flip[D - 1] = z0 + (D == 3 ? i : row) == 0;
    if constexpr (D == 3) return resident_row3<M>(s, col, i, v[i], c, w, flip, any, b[i]);
    else return resident_row2<M>(s, col, row, v[i], c, w, flip, b[i]);
  };
  auto report = [&](bool found) {  // to every CTA, seen after the next meeting
    if (D == 3 && found)
      for (int k = 0; k < R::kCtas; ++k) peer_store(peer_addr(&bad, (uint32_t)k), 1);
  };
  cluster_meet();  // every CTA runs and has cleared its flag
  report(odd);
  cluster_meet();
  for (int it = 0; it < sweeps; ++it) {
    const T *cur = buf[it & 1];
    const int nb = (it + 1) & 1;
    if (act) {
      const bool any = D == 3 && bad != 0;
      T out[N];
#pragma unroll
      for (int i = 0; i < N; ++i) {
        const T yv = apply(cur, i, any);
        jacobi_update<1>(&yv, &b[i], &v[i], c, &out[i]);
      }
      odd = false;
#pragma unroll
      for (int i = 0; i < N; ++i) {
        v[i] = out[i];
        odd |= not_finite(out[i]);
        const T u = stored(out[i]);
        const int r = D == 3 ? i : row;
        buf[nb][(r + 1) * PL + own] = u;
        // the outer rows also to the neighbours' halos
        if (r == 0) peer_store(lo_buf + (uint32_t)((nb * R::kBuf + (R::kSlab + 1) * PL + own) * sizeof(T)), u);
        if (r == R::kSlab - 1) peer_store(hi_buf + (uint32_t)((nb * R::kBuf + own) * sizeof(T)), u);
      }
      report(odd);
    }
    cluster_meet();
  }
  double rr = 0.0;
  stencil_consts<D>(I, omega, true, &c);
  if (act) {
    const bool any = D == 3 && bad != 0;
#pragma unroll
    for (int i = 0; i < N; ++i) {
      b[i] = raw[i];
      const T yv = apply(buf[sweeps & 1], i, any);
      rr = rr + residual2<1>(&yv, &b[i]);
      V[(z0 + (D == 3 ? i : row)) * PL + own] = v[i];
    }
  }
  __shared__ double mine, parts[R::kCtas];
  block_sum_store_at(rr, &mine);  // thread 0 holds it
  if (tid == 0) peer_store(peer_addr(&parts[rank], 0u), mine);
  cluster_meet();
  if (rank == 0 && tid == 0) {
    double sum = 0.0;
    for (int k = 0; k < R::kCtas; ++k) sum = sum + parts[k];
    *r2 = sum;
  }
}

// Launch, or with `ask` only say whether the cluster fits the device.
template <typename T, int D, int M>
static bool resident_launch(bool ask, const DevTree &t, const T *Q, const double *total, T *V, int sweeps, T omega,
                            double *r2, cudaStream_t s) {
  using R = Resident<T, D, M>;
  auto k = k_solve_resident<T, D, M>;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(R::kCtas);
  cfg.blockDim = dim3(R::kThreads);
  cfg.stream = s;
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = R::kCtas;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  if (ask) {
    int n = 0;
    bool ok = cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess &&
              cudaOccupancyMaxActiveClusters(&n, k, &cfg) == cudaSuccess && n > 0;
    if (!ok) cudaGetLastError();
    return ok;
  }
  COUNT(1);
  cudaLaunchKernelEx(&cfg, k, t, Q, total, V, sweeps, omega, r2);
  return true;
}

// The grids it serves: up to 9^3, and 27^2 (FP64, whose pipe is slow on nine SMs) or
// 81^2 (FP32).  27^3 FP32 is as fast in launches over the whole chip: 2.1 us a sweep
// both ways.
template <typename T>
static bool resident_solve(bool ask, const DevTree &t, const T *Q, const double *total, T *V, int sweeps, T omega,
                           double *r2, cudaStream_t s) {
#define PIC_RESIDENT(D_, M_) \
  if (t.d == D_ && t.M == M_) return resident_launch<T, D_, M_>(ask, t, Q, total, V, sweeps, omega, r2, s)
  PIC_RESIDENT(3, 3);
  PIC_RESIDENT(3, 9);
  PIC_RESIDENT(2, 3);
  PIC_RESIDENT(2, 9);
  PIC_RESIDENT(2, 27);
  if constexpr (sizeof(T) == 4) {
    PIC_RESIDENT(2, 81);
  }
#undef PIC_RESIDENT
  return false;
}

}  // namespace pic
