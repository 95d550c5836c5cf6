// Deposit: per-leaf corner sums over the particles, then charges per vertex
// (included by kernels.cu).
#pragma once

namespace pic {

// ---- per leaf -----------------------------------------------------------------
//
// 2^D lanes share a leaf.  They load its next 2^D particles in bucket order
// (PIDT: the leaf's 2^D sub-buckets in corner order), one each, form each
// particle's shape factors once, and exchange them through shared memory: lane e
// adds corner e's over the particles in order, so the sums are those of one
// thread walking the bucket.  The next particles are in flight meanwhile.  (One
// thread per leaf waits for each particle in turn.  One thread a leaf -> here:
// 2e8 two-stream particles, 14 a leaf in 8 sub-buckets, 2.5 -> 1.7 ms; 256 2D
// plasmas with up to 1,370 particles a leaf 304 -> 230 us; 81^3 cells of 8 FP64
// 540 -> 340 us; the FP64 2D bump 177 -> 37 us.)

// What a particle's lane hands over, and the contribution lane e takes from it.
template <typename T, int D>
struct ShapeRow;

template <>
struct ShapeRow<float, 3> {
  static constexpr int kLen = 8, kPad = 8;
  __device__ __forceinline__ static void put(float *row, const float *t, bool ok) {
    const float g0[2] = {1.0f - t[0], t[0]}, g1[2] = {1.0f - t[1], t[1]}, g2[2] = {1.0f - t[2], t[2]};
    float w[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) w[e] = ok ? g0[e & 1] * g1[e >> 1 & 1] * g2[e >> 2] : 0.0f;
    *(float4 *)row = make_float4(w[0], w[1], w[2], w[3]);
    *(float4 *)(row + 4) = make_float4(w[4], w[5], w[6], w[7]);
  }
  __device__ __forceinline__ static float add(const float *row, int e, float acc) { return acc + row[e]; }
};

template <>
struct ShapeRow<float, 2> {
  static constexpr int kLen = 4, kPad = 4;
  __device__ __forceinline__ static void put(float *row, const float *t, bool ok) {
    const float a = 1.0f - t[0], b = 1.0f - t[1];
    *(float4 *)row = ok ? make_float4(a * b, t[0] * b, a * t[1], t[0] * t[1]) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __device__ __forceinline__ static float add(const float *row, int e, float acc) { return acc + row[e]; }
};

// FP64: the last factor is multiplied in by a fused add (fewer operations of the
// FP64 pipe).
template <>
struct ShapeRow<double, 3> {
  static constexpr int kLen = 6, kPad = 4;
  __device__ __forceinline__ static void put(double *row, const double *t, bool ok) {
    const double a = 1.0 - t[0], b = 1.0 - t[1];
    *(double2 *)row = make_double2(a * b, t[0] * b);
    *(double2 *)(row + 2) = make_double2(a * t[1], t[0] * t[1]);
    *(double2 *)(row + 4) = ok ? make_double2(1.0 - t[2], t[2]) : make_double2(0.0, 0.0);
  }
  __device__ __forceinline__ static double add(const double *row, int e, double acc) {
    return fma(row[e & 3], row[4 + (e >> 2)], acc);
  }
};

template <>
struct ShapeRow<double, 2> {
  static constexpr int kLen = 4, kPad = 2;
  __device__ __forceinline__ static void put(double *row, const double *t, bool ok) {
    *(double2 *)row = make_double2(1.0 - t[0], t[0]);
    *(double2 *)(row + 2) = ok ? make_double2(1.0 - t[1], t[1]) : make_double2(0.0, 0.0);
  }
  __device__ __forceinline__ static double add(const double *row, int e, double acc) {
    return fma(row[e & 1], row[2 + (e >> 1)], acc);
  }
};

// Values of shared memory per warp: 32 rows, the rows of each leaf shifted by kPad.
template <typename T, int D>
__host__ __device__ constexpr int shape_slice() {
  return 32 * ShapeRow<T, D>::kLen + (32 >> D) * ShapeRow<T, D>::kPad;
}

__device__ __forceinline__ void local_coord(float x, float, int32_t, float *t) { *t = x; }
__device__ __forceinline__ void local_coord(double x, double s, int32_t c, double *t) {
  *t = unit_clamp(x * s - (double)c);  // rounded as everywhere else
}

template <typename T, int D>
__global__ void k_leaf_partials(DevTree t, const int32_t *__restrict__ start, const T *__restrict__ pos, int64_t n,
                                T *__restrict__ part) {
  constexpr int NC = 1 << D;
  using Row = ShapeRow<T, D>;
  extern __shared__ double2 shape_smem[];
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, e = lane & (NC - 1), grp = lane / NC;
  T *slice = (T *)shape_smem + (threadIdx.x >> 5) * shape_slice<T, D>();
  T *mine = slice + lane * Row::kLen + grp * Row::kPad;
  const T *rows = slice + grp * (NC * Row::kLen + Row::kPad);
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, L = i / NC;
  const bool act = L < t.n_leaves;
  int32_t c[D], b = 0, total = 0, pre = 0, incl = 0;
  T s = (T)0;
#pragma unroll
  for (int k = 0; k < D; ++k) c[k] = 0;
  if (act) {
    if (sizeof(T) == 8 || (t.scheme != 0 && t.uniform)) {
#pragma unroll
      for (int k = 0; k < D; ++k) c[k] = t.leaf_coords[L * D + k];
    }
    if (sizeof(T) == 8) s = (T)c_pow3_64[t.leaf_level[L]];
    int32_t key = (int32_t)L;
    if (t.scheme != 0) {
      if (t.uniform) {
        uint32_t C[D];
#pragma unroll
        for (int k = 0; k < D; ++k) C[k] = (uint32_t)c[k];
        key = push_key<D, true>(t, inst_of_leaf(t, (int32_t)L), (int32_t)L, C, e);
      } else {
        key = t.corner_pv[i] * NC + (NC - 1 - e);
      }
    }
    b = start[key];
    total = start[key + 1] - b;
  }
  const bool sub = t.scheme != 0;  // lane e holds sub-bucket e: prefix over the leaf's lanes
  if (sub) {
    incl = total;
#pragma unroll
    for (int o = 1; o < NC; o <<= 1) {
      const int32_t y = __shfl_up_sync(full, incl, o, NC);
      if (e >= o) incl += y;
    }
    pre = incl - total;
    total = __shfl_sync(full, incl, NC - 1, NC);
  }
  const int32_t most = __reduce_max_sync(full, total);
  auto fetch = [&](int32_t q, T *x) {  // position of the leaf's particle q
    int32_t at = b + q;
    if (sub) {
      int a = 0;
#pragma unroll
      for (int k = 0; k < NC - 1; ++k) a += q >= __shfl_sync(full, incl, k, NC);
      at = __shfl_sync(full, b, a, NC) + q - __shfl_sync(full, pre, a, NC);
    }
#pragma unroll
    for (int k = 0; k < D; ++k) x[k] = q < total ? pos[k * n + at] : (T)0;
  };
  // kAhead rounds of 2^D particles are loaded together, and the next ones while
  // these are summed: in 2D crowded leaves would wait for memory in every round
  // of four (batch 291 -> 230 us; 3D rounds of eight lose by it, 1.7 -> 1.9 ms)
  constexpr int kAhead = D == 2 ? 4 : 1;
  T acc = (T)0, x[kAhead][D];
#pragma unroll
  for (int h = 0; h < kAhead; ++h)
    if (h * NC < most) fetch(e + h * NC, x[h]);
  for (int32_t q0 = 0; q0 < most; q0 += kAhead * NC) {
    T u[kAhead][D];
#pragma unroll
    for (int h = 0; h < kAhead; ++h)
#pragma unroll
      for (int k = 0; k < D; ++k) local_coord(x[h][k], s, c[k], &u[h][k]);
#pragma unroll
    for (int h = 0; h < kAhead; ++h)
      if (q0 + (kAhead + h) * NC < most) fetch(q0 + e + (kAhead + h) * NC, x[h]);
#pragma unroll
    for (int h = 0; h < kAhead; ++h) {
      if (q0 + h * NC >= most) break;
      Row::put(mine, u[h], q0 + e + h * NC < total);
      __syncwarp();
#pragma unroll
      for (int j = 0; j < NC; ++j) acc = Row::add(rows + j * Row::kLen, e, acc);
      __syncwarp();
    }
  }
  if (act) part[i] = acc;
}

// One thread per leaf, for many leaves of few particles in one run (FP32 PIT):
// the lanes above would stand idle in a leaf's last round (5e6 particles on 81^3
// cells, 9 a leaf: 24 us, 37 us with eight lanes a leaf).
template <int D>
__global__ void k_leaf_walk(int64_t n_leaves, const int32_t *__restrict__ start, const float *__restrict__ o, int64_t n,
                            float *__restrict__ part) {
  constexpr int NC = 1 << D;
  const int64_t L = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (L >= n_leaves) return;
  float acc[NC];
#pragma unroll
  for (int e = 0; e < NC; ++e) acc[e] = 0.0f;
  for (int32_t p = start[L]; p < start[L + 1]; ++p) {
    float tl[D];
#pragma unroll
    for (int b = 0; b < D; ++b) tl[b] = o[b * n + p];
#pragma unroll
    for (int e = 0; e < NC; ++e) acc[e] = acc[e] + shape<float>(tl, e, D);
  }
  if (D == 3) store32(part + L * NC, acc);
  else *(float4 *)(part + L * NC) = make_float4(acc[0], acc[1], acc[2], acc[3]);
}

// ---- per vertex ------------------------------------------------------------------

__device__ __forceinline__ double inst_q(const InstInfo &I, double) { return I.q; }
__device__ __forceinline__ float inst_q(const InstInfo &I, float) { return I.q32; }
__device__ __forceinline__ double inst_ion(const InstInfo &I, double) { return I.ion; }
__device__ __forceinline__ float inst_ion(const InstInfo &I, float) { return I.ion32; }

// Sum of the incident leaf corners of a uniform tree's vertex in ascending leaf
// order (the order of uniform_solve.cuh: no sort of the leaf ids).
template <typename T, int D>
__device__ __forceinline__ T incident_sum(int64_t v, const InstInfo &I, const int32_t *spread, const T *part) {
  constexpr int NC = 1 << D;
  const int32_t M = I.M, *sp = spread + I.spread_off;
  int32_t r = (int32_t)(v - I.vert_off), hi[D], lo[D], w[3] = {0, 0, 0};
  bool flip[3] = {false, false, false};
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const int32_t q = r / M, j = r - q * M;
    r = q;
    flip[a] = j == 0;
    hi[a] = __ldg(sp + a * M + j);
    lo[a] = __ldg(sp + a * M + (flip[a] ? M - 1 : j - 1));
    w[a] = hi[a] > lo[a] ? hi[a] - lo[a] : lo[a] - hi[a];
  }
  T u[NC];
#pragma unroll
  for (int f = 0; f < NC; ++f) {
    int32_t leaf = I.leaf_off;
#pragma unroll
    for (int a = 0; a < D; ++a) leaf += (f >> a) & 1 ? lo[a] : hi[a];
    u[NC - 1 - f] = part[(int64_t)leaf * NC + f];
  }
  return ordered_sum<D, false>(u, w, flip);
}

// S = sum of w * partial over incident leaf corners (ascending), Q = q S + ion *
// integral(phi_v); block partial sums of Q in FP64, `per` vertices per thread.
// The FP64 sum over the block is what costs here: five FP64 adds per thread and
// shuffle step, on a pipe of some two lanes a clock.
template <typename T>
__global__ void k_vertex_charge(DevTree t, const T *__restrict__ part, T *__restrict__ Q, double *block_sum, int per) {
  double mine = 0.0;
  for (int u = 0; u < per; ++u) {
    const int64_t v = ((int64_t)blockIdx.x * per + u) * blockDim.x + threadIdx.x;
    if (v >= t.n_vert) break;
    const InstInfo &I = inst_of_vertex(t, v);
    const T q = inst_q(I, (T)0), ion = inst_ion(I, (T)0);
    T S = (T)0;
    if (t.uniform) {
      S = t.d == 3 ? incident_sum<T, 3>(v, I, t.spread, part) : incident_sum<T, 2>(v, I, t.spread, part);
    } else {
      const T *w = inc_weights(t, (T)0);
      for (int32_t j = t.inc_ptr[v]; j < t.inc_ptr[v + 1]; ++j) S = S + w[j] * part[t.inc_lc[j]];
    }
    const T val = q * S + ion * ion_load(t, v, (T)0);
    Q[v] = val;
    mine = mine + (double)val;
  }
  if (block_sum) block_sum_store(mine, block_sum);
}

// The same on the grid of one uniform 3D instance, FP64: blocks of 32 x 8 columns
// march `len` planes, so that a leaf's row of eight partials, which eight
// vertices read, comes from the L2 about once.
__global__ void __launch_bounds__(256) k_vertex_charge_grid(DevTree t, const double *__restrict__ part,
                                                            double *__restrict__ Q, double *block_sum, int len) {
  const InstInfo &I = t.inst[0];
  const int32_t M = I.M, tiles = (M + 31) / 32;
  const int32_t x = (int32_t)(blockIdx.x % tiles) * 32 + (threadIdx.x & 31);
  const int32_t y = (int32_t)(blockIdx.x / tiles) * 8 + (threadIdx.x >> 5), z0 = (int32_t)blockIdx.y * len;
  double mine = 0.0;
  if (x < M && y < M) {
    const int32_t *sp = t.spread;
    const double q = inst_q(I, 0.0), ion = inst_ion(I, 0.0) * ion_load(t, 0, 0.0);
    int32_t w[3], s2[4];
    bool flip[3] = {x == 0, y == 0, false};
    const int32_t x1 = __ldg(sp + x), x0 = __ldg(sp + (flip[0] ? M - 1 : x - 1));
    const int32_t y1 = __ldg(sp + M + y), y0 = __ldg(sp + M + (flip[1] ? M - 1 : y - 1));
    w[0] = abs(x1 - x0);
    w[1] = abs(y1 - y0);
    s2[0] = x1 + y1;
    s2[1] = x0 + y1;
    s2[2] = x1 + y0;
    s2[3] = x0 + y0;
    sp += 2 * M;
    int32_t lo = __ldg(sp + (z0 == 0 ? M - 1 : z0 - 1));
#pragma unroll 3
    for (int32_t z = z0; z < z0 + len; ++z) {
      const int32_t hi = __ldg(sp + z);
      w[2] = abs(hi - lo);
      flip[2] = z == 0;
      double u[8];
#pragma unroll
      for (int f = 0; f < 8; ++f) u[7 - f] = part[(int64_t)(s2[f & 3] + (f >> 2 ? lo : hi)) * 8 + f];
      lo = hi;
      const double val = q * ordered_sum<3, false>(u, w, flip) + ion;
      Q[((int64_t)z * M + y) * M + x] = val;
      mine = mine + (double)val;
    }
  }
  block_sum_store_at(mine, block_sum + (int64_t)blockIdx.y * gridDim.x + blockIdx.x);
}

// FP32: a leaf's row of eight partials goes to eight vertices, so a thread loads it
// whole and hands the values out through shared memory; the upper four wait in
// registers for the next plane.  Loads of single partials, each over the sectors
// of 32 rows, are bound by the L1: 243^3 cells 160 us that way, 117 here (516 MB:
// 76 us).  FP64 rows take twice the registers and shared memory, and lose by it
// (243^3 1.63 -> 1.81 ms with the leaf sums).
constexpr int kChargeX = 32, kChargeY = 8, kChargeRow = kChargeX + 1, kChargeCells = kChargeRow * (kChargeY + 1);
__global__ void __launch_bounds__(256) k_vertex_charge_tile(DevTree t, const float *__restrict__ part,
                                                            float *__restrict__ Q, double *block_sum, int len) {
  __shared__ float plane[2][8][kChargeCells + 7];
  const InstInfo &I = t.inst[0];
  const int32_t M = I.M, tiles = (M + kChargeX - 1) / kChargeX, *sp = t.spread;
  const int32_t bx = (int32_t)(blockIdx.x % tiles) * kChargeX, by = (int32_t)(blockIdx.x / tiles) * kChargeY;
  const int32_t x = bx + (threadIdx.x & 31), y = by + (threadIdx.x >> 5), z0 = (int32_t)blockIdx.y * len;
  const bool act = x < M && y < M;
  // this thread's leaves of a plane, and the cells x - 1, y - 1 of its vertex
  int32_t leaf[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int i = (int)threadIdx.x + h * 256, r = i / kChargeRow;
    const int32_t cx = bx + (i - r * kChargeRow) - 1, cy = by + r - 1;
    leaf[h] = -1;
    if (i < kChargeCells && cx < M && cy < M)
      leaf[h] = __ldg(sp + (cx < 0 ? M - 1 : cx)) + __ldg(sp + M + (cy < 0 ? M - 1 : cy));
  }
  const int at = (int)(threadIdx.x >> 5) * kChargeRow + (int)(threadIdx.x & 31);
  const float q = inst_q(I, 0.0f), ion = inst_ion(I, 0.0f) * ion_load(t, 0, 0.0f);
  int32_t w[3] = {act ? step_weight(sp, M, x) : 0, act ? step_weight(sp + M, M, y) : 0, 0};
  bool flip[3] = {x == 0, y == 0, false};
  sp += 2 * M;
  float row[2][8], below[4];
  auto fetch = [&](int32_t z) {
    const int32_t sz = __ldg(sp + (z < 0 ? M - 1 : z));
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (leaf[h] >= 0) load32(part + (int64_t)(leaf[h] + sz) * 8, row[h]);
  };
  double mine = 0.0;
  fetch(z0 - 1);
  for (int32_t z = z0 - 1; z < z0 + len; ++z) {
    float(*s)[kChargeCells + 7] = plane[(z - z0) & 1];
#pragma unroll
    for (int h = 0; h < 2; ++h)
      if (leaf[h] >= 0) {
#pragma unroll
        for (int e = 0; e < 8; ++e) s[e][threadIdx.x + h * 256] = row[h][e];
      }
    __syncthreads();
    if (z + 1 < z0 + len) fetch(z + 1);
    if (act) {
      float u[8];
#pragma unroll
      for (int f = 0; f < 4; ++f) {
        const int c = at + (f & 1 ? 0 : 1) + (f >> 1 ? 0 : kChargeRow);
        u[7 - f] = s[f][c];
        u[3 - f] = below[f];
        below[f] = s[4 + f][c];
      }
      if (z >= z0) {
        w[2] = step_weight(sp, M, z);
        flip[2] = z == 0;
        const float val = q * ordered_sum<3, false>(u, w, flip) + ion;
        Q[((int64_t)z * M + y) * M + x] = val;
        mine = mine + (double)val;
      }
    }
  }
  block_sum_store_at(mine, block_sum + (int64_t)blockIdx.y * gridDim.x + blockIdx.x);
}

// Per-instance FP64 sums of the vertex charges, one block per instance (fixed order).
template <typename T>
__global__ void k_inst_sum(DevTree t, const T *Q, double *out) {
  const InstInfo &I = t.inst[blockIdx.x];
  double v = 0.0;
  for (int64_t i = threadIdx.x; i < I.n_vert; i += blockDim.x) v += (double)Q[I.vert_off + i];
  __shared__ double sh[32];
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  if (w == 0) {
    v = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0.0;
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    if (lane == 0) out[blockIdx.x] = v;
  }
}

// ---- launches ----------------------------------------------------------------------

template <typename T>
static void vertex_charge(const DevTree &t, const T *part, T *Q, double *block_sum, double *total, cudaStream_t s) {
  if (t.uniform && t.n_inst == 1 && t.d == 3 && t.M >= 81) {
    // FP32 at 243^3, 9 / 27 planes a block: 128 / 117 us; smaller grids need the blocks
    const int len = sizeof(T) == 4 && t.M >= 243 ? 27 : 9;
    const dim3 g((unsigned)((t.M + kChargeX - 1) / kChargeX * ((t.M + kChargeY - 1) / kChargeY)),
                 (unsigned)(t.M / len));
    COUNT(2);
    if constexpr (sizeof(T) == 4) k_vertex_charge_tile<<<g, 256, 0, s>>>(t, part, Q, block_sum, len);
    else k_vertex_charge_grid<<<g, 256, 0, s>>>(t, part, Q, block_sum, len);
    k_sum_blocks<<<1, 1024, 0, s>>>(block_sum, (int64_t)g.x * g.y, total);
    return;
  }
  const unsigned b = bsz(t.block_vert);
  // large grids: eight vertices a thread share the block sum; small ones need the threads
  const int per = t.n_vert >= 1000000 ? 8 : 1;
  const unsigned g = grid_for((t.n_vert + per - 1) / per, b);
  COUNT(1);
  k_vertex_charge<T><<<g, b, 0, s>>>(t, part, Q, t.n_inst > 1 ? nullptr : block_sum, per);
  COUNT(t.n_inst > 1 ? 2 : 1);
  if (t.n_inst > 1) {
    k_inst_sum<T><<<t.n_inst, 1024, 0, s>>>(t, Q, total + 1);
    k_sum_blocks<<<1, 1024, 0, s>>>(total + 1, t.n_inst, total);
  } else {
    k_sum_blocks<<<1, 1024, 0, s>>>(block_sum, g, total);
  }
}

void launch_vertex_charge(const DevTree &t, bool split, const void *part, void *Q, double *block_sum,
                          double *total, cudaStream_t s) {
  if (split) vertex_charge<float>(t, (const float *)part, (float *)Q, block_sum, total, s);
  else vertex_charge<double>(t, (const double *)part, (double *)Q, block_sum, total, s);
}

template <typename T, int D>
static void leaf_partials(const DevTree &t, const int32_t *start, const T *pos, int64_t n, T *part, cudaStream_t s) {
  const unsigned b = bsz(t.block_leaf);
  COUNT(1);
  k_leaf_partials<T, D><<<grid_for(t.n_leaves << D, b), b, sizeof(T) * shape_slice<T, D>() * (b / 32), s>>>(t, start, pos,
                                                                                                          n, part);
}

void launch_deposit(const DevTree &t, bool split, const int32_t *start, const void *pos, int64_t n, void *part,
                    void *Q, double *block_sum, double *total, cudaStream_t s) {
  if (split && t.scheme == 0 && t.n_inst == 1 && t.n_leaves >= 300000 && n < 16 * t.n_leaves) {
    const unsigned b = bsz(t.block_leaf), g = grid_for(t.n_leaves, b);
    COUNT(1);
    if (t.d == 3) k_leaf_walk<3><<<g, b, 0, s>>>(t.n_leaves, start, (const float *)pos, n, (float *)part);
    else k_leaf_walk<2><<<g, b, 0, s>>>(t.n_leaves, start, (const float *)pos, n, (float *)part);
  } else if (split) {
    if (t.d == 3) leaf_partials<float, 3>(t, start, (const float *)pos, n, (float *)part, s);
    else leaf_partials<float, 2>(t, start, (const float *)pos, n, (float *)part, s);
  } else {
    if (t.d == 3) leaf_partials<double, 3>(t, start, (const double *)pos, n, (double *)part, s);
    else leaf_partials<double, 2>(t, start, (const double *)pos, n, (double *)part, s);
  }
  launch_vertex_charge(t, split, part, Q, block_sum, total, s);
}

}  // namespace pic
