// Fused gather, push, re-location, key and mover rank of the generic step
// (included by kernels.cu).
//
// Templated on the dimension (the per-axis loops unroll and the per-particle
// arrays stay in registers), on uniform against adaptive trees, and on batches
// (kBatch, uniform trees).  A batch's particle belongs to the instance of its
// leaf: a state that is handed over may change the numbers of particles per
// instance.  Single plasmas do not wait for that lookup (243 x 243 cells of 100
// particles, five steps: 1.20 ms with it, 1.18 without) and have their grid in the
// kernel's parameters (1e7 free 2D particles: from the instance table 0.111 ms, from
// the parameters 0.109).  3D steps
// write the pushed state as one record per particle, which the re-bin gathers
// whole; 2D steps write rows.
//
// Measured against one kernel for all trees with divisions by 3^k, a descent
// from the root and separate FP64 products and sums: FP64 push of 4.25e6
// particles on 81^3 cells 0.98 -> 0.51 ms, FP64 push of the 1e6-particle 2D bump
// 0.19 -> 0.07 ms (adaptive FP64 trees now expand the field at the leaf corners
// once per field, as FP32 did), 1e7 free 2D particles in a reflecting box 0.17 ->
// 0.11 ms, 2e8 two-stream particles 7.3 -> 5.03 ms (whole-sector corner rows and
// records, four blocks per SM).
#pragma once

namespace pic {

// Artificial work of the paper's experiments (Section 6): `flops` floating
// point operations per particle move (fused multiply-adds, two each), on a
// value the move does not use; the never-taken test keeps them.
template <typename T>
__device__ __forceinline__ void artificial_flops(T seed, int32_t flops, int32_t *err) {
  T acc = seed;
  for (int32_t i = 0; i < flops; i += 2) acc = fma(acc, (T)0.999, (T)1e-3);
  if (acc == (T)-12345.0) atomicOr(err, 0);
}

// Reflection at the walls of the unit box, FP64 (the oracle's reading): the
// free path y folds into [0, 2); y >= 1 mirrors to 2 - y with the velocity
// component negated; the far wall itself goes to the largest double below 1.
__device__ __forceinline__ double fold64(double y, bool *flip) {
  double m = y - 2.0 * floor(y * 0.5);
  *flip = false;
  if (m >= 1.0) {
    m = 2.0 - m;
    *flip = true;
    if (m >= 1.0) m = 0x1.fffffffffffffp-1;
  }
  return m;
}

// The field at the corners of leaf L of an adaptive tree: [corner][axis], whole
// 32-byte units.  PIDT particles of a warp lie in some eighteen leaves, and the
// L1 looks up every leaf's line again for each load.
template <typename T, int D>
__device__ __forceinline__ void corner_row(const T *Ec, int32_t L, T *q) {
  constexpr int N = D << D, W = 32 / (int)sizeof(T);
#pragma unroll
  for (int i = 0; i < N; i += W) load32(Ec + (int64_t)L * N + i, q + i);
}

// The grid of leaf L's instance.  A single plasma's is in the kernel's parameters.
struct PushGrid {
  int32_t M, depth, leaf_off, vert_off, spread_off;
};
template <bool kBatch>
__device__ __forceinline__ PushGrid push_grid(const DevTree &t, int32_t L) {
  if (!kBatch) return PushGrid{t.M, t.depth, 0, 0, 0};
  const InstInfo &I = t.inst[t.inst_of_leaf[L]];
  return PushGrid{I.M, I.depth, I.leaf_off, I.vert_off, I.spread_off};
}

// Level and coordinates of leaf L.
template <int D, bool kUni>
__device__ __forceinline__ int push_leaf(const DevTree &t, const PushGrid &I, int32_t L, int32_t *c) {
  if (kUni) {
#pragma unroll
    for (int k = 0; k < D; ++k) c[k] = t.leaf_coords[(int64_t)L * D + k];
    return I.depth;
  }
  const int4 r = t.leaf_rec[L];
  c[0] = r.x;
  c[1] = r.y;
  if (D == 3) c[D - 1] = r.z;
  return r.w;
}

// Sort key of a particle in leaf L through corner a.  Uniform trees: C is the
// leaf's cell; adaptive ones read the owner-vertex table.
template <int D, bool kUni, typename Grid>
__device__ __forceinline__ int32_t push_key(const DevTree &t, const Grid &I, int32_t L, const uint32_t *C, int a) {
  constexpr int NC = 1 << D;
  if (t.scheme == 0) return L;
  int32_t pv;
  if (kUni) {
    pv = I.vert_off;
    int32_t mul = 1;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      int32_t j = (int32_t)C[k] + ((a >> k) & 1);
      if (j == I.M) j = 0;
      pv += j * mul;
      mul *= I.M;
    }
  } else {
    pv = t.corner_pv[(int64_t)L * NC + a];
  }
  return pv * NC + (NC - 1 - a);
}

// Target cell index of one axis, FP32: cell c of `per`, `fl` cells on,
// periodic.
__device__ __forceinline__ int32_t wrapped_cell(int32_t c, float fl, int32_t per) {
  if (fabsf(fl) < 1.0e9f) {
    int32_t cc = c + (int32_t)fl;
    if ((uint32_t)cc >= (uint32_t)per) {
      cc %= per;
      if (cc < 0) cc += per;
    }
    return cc;
  }
  const int64_t c64 = ((int64_t)c + (int64_t)fminf(fmaxf(fl, -1.0e15f), 1.0e15f)) % per;
  return (int32_t)(c64 < 0 ? c64 + per : c64);
}

// Reflecting walls (the oracle's reading): cell index folded modulo 2 per; the
// mirrored half maps to (2 per - 1 - Im, 1 - f), or to (2 per - Im, 0) when
// f = 0, with the velocity component negated.
__device__ __forceinline__ int32_t reflected_cell(int32_t c, float fl, int32_t per, float *f, float *vn) {
  if (fabsf(fl) < 1.0e9f) {  // inside the box: nothing to fold
    const int32_t cc = c + (int32_t)fl;
    if ((uint32_t)cc < (uint32_t)per) return cc;
  }
  const int64_t p2 = 2 * (int64_t)per;
  int64_t im = ((int64_t)c + (int64_t)fminf(fmaxf(fl, -1.0e15f), 1.0e15f)) % p2;
  if (im < 0) im += p2;
  if (im < per) return (int32_t)im;
  *vn = -*vn;
  if (*f > 0.0f) {
    *f = clamp_off(1.0f - *f);
    return (int32_t)(p2 - 1 - im);
  }
  const int32_t cc = (int32_t)(p2 - im);
  if (cc < per) return cc;
  *f = 0x1.fffffep-1f;
  return per - 1;
}

// Four blocks of 512 per SM (32 registers): the push waits for memory, and more
// warps wait together.  It costs 16 to 36 bytes of spills a thread (56 in 3D
// batches).  Three blocks -> four: 1e7 free 2D particles 0.122 -> 0.109 ms, 2e8
// two-stream particles 5.35 -> 5.07; uniform PIDT, 8e6 particles on 729^2 cells 0.139
// -> 0.133, 8e6 on 81^3 0.171 -> 0.164, 3e7 on 243^3 0.796 -> 0.793.
template <int D, bool kUni, bool kBatch>
__global__ void __launch_bounds__(512, 4) k_push32(DevTree t, Push32Args a) {
  constexpr int NC = 1 << D;
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, n = a.n;
  int32_t knew = 0;
  bool moved = false;
  if (p < n) {
    const int32_t L = a.leaf[p];
    float o[D], v[D];
#pragma unroll
    for (int k = 0; k < D; ++k) o[k] = a.o[k * n + p];
#pragma unroll
    for (int k = 0; k < D; ++k) v[k] = a.v[k * n + p];
    const int32_t kold = t.scheme == 0 ? L : a.key[p];
    const PushGrid Ins = push_grid<kBatch>(t, L);
    int32_t c[D];
    const int lev = push_leaf<D, kUni>(t, Ins, L, c);
    const bool field = a.E || a.Ec;
    if (field) {
      float E[D];
#pragma unroll
      for (int k = 0; k < D; ++k) E[k] = 0.0f;
      if (kUni) {
        int32_t vid[8];
        corner_vertices(Ins, c, D, vid);
#pragma unroll
        for (int e = 0; e < NC; ++e) {
          const float w = shape<float>(o, e, D);
#pragma unroll
          for (int k = 0; k < D; ++k) E[k] = E[k] + w * a.E[k * t.n_vert + vid[e]];
        }
      } else {  // the corner values, expanded once per field
        float q[NC * D];
        corner_row<float, D>(a.Ec, L, q);
#pragma unroll
        for (int e = 0; e < NC; ++e) {
          const float w = shape<float>(o, e, D);
#pragma unroll
          for (int k = 0; k < D; ++k) E[k] = E[k] + w * q[e * D + k];
        }
      }
#pragma unroll
      for (int k = 0; k < D; ++k) v[k] = v[k] + a.qmdt * E[k];
    }
    const int32_t per = kUni ? Ins.M : (int32_t)c_pow3[lev];
    const float sl = a.sl[lev];
    uint32_t I[D];
    float f[D];
    bool bad = false, inside = true;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      float tt = o[k] + v[k] * sl;
      if (!isfinite(v[k]) || !isfinite(tt)) { bad = true; tt = 0.0f; }
      const float fl = floorf(tt);
      f[k] = tt - fl;
      const int32_t cc = a.reflect ? reflected_cell(c[k], fl, per, &f[k], &v[k]) : wrapped_cell(c[k], fl, per);
      I[k] = (uint32_t)cc;
      inside &= cc == c[k];
    }
    if (a.flops > 0) artificial_flops<float>(o[0], a.flops, a.err);
    if (bad) atomicOr(a.err, 1);
    float o2[D];
    int32_t L2;
    if (kUni) {  // the covering leaf is the target cell itself; o = f
      int32_t cc[3] = {(int32_t)I[0], (int32_t)I[1], D == 3 ? (int32_t)I[D - 1] : 0};
      L2 = Ins.leaf_off + uniform_leaf_of_cell(t.spread + Ins.spread_off, Ins.M, cc, D);
    } else if (inside) {
      // still inside its leaf (the radius of operation of Section 5.3): no
      // lift, no drop -- the covering leaf is the old one and o = f
      L2 = L;
    }
    if (kUni || inside) {
#pragma unroll
      for (int k = 0; k < D; ++k) o2[k] = clamp_off(f[k]);
    } else {
      L2 = locate_split<D>(t, lev, I, f, o2, 0);
    }
    knew = push_key<D, kUni>(t, Ins, L2, I, pidt_corner_o(o2, D));
    moved = knew != kold;
    if (D == 3) {
      const float r[8] = {o2[0], o2[1], o2[D - 1], v[0], v[1], v[D - 1], __int_as_float(L2), __int_as_float(knew)};
      store32((float *)(a.rec + 2 * p), r);
    } else {
#pragma unroll
      for (int k = 0; k < D; ++k) a.tv[k * n + p] = v[k];
#pragma unroll
      for (int k = 0; k < D; ++k) a.to[k * n + p] = o2[k];
      a.tleaf[p] = L2;
    }
    if (D == 3 || t.scheme != 0) a.keyn[p] = knew;  // PIT rows: the key array is the leaf array
  }
  rank_movers<D == 3>(p, moved, knew, a.count, a.words, a.rank);
}

// ---- FP64: the FP64 pipe bounds the push (some two operations a clock and SM),
// so comparisons look at the high word and products feed fused adds.

__device__ __forceinline__ uint32_t hi_bits(double x) { return (uint32_t)__double2hiint(x); }

// Local coordinate in [0, 1].
__device__ __forceinline__ double unit_clamp(double u) {
  const uint32_t h = hi_bits(u);
  return (h >> 31) ? 0.0 : h >= 0x3ff00000u ? 1.0 : u;
}

// quantise() of a wrapped position (in [0, 1)): truncation is the floor, the
// upper bound holds for the integer.
__device__ __forceinline__ uint32_t quantise_unit(double y) {
  const uint32_t q = __double2uint_rz(y * 774840978.0);
  return q > 774840977u ? 774840977u : q;
}

template <int D, bool kUni, bool kBatch>
__global__ void k_push64(DevTree t, Push64Args a) {
  constexpr int NC = 1 << D;
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, n = a.n;
  int32_t knew = 0;
  bool moved = false;
  if (p < n) {
    const int32_t L = a.leaf[p];
    double x[D], v[D];
#pragma unroll
    for (int k = 0; k < D; ++k) x[k] = a.x[k * n + p];
#pragma unroll
    for (int k = 0; k < D; ++k) v[k] = a.v[k * n + p];
    const int32_t kold = t.scheme == 0 ? L : a.key[p];
    const PushGrid Ins = push_grid<kBatch>(t, L);
    int32_t c[D];
    const int lev = push_leaf<D, kUni>(t, Ins, L, c);
    double t0 = 0.0;
    if (a.E) {
      const double s = c_pow3_64[lev];
      double tl[D], E[D];
#pragma unroll
      for (int k = 0; k < D; ++k) {
        tl[k] = unit_clamp(x[k] * s - (double)c[k]);
        E[k] = 0.0;
      }
      t0 = tl[0];
      int32_t vid[8];
      double q[NC * D];
      if (kUni) corner_vertices(Ins, c, D, vid);
      else corner_row<double, D>(a.Ec, L, q);
#pragma unroll
      for (int e = 0; e < NC; ++e) {
        const double w = shape<double>(tl, e, D);
#pragma unroll
        for (int k = 0; k < D; ++k)
          E[k] = fma(w, kUni ? a.E[k * t.n_vert + vid[e]] : q[e * D + k], E[k]);
      }
#pragma unroll
      for (int k = 0; k < D; ++k) v[k] = fma(a.qmdt, E[k], v[k]);
    }
    uint32_t Q[D];
    bool bad = false;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      const double y = x[k] + v[k] * a.dt;
      if (hi_bits(y) < 0x3ff00000u) {  // in [0, 1): no wall
        x[k] = y;
      } else if (a.reflect) {
        bool flip;
        x[k] = fold64(y, &flip);
        if (flip) v[k] = -v[k];
      } else {
        x[k] = wrap01(y);
      }
      if ((hi_bits(v[k]) & 0x7ff00000u) == 0x7ff00000u || (hi_bits(x[k]) & 0x7ff00000u) == 0x7ff00000u) {
        bad = true;
        x[k] = 0.0;
      }
      Q[k] = quantise_unit(x[k]);
    }
    if (a.flops > 0) artificial_flops<double>(t0, a.flops, a.err);
    if (bad) atomicOr(a.err, 1);
    int lev2 = lev;
    int32_t L2 = L;
    uint32_t C[D];
    bool inside = true;
#pragma unroll
    for (int k = 0; k < D; ++k) {
      C[k] = div_pow3(Q[k] >> 1, 18 - lev);
      inside &= C[k] == (uint32_t)c[k];
    }
    if (kUni) {
      const int32_t cc[3] = {(int32_t)C[0], (int32_t)C[1], D == 3 ? (int32_t)C[D - 1] : 0};
      L2 = Ins.leaf_off + uniform_leaf_of_cell(t.spread + Ins.spread_off, Ins.M, cc, D);
    } else if (!inside) {  // still inside its leaf: the covering leaf is the old one, no descent
      L2 = locate_q<D>(t, Q, 0, &lev2, C);
    }
    int corner = 0;
    if (t.scheme != 0) {  // upper half of the leaf on each axis
      const uint32_t s = c_pow3[18 - lev2];
#pragma unroll
      for (int k = 0; k < D; ++k)
        if (Q[k] - C[k] * (2u * s) >= s) corner |= 1 << k;
    }
    knew = push_key<D, kUni>(t, Ins, L2, C, corner);
    moved = knew != kold;
    if (D == 3) {  // one 64-byte record per particle: the re-bin gathers it whole
      const double r[8] = {x[0], x[1], x[D - 1], v[0], v[1], v[D - 1],
                           __longlong_as_double((long long)(((uint64_t)(uint32_t)knew << 32) | (uint32_t)L2)), 0.0};
      store32((double *)(a.rec + 4 * p), r);
      store32((double *)(a.rec + 4 * p + 2), r + 4);
    } else {
#pragma unroll
      for (int k = 0; k < D; ++k) a.tv[k * n + p] = v[k];
#pragma unroll
      for (int k = 0; k < D; ++k) a.tx[k * n + p] = x[k];
      a.tleaf[p] = L2;
    }
    if (D == 3 || t.scheme != 0) a.keyn[p] = knew;  // PIT rows: the key array is the leaf array
  }
  rank_movers<D == 3>(p, moved, knew, a.count, a.words, a.rank);
}

}  // namespace pic
