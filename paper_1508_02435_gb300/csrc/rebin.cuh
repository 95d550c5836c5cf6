// Stable counting sort of the pushed particles into their buckets (included by
// kernels.cu).
//
// The storage order before the step is sorted by old key, and a bucket's new
// order is: its stayers in storage order, then its movers in storage order.
//   push       one ballot word of movers per warp; every mover takes a rank
//              among the movers of its new key from the key's atomic counter
//              (the ranks of a bucket are those of the movers, in any order)
//   words      exclusive scan of the words' mover counts: with it the movers,
//              hence the stayers, before any particle are one load and a popc
//   keys       stayers of bucket k = its old size less the movers among them;
//              scan of stayers + movers: bucket start, first mover slot (base)
//              and the shift that takes a stayer to its slot
//   place      perm[slot] = particle: stayers at p - movers(p) + shift[key],
//              movers at base[key] + rank
//   gather     a slot among the movers of its bucket counts the smaller
//              particle numbers of the bucket's mover slots: that is its place
//              in storage order.  Buckets with more than kRankMax movers are
//              sorted before the gather instead.
// No pass runs over one bucket per thread, and stayers take no atomic.
// Measured per step, before (a thread per bucket for the stayers and for the
// mover sort, a mover list, a second atomic) -> now: re-bin and permutation of
// the 2e8-particle 3D two-stream PIDT step 9.4 -> 5.7 ms (the push waits for the
// ranks, some 0.5 ms); whole step of 256 2D plasmas, 3.5e7 particles, 3.26 ->
// 1.50 ms; 1e7 free 2D particles 0.49 -> 0.16 ms.  Three launches fewer for large
// trees, eight for small ones.
#pragma once

namespace pic {

// Longest mover segment ordered by counting in the gather: m loads a slot, from
// the L1, against the warp's sort (256 2D plasmas, ten steps: 64 17.0 ms, 96 16.4,
// 128 16.2, 192 16.1, 384 16.2).
constexpr int kRankMax = 128;
static_assert(kRankMax == kRankSegment, "list sizes in launch.hpp");

// Movers before particle x in storage order.
struct MoverBits {
  const uint32_t *word;
  const int32_t *pre;
  __device__ __forceinline__ int32_t before(int32_t x) const {
    return pre[x >> 5] + __popc(word[x >> 5] & ((1u << (x & 31)) - 1u));
  }
};

// Ballot word of the warp's movers, and every mover's rank among the movers of
// its new key.  kRuns: one atomic per run of equal keys in adjacent lanes (3D,
// where most movers of a warp take distinct keys); else one per distinct key
// (2D, where repeats are often apart; measured faster on each).
template <bool kRuns>
__device__ __forceinline__ void rank_movers(int64_t p, bool mover, int32_t key, int32_t *count, uint32_t *words,
                                            int32_t *rank) {
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const unsigned below = (1u << lane) - 1u;
  const unsigned mv = __ballot_sync(full, mover);
  if (lane == 0) words[p >> 5] = mv;
  if (mv == 0u) return;
  int head, at, len;
  if (kRuns) {
    const int32_t prev = __shfl_up_sync(full, key, 1);
    const unsigned heads = __ballot_sync(full, mover && (lane == 0 || !((mv >> (lane - 1)) & 1u) || prev != key));
    head = 31 - __clz(heads & (below | (1u << lane)));
    at = lane - head;
    const unsigned stop = (heads | ~mv) & ~((2u << lane) - 1u);  // lanes above this one
    len = (stop ? __ffs(stop) - 1 : 32) - lane;
  } else {
    const unsigned peers = __match_any_sync(full, mover ? key : -1);
    head = __ffs(peers) - 1;
    at = __popc(peers & below);
    len = __popc(peers);
  }
  int32_t first = 0;
  if (mover && lane == head) first = atomicAdd(&count[key], len);
  first = __shfl_sync(full, first, head < 0 ? 0 : head);
  if (mover) rank[p] = first + at;
}

// Ranks of freshly converted particles (every particle a mover).
__global__ void k_count_all(const int32_t *key, int64_t n, int32_t *count, uint32_t *words, int32_t *rank) {
  const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool act = p < n;
  rank_movers<false>(p, act, act ? key[p] : 0, count, words, rank);
}

// ---- scans ----------------------------------------------------------------------

// Exclusive scan over the block; *total (may be NULL) gets the block's sum.
__device__ __forceinline__ int32_t block_exclusive_scan(int32_t v, int32_t *total) {
  __shared__ int32_t sh[32];
  int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t x = v;
  for (int o = 1; o < 32; o <<= 1) {
    int32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh[w] = x;
  __syncthreads();
  if (w == 0) {
    int32_t s = lane < (int)(blockDim.x >> 5) ? sh[lane] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      int32_t y = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += y;
    }
    sh[lane] = s;
  }
  __syncthreads();
  int32_t before = w > 0 ? sh[w - 1] : 0;
  if (total) *total = sh[(blockDim.x >> 5) - 1];
  int32_t r = before + x - v;
  __syncthreads();
  return r;
}

// Eight consecutive values from `base` (a multiple of 8), zero from n on.
__device__ __forceinline__ void load8(const int32_t *in, int64_t base, int64_t n, int32_t *v) {
  if (base + 8 <= n && ((uintptr_t)in & 15) == 0) {
    const int4 a = *(const int4 *)(in + base), b = *(const int4 *)(in + base + 4);
    v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
    v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
  } else {
    for (int i = 0; i < 8; ++i) v[i] = base + i < n ? in[base + i] : 0;
  }
}
__device__ __forceinline__ void store8(int32_t *out, int64_t base, int64_t n, const int32_t *v) {
  if (base + 8 <= n && ((uintptr_t)out & 15) == 0) {
    *(int4 *)(out + base) = make_int4(v[0], v[1], v[2], v[3]);
    *(int4 *)(out + base + 4) = make_int4(v[4], v[5], v[6], v[7]);
  } else {
    for (int i = 0; i < 8; ++i)
      if (base + i < n) out[base + i] = v[i];
  }
}

struct ScanInts {
  const int32_t *in;
  __device__ __forceinline__ void load(int64_t base, int64_t n, int32_t *v) const { load8(in, base, n, v); }
};
struct ScanWords {  // movers per ballot word
  const uint32_t *in;
  __device__ __forceinline__ void load(int64_t base, int64_t n, int32_t *v) const {
    load8((const int32_t *)in, base, n, v);
    for (int i = 0; i < 8; ++i) v[i] = __popc((uint32_t)v[i]);
  }
};

template <class In>
__global__ void k_scan_reduce(In in, int64_t n, int32_t *tile_sums) {
  int32_t v[kScanItems], s = 0, tot;
  in.load((int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems, n, v);
  for (int i = 0; i < kScanItems; ++i) s += v[i];
  block_exclusive_scan(s, &tot);
  if (threadIdx.x == 0) tile_sums[blockIdx.x] = tot;
}

// Single block: exclusive scan of the tile sums in place, total to *total.
__global__ void k_scan_tiles(int32_t *tile_sums, int64_t nt, int32_t *total) {
  int32_t carry = 0;
  for (int64_t base = 0; base < nt; base += blockDim.x) {
    int64_t i = base + threadIdx.x;
    int32_t v = i < nt ? tile_sums[i] : 0;
    int32_t tot;
    int32_t ex = block_exclusive_scan(v, &tot);
    if (i < nt) tile_sums[i] = carry + ex;
    carry += tot;
  }
  if (threadIdx.x == 0) *total = carry;
}

// The scan of one tile from `carry`; returns the tile's sum.
template <class In>
__device__ __forceinline__ int32_t scan_tile(const In &in, int64_t tile, int64_t n, int32_t carry, int32_t *out) {
  const int64_t base = tile * kScanTile + (int64_t)threadIdx.x * kScanItems;
  int32_t v[kScanItems], s = 0, tot;
  in.load(base, n, v);
  for (int i = 0; i < kScanItems; ++i) s += v[i];
  int32_t ex = block_exclusive_scan(s, &tot) + carry;
  for (int i = 0; i < kScanItems; ++i) {
    const int32_t x = v[i];
    v[i] = ex;
    ex += x;
  }
  store8(out, base, n, v);
  return tot;
}

template <class In>
__global__ void k_scan_apply(In in, int64_t n, const int32_t *tile_offsets, int32_t *out, const int32_t *total) {
  scan_tile(in, blockIdx.x, n, tile_offsets[blockIdx.x], out);
  if (blockIdx.x == 0 && threadIdx.x == 0) out[n] = *total;
}

// Up to kOneBlockTiles tiles: the whole scan in one block, one launch instead
// of three (2-3 us each).
constexpr int64_t kOneBlockTiles = 3;
template <class In>
__device__ __forceinline__ void scan_one(const In &in, int64_t n, int32_t *out, int32_t *total) {
  int32_t carry = 0;
  for (int64_t tile = 0; tile * kScanTile < n; ++tile) carry += scan_tile(in, tile, n, carry, out);
  if (threadIdx.x == 0) {
    out[n] = carry;
    *total = carry;
  }
}
template <class In>
__global__ void k_scan_one(In in, int64_t n, int32_t *out, int32_t *total) { scan_one(in, n, out, total); }

// Sum of the counts and the stayers of one tile of keys.
__global__ void k_keys_reduce(RebinArgs r, int32_t *tile_sums) {
  const int64_t width = (int64_t)blockDim.x * kScanItems, t0 = (int64_t)blockIdx.x * width;
  int32_t v[kScanItems], s = 0, tot;
  load8(r.count, t0 + (int64_t)threadIdx.x * kScanItems, r.n_keys, v);
  for (int i = 0; i < kScanItems; ++i) s += v[i];
  block_exclusive_scan(s, &tot);
  if (threadIdx.x == 0) {
    if (r.old_start) {
      const MoverBits mb{r.words, r.word_pre};
      const int64_t t1 = t0 + width < r.n_keys ? t0 + width : r.n_keys;
      const int32_t a = r.old_start[t0], b = r.old_start[t1];
      tot += (b - a) - (mb.before(b) - mb.before(a));
    }
    tile_sums[blockIdx.x] = tot;
  }
}

// One tile of keys: bucket starts, first mover slots, stayer shifts, the list
// of long mover segments and the largest bucket.  Returns the tile's sum.
__device__ __forceinline__ int32_t keys_tile(const RebinArgs &r, int64_t tile, int32_t carry) {
  const int64_t base = (tile * blockDim.x + threadIdx.x) * kScanItems, n = r.n_keys;
  int32_t mc[kScanItems], nst[kScanItems], sh[kScanItems], s = 0, tot, big = 0;
  load8(r.count, base, n, mc);
  for (int i = 0; i < kScanItems; ++i) nst[i] = sh[i] = 0;
  if (r.old_start && base < n) {
    const MoverBits mb{r.words, r.word_pre};
    int32_t os[kScanItems + 1];
    load8(r.old_start, base, n, os);
    for (int i = 0; i < kScanItems; ++i)
      if (base + i >= n) os[i] = (int32_t)r.n;
    os[kScanItems] = base + kScanItems <= n ? r.old_start[base + kScanItems] : (int32_t)r.n;
    int32_t before = os[0] - mb.before(os[0]);  // stayers before the bucket
    for (int i = 0; i < kScanItems; ++i) {
      const int32_t next = os[i + 1] == os[i] ? before : os[i + 1] - mb.before(os[i + 1]);
      nst[i] = next - before;
      sh[i] = -before;
      before = next;
    }
  }
  for (int i = 0; i < kScanItems; ++i) {
    s += mc[i] + nst[i];
    big = max(big, mc[i] + nst[i]);
  }
  int32_t ex = block_exclusive_scan(s, &tot) + carry;
  int32_t start[kScanItems], first[kScanItems];
  for (int i = 0; i < kScanItems; ++i) {
    start[i] = ex;
    first[i] = ex + nst[i];
    sh[i] += ex;
    ex += mc[i] + nst[i];
    if (mc[i] > kRankMax) {
      if (mc[i] <= kMedSeg) r.med[atomicAdd(r.scalars + 7, 1)] = (int32_t)(base + i);
      else r.large[atomicAdd(r.scalars + 5, 1)] = (int32_t)(base + i);
    }
  }
  store8(r.new_start, base, n, start);
  if (r.old_start) {
    store8(r.base, base, n, first);
    store8(r.shift, base, n, sh);
    big = __reduce_max_sync(0xffffffffu, big);
    if ((threadIdx.x & 31) == 0 && big > 0 && big > *(volatile int32_t *)(r.scalars + 2)) atomicMax(r.scalars + 2, big);
  }
  return tot;
}

__global__ void __launch_bounds__(1024) k_keys_apply(RebinArgs r, const int32_t *tile_offsets) {
  keys_tile(r, blockIdx.x, tile_offsets[blockIdx.x]);
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    r.new_start[r.n_keys] = r.scalars[0];
    if (!r.old_start) r.scalars[1] = (int32_t)r.n;
  }
}

// Both scans in one block (few words and few keys).
__global__ void __launch_bounds__(1024) k_scan_small(RebinArgs r) {
  if (r.old_start) {
    scan_one(ScanWords{r.words}, (r.n + 31) / 32, r.word_pre, r.scalars + 1);
    __syncthreads();
  } else if (threadIdx.x == 0) {
    r.scalars[1] = (int32_t)r.n;
  }
  int32_t carry = 0;
  for (int64_t tile = 0; tile * kScanTile < r.n_keys; ++tile) carry += keys_tile(r, tile, carry);
  if (threadIdx.x == 0) {
    r.new_start[r.n_keys] = carry;
    r.scalars[0] = carry;
  }
}

// ---- place, sort, gather ---------------------------------------------------------

// Four particles per thread: their lookups are in flight together (1e7 free 2D
// particles 46 -> 24 us; 2e8 two-stream particles 1.42 -> 1.39 ms).
constexpr int kPlaceVec = 4;
__global__ void __launch_bounds__(256) k_place(RebinArgs r) {
  const int64_t p0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * kPlaceVec;
  if (p0 >= r.n) return;
  const int m = r.n - p0 < kPlaceVec ? (int)(r.n - p0) : kPlaceVec;
  const int32_t *base = r.old_start ? r.base : r.new_start;
  int32_t k[kPlaceVec], rank[kPlaceVec], slot[kPlaceVec];
  const uint32_t word = r.old_start ? r.words[p0 >> 5] : 0xffffffffu;
  const int32_t pre = r.old_start ? r.word_pre[p0 >> 5] : 0;
  if (m == kPlaceVec) {
    const int4 a = *(const int4 *)(r.keyn + p0), b = *(const int4 *)(r.rank + p0);
    k[0] = a.x; k[1] = a.y; k[2] = a.z; k[3] = a.w;
    rank[0] = b.x; rank[1] = b.y; rank[2] = b.z; rank[3] = b.w;
  } else {
    for (int i = 0; i < kPlaceVec; ++i) {
      k[i] = i < m ? r.keyn[p0 + i] : -1;
      rank[i] = i < m ? r.rank[p0 + i] : 0;
    }
  }
#pragma unroll
  for (int i = 0; i < kPlaceVec; ++i) {
    const int lane = (int)(p0 & 31) + i;
    if (i >= m) slot[i] = -1;
    else if ((word >> lane) & 1u) slot[i] = base[k[i]] + rank[i];
    else slot[i] = r.shift[k[i]] + (int32_t)p0 + i - pre - __popc(word & ((1u << lane) - 1u));
  }
#pragma unroll
  for (int i = 0; i < kPlaceVec; ++i)
    if (slot[i] >= 0) r.perm[slot[i]] = (int32_t)p0 + i;
}

// One warp per listed segment of at most kMedSeg movers (grid-stride over the
// list): the segment is copied into the warp's shared slice, sorted by the
// bitonic network of segsort.cuh and copied back.
__global__ void __launch_bounds__(kMedThreads) k_sort_medium(RebinArgs r) {
  extern __shared__ int32_t sw[];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, wpb = kMedThreads / 32;
  int32_t *v = sw + wib * kMedSeg;
  const int32_t *first = r.old_start ? r.base : r.new_start;
  const int nm = r.scalars[7];
  for (int li = blockIdx.x * wpb + wib; li < nm; li += gridDim.x * wpb) {
    const int32_t k = r.med[li];
    const int32_t b = first[k], m = r.new_start[k + 1] - b;
    for (int i = lane; i < m; i += 32) v[i] = r.perm[b + i];
    __syncwarp();
    warp_sort_direct<int32_t>(v, m);
    for (int i = lane; i < m; i += 32) r.perm[b + i] = v[i];
    __syncwarp();
  }
}

// One block per long segment (grid-stride over the list): the in-place
// bitonic network of segsort.cuh, chunks of kLargeSeg in shared memory, so a
// bucket of any size sorts in O(m log^2 m).
__global__ void __launch_bounds__(kLargeThreads) k_sort_large(RebinArgs r) {
  extern __shared__ int32_t sv[];
  const int32_t *first = r.old_start ? r.base : r.new_start;
  const int nl = r.scalars[5];
  for (int li = blockIdx.x; li < nl; li += gridDim.x) {
    const int32_t k = r.large[li];
    const int32_t b = first[k], m = r.new_start[k + 1] - b;
    block_sort_global<int32_t, int32_t>(r.perm + b, nullptr, m, sv, nullptr, kLargeSeg);
    __syncthreads();
  }
}

// Where the particle i of key k at slot s of perm belongs.
struct SlotOrder {
  const int32_t *perm, *base, *new_start;
  __device__ __forceinline__ int32_t place(int32_t s, int32_t i, int32_t k) const {
    const int32_t b = base[k];
    if (s < b) return s;  // a stayer
    const int32_t e = new_start[k + 1];
    if (e - b == 1 || e - b > kRankMax) return s;
    int32_t at = b;
    for (int32_t j = b; j < e; ++j) at += perm[j] < i;
    return at;
  }
};

// The whole particle state into bucket order in one pass: positions and
// velocities ([D][n]), leaves, and keys (PIDT; PIT keys are the leaves) and ids
// where given.
// FP32: two slots per thread, a block apart, so that twice the scattered reads are
// in flight (ten steps of 256 2D plasmas 15.7 -> 15.0 ms; four slots 15.4); FP64
// has twice the bytes per read and gains nothing.
template <typename T>
__host__ __device__ constexpr int rows_per_thread() { return sizeof(T) == 4 ? 2 : 1; }
// kQuad: x is one float4 per particle (two offsets, two velocities).
template <typename T, int D, bool kQuad>
__global__ void __launch_bounds__(256) k_gather_state(
    SlotOrder so, int64_t n, const T *__restrict__ x, T *__restrict__ x2, const T *__restrict__ v, T *__restrict__ v2,
    const int32_t *__restrict__ leaf, int32_t *__restrict__ leaf2, const int32_t *__restrict__ key,
    int32_t *__restrict__ key2, const int32_t *__restrict__ ids, int32_t *__restrict__ ids2) {
  constexpr int kRowsVec = rows_per_thread<T>();
  const int64_t s0 = (int64_t)blockIdx.x * (256 * kRowsVec) + threadIdx.x;
  int32_t i[kRowsVec], L[kRowsVec], kk[kRowsVec], id[kRowsVec];
  T a[kRowsVec][D], b[kRowsVec][D];
#pragma unroll
  for (int u = 0; u < kRowsVec; ++u) i[u] = s0 + 256 * u < n ? so.perm[s0 + 256 * u] : -1;
#pragma unroll
  for (int u = 0; u < kRowsVec; ++u) {
    if (i[u] < 0) continue;
    L[u] = leaf[i[u]];
    kk[u] = key ? key[i[u]] : L[u];
    id[u] = ids ? ids[i[u]] : 0;
    if constexpr (kQuad) {
      const float4 q = __ldg((const float4 *)x + i[u]);
      a[u][0] = q.x;
      a[u][1] = q.y;
      b[u][0] = q.z;
      b[u][1] = q.w;
    } else {
#pragma unroll
      for (int k = 0; k < D; ++k) a[u][k] = x[k * n + i[u]];
#pragma unroll
      for (int k = 0; k < D; ++k) b[u][k] = v[k * n + i[u]];
    }
  }
#pragma unroll
  for (int u = 0; u < kRowsVec; ++u) {
    if (i[u] < 0) continue;
    const int64_t p = so.place((int32_t)(s0 + 256 * u), i[u], kk[u]);
#pragma unroll
    for (int k = 0; k < D; ++k) x2[k * n + p] = a[u][k];
#pragma unroll
    for (int k = 0; k < D; ++k) v2[k * n + p] = b[u][k];
    leaf2[p] = L[u];
    if (key) key2[p] = kk[u];
    if (ids) ids2[p] = id[u];
  }
}

// 32 bytes in one load (eight floats, four doubles), from a 32-byte boundary.
__device__ __forceinline__ void load32(const float *p, float *v) {
  asm("ld.global.nc.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
      : "l"(p));
}
__device__ __forceinline__ void load32(const double *p, double *v) {
  asm("ld.global.nc.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(v[0]), "=d"(v[1]), "=d"(v[2]), "=d"(v[3]) : "l"(p));
}

// The same from the pushed-state records of the 3D step (one or two 32-byte
// loads per particle instead of one scattered 4- or 8-byte load per array).
__global__ void k_gather_rec32(SlotOrder so, int64_t n, const float *__restrict__ rec, float *__restrict__ x2,
                               float *__restrict__ v2, int32_t *__restrict__ leaf2, int32_t *__restrict__ key2,
                               const int32_t *__restrict__ ids, int32_t *__restrict__ ids2) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int32_t i = so.perm[s];
  float r[8];
  load32(rec + 8 * (int64_t)i, r);
  const int32_t id = ids ? ids[i] : 0;
  const int64_t p = so.place((int32_t)s, i, __float_as_int(r[7]));
#pragma unroll
  for (int k = 0; k < 3; ++k) x2[k * n + p] = r[k];
#pragma unroll
  for (int k = 0; k < 3; ++k) v2[k * n + p] = r[3 + k];
  leaf2[p] = __float_as_int(r[6]);
  if (key2) key2[p] = __float_as_int(r[7]);
  if (ids) ids2[p] = id;
}

__global__ void k_gather_rec64(SlotOrder so, int64_t n, const double *__restrict__ rec, double *__restrict__ x2,
                               double *__restrict__ v2, int32_t *__restrict__ leaf2, int32_t *__restrict__ key2,
                               const int32_t *__restrict__ ids, int32_t *__restrict__ ids2) {
  const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= n) return;
  const int32_t i = so.perm[s];
  double r[8];
  load32(rec + 8 * (int64_t)i, r);
  load32(rec + 8 * (int64_t)i + 4, r + 4);
  const uint64_t lk = (uint64_t)__double_as_longlong(r[6]);
  const int32_t id = ids ? ids[i] : 0, k = (int32_t)(uint32_t)(lk >> 32);
  const int64_t p = so.place((int32_t)s, i, k);
#pragma unroll
  for (int a = 0; a < 3; ++a) x2[a * n + p] = r[a];
#pragma unroll
  for (int a = 0; a < 3; ++a) v2[a * n + p] = r[3 + a];
  leaf2[p] = (int32_t)(uint32_t)lk;
  if (key2) key2[p] = k;
  if (ids) ids2[p] = id;
}

// ---- launches ----------------------------------------------------------------------

template <class In>
static void exclusive_scan(In in, int64_t n, int32_t *out, int32_t *tile_sums, int32_t *total, cudaStream_t s) {
  const int64_t nt = std::max<int64_t>(1, scan_tiles_needed(n));
  if (nt <= kOneBlockTiles) {
    COUNT(1);
    k_scan_one<<<1, kScanThreads, 0, s>>>(in, n, out, total);
    return;
  }
  COUNT(3);
  k_scan_reduce<<<(unsigned)nt, kScanThreads, 0, s>>>(in, n, tile_sums);
  k_scan_tiles<<<1, kScanThreads, 0, s>>>(tile_sums, nt, total);
  k_scan_apply<<<(unsigned)nt, kScanThreads, 0, s>>>(in, n, tile_sums, out, total);
}

int64_t scan_tiles_needed(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

void launch_exclusive_scan(const int32_t *in, int64_t n, int32_t *out, int32_t *tile_sums, int32_t *total,
                           cudaStream_t s) {
  exclusive_scan(ScanInts{in}, n, out, tile_sums, total, s);
}

void launch_count_all(const int32_t *key, int64_t n, int32_t *count, uint32_t *words, int32_t *rank, cudaStream_t s) {
  if (n > 0) { COUNT(1); k_count_all<<<grid_for(n), kBlock, 0, s>>>(key, n, count, words, rank); }
}

void launch_rebin(const RebinArgs &r, cudaStream_t s) {
  const int64_t nw = (r.n + 31) / 32, tw = scan_tiles_needed(nw), tk = std::max<int64_t>(1, scan_tiles_needed(r.n_keys));
  if ((!r.old_start || tw <= kOneBlockTiles) && tk <= kOneBlockTiles) {
    COUNT(1);
    k_scan_small<<<1, kScanThreads, 0, s>>>(r);
  } else {
    if (r.old_start) exclusive_scan(ScanWords{r.words}, nw, r.word_pre, r.tile_sums2, r.scalars + 1, s);
    // up to a million keys in quarter tiles: more blocks share the lookups (59,049
    // keys: 14 -> 7 us)
    const unsigned threads = r.n_keys < 1000000 ? kScanThreads / 4 : kScanThreads;
    const int64_t nt = (r.n_keys + threads * kScanItems - 1) / (threads * kScanItems);
    COUNT(3);
    k_keys_reduce<<<(unsigned)nt, threads, 0, s>>>(r, r.tile_sums);
    k_scan_tiles<<<1, kScanThreads, 0, s>>>(r.tile_sums, nt, r.scalars + 0);
    k_keys_apply<<<(unsigned)nt, threads, 0, s>>>(r, r.tile_sums);
  }
  if (r.n <= 0) return;
  { COUNT(1); k_place<<<grid_for((r.n + kPlaceVec - 1) / kPlaceVec), kBlock, 0, s>>>(r); }
  if (r.n > kRankMax) {
    COUNT(1);
    k_sort_medium<<<kMedBlocks, kMedThreads, sizeof(int32_t) * kMedSeg * (kMedThreads / 32), s>>>(r);
  }
  if (r.n > kMedSeg) {
    COUNT(1);
    k_sort_large<<<304, kLargeThreads, sizeof(int32_t) * kLargeSeg, s>>>(r);
  }
}

void launch_gather_state(bool split, const RebinArgs &r, int d, const void *x, void *x2, const void *v, void *v2,
                         const int32_t *leaf, int32_t *leaf2, const int32_t *key, int32_t *key2, const int32_t *ids,
                         int32_t *ids2, cudaStream_t s) {
  if (r.n <= 0) return;
  COUNT(1);
  const SlotOrder so{r.perm, r.old_start ? r.base : r.new_start, r.new_start};
  const unsigned g = grid_for(r.n, 256 * (split ? rows_per_thread<float>() : rows_per_thread<double>()));
  if (split) {
    if (d == 3)
      k_gather_state<float, 3, false><<<g, 256, 0, s>>>(so, r.n, (const float *)x, (float *)x2, (const float *)v,
                                                           (float *)v2, leaf, leaf2, key, key2, ids, ids2);
    else if (v)
      k_gather_state<float, 2, false><<<g, 256, 0, s>>>(so, r.n, (const float *)x, (float *)x2, (const float *)v,
                                                           (float *)v2, leaf, leaf2, key, key2, ids, ids2);
    else
      k_gather_state<float, 2, true><<<g, 256, 0, s>>>(so, r.n, (const float *)x, (float *)x2, nullptr, (float *)v2,
                                                          leaf, leaf2, key, key2, ids, ids2);
  } else if (d == 3) {
    k_gather_state<double, 3, false><<<g, 256, 0, s>>>(so, r.n, (const double *)x, (double *)x2, (const double *)v,
                                                          (double *)v2, leaf, leaf2, key, key2, ids, ids2);
  } else {
    k_gather_state<double, 2, false><<<g, 256, 0, s>>>(so, r.n, (const double *)x, (double *)x2, (const double *)v,
                                                          (double *)v2, leaf, leaf2, key, key2, ids, ids2);
  }
}

void launch_gather_records(bool split, const RebinArgs &r, const void *rec, void *x2, void *v2, int32_t *leaf2,
                           int32_t *key2, const int32_t *ids, int32_t *ids2, cudaStream_t s) {
  if (r.n <= 0) return;
  COUNT(1);
  const SlotOrder so{r.perm, r.old_start ? r.base : r.new_start, r.new_start};
  if (split)
    k_gather_rec32<<<grid_for(r.n), kBlock, 0, s>>>(so, r.n, (const float *)rec, (float *)x2, (float *)v2, leaf2, key2,
                                                    ids, ids2);
  else
    k_gather_rec64<<<grid_for(r.n), kBlock, 0, s>>>(so, r.n, (const double *)rec, (double *)x2, (double *)v2, leaf2,
                                                    key2, ids, ids2);
}

}  // namespace pic
