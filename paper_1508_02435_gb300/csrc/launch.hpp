// Kernel launch interface between the C-ABI layer (pic_api.cu) and the
// kernels (kernels.cu).  All launches are stream-ordered on `s`.
#pragma once
#include <cuda_runtime.h>

#include <cstdint>

namespace pic {

struct DevTree;
struct TabEntry;

struct Push64Args {
  int64_t n;
  const double *x, *v;          // current state, bucket-sorted
  const int32_t *leaf, *key;    // key used by PIDT only
  double2 *rec;                 // [n][4] pushed state: x0 x1 | x2 v0 | v1 v2 | (leaf, key as bits), 0, or NULL:
  double *tx, *tv;              // the pushed state in rows [d][n] and tleaf
  int32_t *tleaf, *keyn;        // keyn: new key per particle (PIT: the leaf)
  const double *E;              // [d][n_vert]; NULL: no field (the particle-handling move, no kick)
  const double *Ec;             // adaptive trees: field at every leaf corner [leaf][corner][axis]
  double qmdt, dt;
  int32_t *count;               // movers per key, zeroed before the launch
  uint32_t *words;              // one ballot word of movers per 32 particles
  int32_t *rank;                // movers: rank among the movers of the new key
  int32_t *err;
  int32_t reflect;              // 1: reflecting walls of the unit box; 0: periodic
  int32_t flops;                // artificial floating-point operations per particle move
};

struct Push32Args {
  int64_t n;
  const float *o, *v;
  const int32_t *leaf, *key;
  float4 *rec;                  // [n][2] pushed state: o0 o1 o2 v0 | v1 v2 leaf key (leaf, key as bits), or NULL:
  float *to, *tv;               // the pushed state in rows [d][n] and tleaf
  int32_t *tleaf, *keyn;        // keyn: new key per particle (PIT: the leaf)
  const float *E;               // NULL (and Ec NULL): no field (the particle-handling move, no kick)
  const float *Ec;              // adaptive trees: field at every leaf corner [leaf][corner][axis]
  float qmdt;
  double dt;
  float sl[19];                 // RN32(dt * 3^level) per level
  int32_t *count;
  uint32_t *words;
  int32_t *rank;
  int32_t *err;
  int32_t reflect;              // 1: reflecting walls of the unit box; 0: periodic
  int32_t flops;                // artificial floating-point operations per particle move
};

struct RebinArgs {
  int64_t n, n_keys;
  const int32_t *count;         // movers per new key
  const int32_t *keyn;          // new key per particle (storage order)
  const int32_t *old_start;     // CSR of the current order, NULL for fresh particles (all movers)
  int32_t *new_start;           // [n_keys + 1]
  const uint32_t *words;        // mover bits
  int32_t *word_pre;            // [words + 1] movers before each word
  const int32_t *rank;
  int32_t *base, *shift;        // [n_keys] first mover slot; stayer slot less stayers before
  int32_t *perm;
  int32_t *med, *large;         // keys with long mover segments
  int32_t *tile_sums, *tile_sums2;
  int32_t *scalars;             // [0] n, [1] movers, [2] max bucket, [5] long, [7] medium segments (2, 5, 7 zeroed before)
};
// Mover segments of up to this many are put in order by the gather; longer
// ones (at most n / (kRankSegment + 1)) are listed and sorted.
constexpr int64_t kRankSegment = 128;

// Elements per tile of launch_exclusive_scan: a scan of n elements writes
// scan_tiles_needed(n) = ceil(n / kScanTileElems) tile sums.
constexpr int64_t kScanTileElems = 8192;

// Kernels launched by this library so far (all handles of the process).
int64_t launches();
void count_launches(int64_t k);

// Brick path (uniform trees, PIT, split precision): see brick.cu.
struct BrickGeom {
  int d, kb, B, LB, nbx, depth;  // B = 3^kb leaves per brick axis, LB = B^d, nbx bricks per axis
  int64_t n_bricks;
  const uint32_t *decodeL;       // local depth-first index -> x | y << 10 | z << 20
};

// Staging between K1 and K2: every pushed particle is appended to the area of
// its destination unit U (half a brick: local leaves below or from (LB+1)/2),
// slots [U cap, U cap + cap) of each row; arrivals beyond cap go to an
// overflow list.
struct BrickStage {
  int32_t cap;                   // slots per destination unit (a multiple of 8)
  int64_t row;                   // slots in all (2 n_bricks cap, padded)
  float *rec;                    // [row][4] o0 o1 v0 v1; 3D: o0 o1 o2 v0, then [row][2] v1 v2
  uint16_t *code;                // destination local leaf | stayer bit
  uint32_t *key;                 // moved << 31 | storage index before the step (canonical order)
  int32_t *id;                   // particle ids (tracked ids only)
  int32_t *fill;                 // [2 n_bricks] arrivals per destination unit (may exceed cap)
  int32_t *over;                 // units listed for the global-memory pull
  int32_t *over_units;           // [2 n_bricks] units over their staging capacity (any order)
  int32_t *ovf_n;                // overflow count
  int32_t ovf_cap;
  int32_t *ovf_dest;             // [ovf_cap] destination unit
  float *ovf_o, *ovf_v;          // [D][ovf_cap]
  uint16_t *ovf_code;
  uint32_t *ovf_key;
  int32_t *ovf_id;
};

struct BrickPushArgs {
  int64_t n;
  const float *o, *v;
  const int32_t *start;          // current leaf offsets
  const int32_t *ids;            // NULL unless ids are tracked
  const float *E;
  const void *Ebrick;            // the field brick by brick: (9+1)^d vertices per brick, float4 (3D) / float2 (2D)
  float qmdt, sl;
  BrickStage st;
  int32_t *n_movers;
  int32_t *err;
  long long wait_cycles;         // limit of the bounded wait for the bulk copies (SM clocks)
};

struct BrickPullArgs {
  int64_t n;
  BrickStage st;
  const int32_t *fstart;         // overflow arrivals sorted per destination brick
  int32_t *fstart_w;
  const int32_t *ovf_sorted;     // overflow list positions, grouped by destination brick
  int32_t *ovf_sorted_w;
  int32_t *tot_w;
  const int32_t *tot;            // incoming particles per destination brick
  const int32_t *bstart;
  int32_t *bstart_w;
  float *o, *v;
  int32_t *ids;
  int32_t *new_start;
  int32_t *max_bucket;
  int32_t *err;
  float *part;                   // leaf-corner deposit partials of the new positions, or NULL
  uint32_t *fb_key;              // [n] scratch of the global-memory kernel
  int32_t *fb_idx;
  long long wait_cycles;         // limit of the bounded wait for the bulk copies (SM clocks)
};

cudaError_t brick_configure(const BrickGeom &g);
int32_t brick_stage_cap(int64_t n, int64_t n_units);  // staging slots per destination unit
bool brick_crowded(int64_t n, int64_t n_units);       // most half bricks hold more than the shared-memory kernels take
void launch_brick_push(const DevTree &t, const BrickGeom &g, const BrickPushArgs &pa, cudaStream_t s);
void launch_brick_pull(const DevTree &t, const BrickGeom &g, const BrickPullArgs &qa, int32_t *fcount,
                       int32_t *fcursor, int32_t *tile_sums, int32_t *scratch_total, cudaStream_t s);
void launch_expand_leaves(const int32_t *start, int64_t n_leaves, int32_t *leaf, cudaStream_t s);
// The vertex field E[d][n_vert] re-laid brick by brick for K1: brick b holds
// the (9+1)^d vertices from its origin on (periodic), x fastest, one vector
// (E_x, E_y[, E_z, 0]) per vertex.
void launch_brick_field(const DevTree &t, const BrickGeom &g, const float *E, float *Ebrick, cudaStream_t s);
// One CTA arms an mbarrier for 16 bytes that are never sent and waits for it
// with the bounded wait of the brick kernels (limit `cycles`); *flag becomes
// 1 when the wait gave up (the expected outcome), 2 if it completed.
void launch_wait_selftest(long long cycles, int32_t *flag, cudaStream_t s);

cudaError_t set_constants(cudaStream_t s);
int64_t scan_tiles_needed(int64_t n);

void launch_init64(const DevTree &t, double *x, int64_t n, int32_t *leaf, int32_t *key, int32_t *err,
                   cudaStream_t s);
void launch_init32(const DevTree &t, const double *x, const double *v, int64_t n, int32_t *leaf, float *o,
                   float *vf, int32_t *key, int32_t *err, cudaStream_t s);
// Rows of a split state: offsets and velocities [d][n], leaves.
struct StateRows {
  float *o, *v;
  int32_t *leaf;
};
// A given split state as fresh particles: keys, ranks, *unsorted = 1 unless the
// keys ascend; the state itself into the records (3D) or, unless it is `given`
// there, the rows r (2D).  *err |= 2 where a leaf or an offset is out of range;
// such a value is stored as 0, in the rows too.
void launch_fresh32(const DevTree &t, const int32_t *leaf, const float *o, const float *v, int64_t n, int32_t *key,
                    void *rec, const StateRows &r, bool given, int32_t *count, uint32_t *words, int32_t *rank,
                    int32_t *unsorted, int32_t *err, cudaStream_t s);
void launch_record_rows(int64_t n, const void *rec, const StateRows &r, cudaStream_t s);
void launch_check_sorted(const int32_t *key, int64_t n, int32_t *flag, cudaStream_t s);
void launch_count_all(const int32_t *key, int64_t n, int32_t *count, uint32_t *words, int32_t *rank, cudaStream_t s);
// *changed = 1 unless every leaf of t passes the particles-per-cell criterion,
// i.e. unless the criterion gives back the installed tree.  The counts of its
// cells on levels dmin .. dmax-1 (level m at count + coff[m]) come from the
// buckets (start); no particle is read.
void launch_adapt_check(const DevTree &t, const int32_t *start, int32_t *count, const int64_t *coff, int dmin, int dmax,
                        int64_t ppc, int32_t *changed, cudaStream_t s);
// Threshold bits (count > ppc) of every cell on levels dmin .. dmax-1: particles
// counted per cell of level dmax-1, summed up child by child; level m's counts
// at count + cnt_off[m], its bits at bits + bit_off[m].
void launch_adapt_bits(const DevTree &t, bool split, const void *pos, const int32_t *leaf, int64_t n, int dmin, int dmax,
                       int64_t ppc, int32_t *count, const int64_t *cnt_off, uint32_t *bits, const int64_t *bit_off,
                       cudaStream_t s);
// One record per particle from the rows of a fresh 3D state.
void launch_make_records(bool split, int64_t n, const void *x, const void *v, const int32_t *leaf, const int32_t *key,
                         void *rec, cudaStream_t s);
void launch_relocate32(const DevTree &from, const DevTree &to, const int32_t *leaf, const float *o, const float *v,
                       int64_t n, int32_t *leaf2, float *o2, float *v2, cudaStream_t s);

// Vertex charges and FP64 total from leaf-corner partials already computed.
void launch_vertex_charge(const DevTree &t, bool split, const void *part, void *Q, double *block_sum,
                          double *total, cudaStream_t s);
// Charges per instance: q and ion density come from the instance table;
// total[0] is the FP64 sum over all vertices, total[1 + i] per instance.
void launch_deposit(const DevTree &t, bool split, const int32_t *start, const void *pos, int64_t n, void *part,
                    void *Q, double *block_sum, double *total, cudaStream_t s);
// Assembled rows of the FP64 solve on an adaptive tree, in slices of 32 rows; val
// NULL: not assembled.
struct RowMatrix {
  const int32_t *ptr;           // first entry of every slice
  const int32_t *col;
  const double *val;
  const double *scale;          // omega / diag per vertex
  const double *rest;           // 2D: minus the sum of the row's entries, zero but for their rounding
};
// Whether the solve of t runs as one cluster (small uniform trees).
bool resident_solve_fits(const DevTree &t, bool split);
// part: scratch of one value per leaf corner, free after the vertex charges are
// summed.
void launch_solve(const DevTree &t, const RowMatrix &A, bool split, const void *Q, const double *total, void *b, void *V,
                  void *Vtmp, void *part, int sweeps, double omega, double *block_sum, double *resid2, cudaStream_t s);
// Assembly of the rows: entries per slice (row_slices of them), their scan is
// RowMatrix::ptr, then columns and values.
int64_t row_slices(const DevTree &t);
int64_t row_capacity(const DevTree &t);  // entries reserved for them
void launch_row_count(const DevTree &t, int32_t *slice, int32_t *too_long, cudaStream_t s);
void launch_row_fill(const DevTree &t, const int32_t *ptr, double omega, int32_t *cols, double *vals, double *scale,
                     double *rest, cudaStream_t s);
void launch_efield(const DevTree &t, bool split, const void *V, void *E, void *part, cudaStream_t s);
void launch_push64(const DevTree &t, const Push64Args &a, cudaStream_t s);
void launch_push32(const DevTree &t, const Push32Args &a, cudaStream_t s);
// Field at every leaf corner of an adaptive tree, [leaf][corner][axis], the
// corner expansion applied once per field.
size_t corner_field_bytes(const DevTree &t, bool split);
void launch_corner_field(const DevTree &t, bool split, const void *E, void *Ec, cudaStream_t s);
// Coordinates (x, y, z) and level (w) of every leaf.
void launch_leaf_records(const DevTree &t, int4 *rec, cudaStream_t s);
// The jump table of t (jump_level and jump_cells set) into `jump`.
void launch_jump_table(const DevTree &t, TabEntry *jump, cudaStream_t s);
void launch_exclusive_scan(const int32_t *in, int64_t n, int32_t *out, int32_t *tile_sums, int32_t *total,
                           cudaStream_t s);
void launch_rebin(const RebinArgs &r, cudaStream_t s);
// The pushed state into bucket order after launch_rebin, in one kernel: from the
// rows (positions, velocities [d][n], leaves and, where not NULL, keys and ids;
// split: float, else double; 2D, split, v NULL: x holds a float4 per particle,
// launch_pack_rows) or from the records of the 3D step.  key NULL: PIT.
void launch_pack_rows(int64_t n, const float *o, const float *v, void *quad, cudaStream_t s);
void launch_gather_state(bool split, const RebinArgs &r, int d, const void *x, void *x2, const void *v, void *v2,
                         const int32_t *leaf, int32_t *leaf2, const int32_t *key, int32_t *key2, const int32_t *ids,
                         int32_t *ids2, cudaStream_t s);
void launch_gather_records(bool split, const RebinArgs &r, const void *rec, void *x2, void *v2, int32_t *leaf2,
                           int32_t *key2, const int32_t *ids, int32_t *ids2, cudaStream_t s);
void launch_absolute_split(const DevTree &t, const int32_t *leaf, const float *o, int64_t n, double *x,
                           cudaStream_t s);
void launch_widen(const float *in, int64_t n, double *out, cudaStream_t s);
void launch_gather_only(const DevTree &t, bool split, const void *pos, const int32_t *leaf, int64_t n,
                        const void *Ev, void *Ep, cudaStream_t s);
void launch_half_kick(bool split, const void *Ep, int64_t n_total, double c, void *v, cudaStream_t s);
// raPIDT v_max: per leaf (largest |velocity component| of its particles, or
// of its vertices' particles for PIDT), then per node of the level-ordered
// tree bottom-up (level_begin[l] = first node of level l, depth + 2 entries).
void launch_vmax(const DevTree &t, bool split, const int32_t *start, const void *v, int64_t n, const int32_t *child0,
                 const int32_t *leaf_of_node, const int64_t *level_begin, int depth, double *leaf_vmax,
                 double *node_vmax, cudaStream_t s);
// lift and drop counts (diagnostic): counts[0..2] = lifts, drops, tunnellers
void launch_scatter_by_id(const int32_t *ids, const int32_t *leaf, int64_t n, int32_t *by_id, cudaStream_t s);
void launch_lift_drop(const DevTree &t, const int32_t *ids, const int32_t *leaf, const int32_t *old_by_id, int64_t n,
                      unsigned long long *counts, cudaStream_t s);
// PIDT: pv_level / pv_j are the owner-vertex table (adaptive trees; unused on
// uniform ones); counts[0..2] = lifts, drops, tunnellers.
void launch_lift_drop_pidt(const DevTree &t, const int32_t *pv_level, const int32_t *pv_j, const int32_t *ids,
                           const int32_t *leaf, const int32_t *key, const int32_t *old_leaf_by_id,
                           const int32_t *old_key_by_id, int64_t n, unsigned long long *counts, cudaStream_t s);

}  // namespace pic
