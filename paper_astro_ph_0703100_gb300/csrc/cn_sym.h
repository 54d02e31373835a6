// Symmetric (each unordered pair once) evaluation of an i set equal to the
// j set: launch arguments and entry points of the sym_kernel forms.
#pragma once

#include "cn_kernels.h"

namespace cn {

// The unordered pairs of n particles, cut into rows of tiles. A tile is B =
// threads x K particles (the i side, in registers); a block is 32
// particles (the j side of one warp sweep). Row I is the blocks from the
// tile's own first block on: the tile's own B / 32 ("diagonal") blocks,
// evaluated one-sided, then all later ones, evaluated for both sides. A
// block costs kSymCostDiag or kSymCostPair; the cost line of a launch's rows
// is split evenly over its CTAs, and a unit (I, block) belongs to the CTA
// in whose part it starts. A part is at least kSymCostPair long, so that
// every CTA has a unit.
constexpr int kSymCostDiag = 3;
constexpr int kSymCostPair = 4;
constexpr int kSymBlock = 32;

struct SymGrid {
  int64_t n;           // particles
  int32_t n_tiles;     // ceil(n / tile)
  int32_t n_blocks;    // ceil(n / 32)
  int32_t tile_blocks; // B / 32
  int32_t row0;        // the launch's rows
  int32_t row1;
  int32_t grid;        // its CTAs
  int64_t cost0;       // cost line position of row0
  int64_t cost;        // its length over rows row0 .. row1 - 1

  // cost line position of a row's first unit (row <= n_tiles)
  __host__ __device__ int64_t row_start(int64_t row) const {
    const int64_t r = row < n_tiles ? row : n_tiles - 1;
    int64_t s = static_cast<int64_t>(kSymCostDiag) * tile_blocks * r +
                static_cast<int64_t>(kSymCostPair) * (r * n_blocks - static_cast<int64_t>(tile_blocks) * (r * (r + 1) / 2));
    if (row >= n_tiles) s += static_cast<int64_t>(kSymCostDiag) * (n_blocks - r * tile_blocks);
    return s;
  }
  // one past a row's last diagonal block
  __host__ __device__ int32_t diag_end(int32_t row) const {
    const int64_t e = static_cast<int64_t>(row + 1) * tile_blocks;
    return static_cast<int32_t>(e < n_blocks ? e : n_blocks);
  }
  // where CTA g's part of the cost line begins
  __host__ __device__ int64_t part(int64_t g) const { return cost0 + (g * cost + grid - 1) / grid; }
  // the CTA that holds the unit starting at s
  __host__ __device__ int64_t owner(int64_t s) const { return ((s - cost0) * grid) / cost; }
};

// A CTA's walk along the cost line, one staged chunk (up to `most` blocks of
// one row, all diagonal or all not) at a time.
struct SymCursor {
  int64_t s;    // cost line position of the next unit
  int32_t row;
  int32_t blk;  // its block

  // the first unit starting at or after x
  __host__ __device__ void seek(const SymGrid& g, int64_t x) {
    int32_t lo = g.row0, hi = g.row1 - 1;
    while (lo < hi) {
      const int32_t mid = (lo + hi + 1) >> 1;
      if (g.row_start(mid) <= x)
        lo = mid;
      else
        hi = mid - 1;
    }
    row = lo;
    s = g.row_start(lo);
    const int64_t r = x - s;
    const int32_t first = lo * g.tile_blocks, nd = g.diag_end(lo) - first;
    int64_t idx;
    if (r <= static_cast<int64_t>(kSymCostDiag) * nd)
      idx = (r + kSymCostDiag - 1) / kSymCostDiag;
    else
      idx = nd + (r - static_cast<int64_t>(kSymCostDiag) * nd + kSymCostPair - 1) / kSymCostPair;
    s += idx <= nd ? kSymCostDiag * idx : static_cast<int64_t>(kSymCostDiag) * nd + kSymCostPair * (idx - nd);
    blk = first + static_cast<int32_t>(idx);
    if (blk >= g.n_blocks) {
      ++row;
      blk = row * g.tile_blocks;
    }
  }
  // takes the next chunk before position `end`: its row, first block, blocks
  // and kind; advances past it
  __host__ __device__ void take(const SymGrid& g, int64_t end, int32_t most, int32_t* row_out, int32_t* blk_out,
                                int32_t* count, bool* diag) {
    const int32_t de = g.diag_end(row);
    const bool dg = blk < de;
    const int32_t w = dg ? kSymCostDiag : kSymCostPair;
    const int64_t left = dg ? (end - s + kSymCostDiag - 1) / kSymCostDiag : (end - s + kSymCostPair - 1) / kSymCostPair;
    int32_t c = (dg ? de : g.n_blocks) - blk;
    if (c > most) c = most;
    if (c > left) c = static_cast<int32_t>(left);
    *row_out = row;
    *blk_out = blk;
    *count = c;
    *diag = dg;
    s += static_cast<int64_t>(w) * c;
    blk += c;
    if (blk >= g.n_blocks) {
      ++row;
      blk = row * g.tile_blocks;
    }
  }
};

// An ensemble's rows: every cluster's own triangle, one after the other on
// one cost line. Slots are kept for the off-diagonal blocks only.
struct SymRow {
  int64_t cost;      // cost line position of the row's first unit
  int64_t p0;        // the cluster's first particle
  int64_t slot;      // j-side slots: sum d of block b is at slot + d * plane + (b - diag_end) * 32
  int32_t n;         // the cluster's particles
  int32_t n_blocks;  // its blocks
  int32_t blk0;      // the row's first block
  int32_t diag_end;  // one past its last diagonal block
  int32_t plane;     // (n_blocks - diag_end) * 32
  float eps2;

  __host__ __device__ int64_t length() const {
    return static_cast<int64_t>(kSymCostDiag) * (diag_end - blk0) +
           static_cast<int64_t>(kSymCostPair) * (n_blocks - diag_end);
  }
  // cost line position of its last unit
  __host__ __device__ int64_t last() const {
    return cost + length() - (diag_end < n_blocks ? kSymCostPair : kSymCostDiag);
  }
};

// seek and take along an ensemble's rows (as SymCursor's own, by table)
inline __host__ __device__ void sym_seek_rows(SymCursor& c, const SymRow* rows, int32_t n_rows, int64_t x) {
  int32_t lo = 0, hi = n_rows - 1;
  while (lo < hi) {
    const int32_t mid = (lo + hi + 1) >> 1;
    if (rows[mid].cost <= x)
      lo = mid;
    else
      hi = mid - 1;
  }
  const SymRow r = rows[lo];
  const int64_t left = x - r.cost, nd = r.diag_end - r.blk0;
  int64_t idx;
  if (left <= kSymCostDiag * nd)
    idx = (left + kSymCostDiag - 1) / kSymCostDiag;
  else
    idx = nd + (left - kSymCostDiag * nd + kSymCostPair - 1) / kSymCostPair;
  c.row = lo;
  c.s = r.cost + (idx <= nd ? kSymCostDiag * idx : kSymCostDiag * nd + kSymCostPair * (idx - nd));
  c.blk = r.blk0 + static_cast<int32_t>(idx);
  if (c.blk >= r.n_blocks) {
    ++c.row;
    c.blk = c.row < n_rows ? rows[c.row].blk0 : 0;
  }
}
inline __host__ __device__ void sym_take_rows(SymCursor& c, const SymRow* rows, int32_t n_rows, int64_t end,
                                              int32_t most, int32_t* row, int32_t* blk, int32_t* count, bool* diag) {
  const SymRow r = rows[c.row];
  const bool dg = c.blk < r.diag_end;
  const int64_t left = dg ? (end - c.s + kSymCostDiag - 1) / kSymCostDiag : (end - c.s + kSymCostPair - 1) / kSymCostPair;
  int32_t n = (dg ? r.diag_end : r.n_blocks) - c.blk;
  if (n > most) n = most;
  if (n > left) n = static_cast<int32_t>(left);
  *row = c.row;
  *blk = c.blk;
  *count = n;
  *diag = dg;
  c.s += static_cast<int64_t>(dg ? kSymCostDiag : kSymCostPair) * n;
  c.blk += n;
  if (c.blk >= r.n_blocks) {
    ++c.row;
    c.blk = c.row < n_rows ? rows[c.row].blk0 : 0;
  }
}

// 32 particles of an ensemble in the merge: their block, their row and their
// cluster's first row.
struct SymMergeBlock {
  int32_t first;
  int32_t row;
  int32_t blk;
};

// A launch. Sum d of the i side of particle p goes to plane d of the (CTA c,
// row I) segment, slots_seg[((c + I - row0) * planes + d) * tile + p - I tile]
// (c + I - row0 is unique per segment, since along the cost line neither the
// CTA nor the row decreases); the force forms have a second plane each, for
// the sums' low words where both_words is set. Sum d of the j side under row I to
// slots_j[((I - row0) * sums + d) * n_pad + p].
struct SymArgs {
  SymGrid g;
  const float4* pos;   // [n] (x, y, z, m)
  const float4* rec2;  // second record (velocity, loss weight) or NULL
  float* slots_seg;
  float* slots_j;
  int* status;
  int32_t both_words;
  int64_t n_seg;       // allocated segments
  int64_t n_pad;       // n_blocks * 32
  int32_t chunk;       // j records per ring stage (multiple of 32)
  int32_t fold;        // blocks summed in registers between folds (at least a stage's)
  int32_t stages;
  float eps2;
  float fast;          // forms with a second record: its largest component for the mass-free terms
  uint64_t wait_ns;
  const SymRow* rows;  // ensembles: the rows (g then holds only the cost line and the CTAs)
  int32_t n_rows;
};

// Per-particle merge of one launch: the j-side slots of rows I < P (the
// particle's tile) in ascending order, then the segments of row P in CTA
// order, summed in (hi, lo) pairs by TwoSum; with several bands the sums
// are carried in FP64 and the last band writes the outputs.
struct SymMerge {
  SymGrid g;
  const float* slots_seg;
  const float* slots_j;
  double* carry;      // [sums][n_pad] running sums, NULL with a single band
  float* out[3];      // outputs, by form
  int64_t n_pad;
  int32_t tile;
  int32_t first;
  int32_t last;
  const SymRow* rows;            // ensembles
  const SymMergeBlock* blocks;
  int32_t n_merge;               // merge CTAs
};

enum SymForm : int {
  kSymForce = 0,
  kSymForcePot = 1,
  kSymJerk = 2,
  kSymJerkPot = 3,
  kSymAdjoint = 4,
  kSymBatched = 5,
  kSymBatchedPot = 6,
};

// A form's kernels: sums per particle, planes of a segment, most particles per
// thread and records per stage, shared
// memory of a shape, resident CTAs per SM, and the launch of one band (pair
// kernel and merge).
struct SymOps {
  int sums;
  int planes;
  int max_k;
  int max_stage;
  size_t (*smem)(int threads, int k, int chunk, int stages);
  cudaError_t (*occupancy)(int k, bool guard, int threads, size_t smem, int* ctas);
  cudaError_t (*launch)(const SymArgs& a, const SymMerge& m, int k, bool guard, int threads, size_t smem,
                        cudaStream_t s);
};

SymOps sym_force_ops(bool pot);    // cn_sym.cu
SymOps sym_jerk_ops(bool pot);     // cn_sym_jerk.cu
SymOps sym_adjoint_ops();          // cn_sym_adjoint.cu
SymOps sym_batched_ops(bool pot);  // cn_sym_batched.cu
inline SymOps sym_ops(SymForm form) {
  switch (form) {
    case kSymForce: return sym_force_ops(false);
    case kSymForcePot: return sym_force_ops(true);
    case kSymJerk: return sym_jerk_ops(false);
    case kSymJerkPot: return sym_jerk_ops(true);
    case kSymBatched: return sym_batched_ops(false);
    case kSymBatchedPot: return sym_batched_ops(true);
    default: return sym_adjoint_ops();
  }
}

}  // namespace cn
