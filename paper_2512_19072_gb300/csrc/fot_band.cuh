// Banded axis pass: arguments and entry points shared by the plan and window kernels
// (fot_band.cu, fot_window.cuh), the single-problem half-step and the batched solver
// (fot_batch.cu).
#pragma once

#include "fot_common.cuh"

namespace fot {

// Arithmetic of the window sums: FP32 operands (three TF32 products per term), split BF16
// (three products), single BF16 for the rows (two).
enum WindowForm : int { kFormFp32 = 0, kFormSplit = 1, kFormSingle = 2 };

// One problem's pass over rows of x: y[o][r] = log2 sum_m 2^(x[r][m] x_scale - (o + shift - m)^2 c).
// plan holds, per (tile of tile_w outputs, row) at t * plan_stride + r, three arrays of
// n_tiles * plan_stride words each: the offset alpha (float), the window start | length << 16
// (positions) and mh, the position the offset was taken at.
struct BandArgs {
  const float* x;      // [n_rows][len] input
  float* plan;
  const float* lmarg;  // potential-update mode: natural log marginal, layout of y
  float* y;            // [n_out][n_rows] output (transposed)
  float* logsum;       // potential-update mode: optional natural-log LSE, layout of y
  int* err;
  unsigned long long* terms;   // [kTermSlots][4] counters of (row, output, m) triples: GEMM on
                               // FP32 operands, exact windows, GEMM on BF16 operands
  int4* items;         // the window kernel's items in its order: row group, four tiles, span of the
                       // rows they read (written by the plan)
  int* order;          // [2] items placed at the front and at the back so far
  const uint4* tilt;           // BF16 forms: operand fragments of the tilt matrix for (c, tile_w)
  // moment passes only (fot_moments.cu): term weights, a second output, the logarithm of the
  // divisor, and the coordinate of index m, coord0 + m coord_step
  const float* w;      // [n_rows][len]
  float* y2;           // layout of y
  const float* off;    // natural log, layout of y
  float coord0, coord_step;
  float x_scale, c, eps, shift;
  int n_rows, len, n_out;
  int tile_w;          // outputs per plan tile and window unit: 16 or 32
  int group;           // rows per window unit: 8, or 2 where every unit takes exact window sums
  int n_chunks, n_tiles, plan_stride;
  int parts;                   // one-kernel products: CTAs that share a row group's tiles
  int plan_base, item_base;    // first plan CTA and first window item of this problem
  int items_row, n_items;      // window items along the outputs of a row group, and in all
  int wide_span;               // items whose windows span more go first
  int vec;                     // bit 0: rows of x are 16-byte aligned; bit 1: pairs of outputs are
                               // 8-byte aligned
  float step[33];              // 2^(32 kap c), kap = i - 16: the accumulators' scale per window
                               // step, rounded once from 64 bits
  float step_err[33];          // log2 of what that rounding leaves out, per position of the walk
};

constexpr int kMaxBatch = 64;
constexpr int kTermSlots = 64;   // counter copies (CTA index mod kTermSlots): one address would
                                 // serialise thousands of atomics per pass

// A launch covers every problem of the table; the kernels map a plan CTA or a window item to its
// problem by the *_base prefix sums.  Passed by value (__grid_constant__).
template <int MAXP>
struct BandTable {
  int n;                                 // problems
  int plans, items;                      // plan CTAs and window items in all
  int plan_items;                        // items of the widest row group
  int plan_tpr_log2;                     // plan threads per row
  int plan_row_floats;                   // shared memory of one plan row
  int pitch_max;                         // floats per staged row of the window kernel
  int spin_limit;                        // polls of a bounded wait
  BandArgs p[MAXP];
};
static_assert(sizeof(BandTable<kMaxBatch>) <= 32764, "kernel parameter limit");

// problem owning plan CTA (WHICH 0) or window item (WHICH 1) gi: binary search over the prefix sums
template <int MAXP, int WHICH>
__device__ __forceinline__ int find_prob(const BandTable<MAXP>& t, int gi) {
  if (MAXP == 1) return 0;
  int lo = 0, hi = t.n - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if ((WHICH == 0 ? t.p[mid].plan_base : t.p[mid].item_base) <= gi)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

// Tile width of a pass with kernel constant c: outputs per window unit, 32 or 16; 0 where
// eps is too small for the tilted product (the pass then runs exact window sums in units of 2 rows x 16
// outputs).
int tile_width_for(float c);

// tiles of n outputs that a plan must have room for: 16-wide ones
inline size_t plan_tiles(int n) { return ((size_t)n + 15) / 16; }

// the fields of a pass that follow from eps: kernel constant, tile width, step scales
void band_set_eps(BandArgs& a, double eps);

// fill one pass's arguments; the tilt fragments and the outputs are set by the caller
BandArgs band_args(fot_ctx* c, const float* x, int n_rows, int len, double eps, float x_scale);

// one pass of every problem of the table: the window plan, then the window sums (MODE 0:
// log-sum output; MODE 1: potential update).  Returns the kernels launched: two, or one for small
// problems.
template <int MODE, int MAXP>
int band_pass(cudaStream_t s, BandTable<MAXP>& t, int form);

// the window plan alone, for a table whose window kernel the caller launches (fot_moments.cu)
template <int MAXP>
void plan_pass(cudaStream_t s, BandTable<MAXP>& t);

// work space of the second problem of a two-problem pass
struct PairSpace {
  float* plan;
  int4* items;
  int* order;          // zeroed before the first use
  float* R;
};
// logsums of two inputs of a context's half-step in two-problem passes (outA, outB: potentials)
void half_step_band_pair(fot_ctx* c, const float* inA, const float* inB, const float* lmarg, double eps, float* outA,
                         float* outB, float* logsumA, float* logsumB, const PairSpace& second);

// words of the window plan and items of the window kernel for a context's passes
inline size_t band_plan_words(int rows, int cols) {
  const size_t pr = (size_t)(rows + 7) / 8 * 8, pc = (size_t)(cols + 7) / 8 * 8;
  const size_t a = pr * plan_tiles(cols), b = pc * plan_tiles(rows);
  return 3 * (a > b ? a : b);
}
inline size_t band_items(int rows, int cols) {
  const size_t a = (size_t)(rows + 7) / 8 * ((plan_tiles(cols) + 3) / 4), b = (size_t)(cols + 7) / 8 * ((plan_tiles(rows) + 3) / 4);
  return a > b ? a : b;
}

int form_of(const fot_ctx* c);

constexpr int kTiltTables = 256;   // tilt tables a context holds

// Tilt tables of context c for the BF16 forms: one table per distinct kernel constant of the
// coming passes (host array of per-iteration eps), written by one launch.  tilt_for returns the
// table of eps (writing it first when the context does not hold it).
void tilt_prepare(fot_ctx* c, const double* eps, int n, int64_t* launches);
const uint4* tilt_for(fot_ctx* c, double eps, int tile_w, int64_t* launches);
// forget what the device holds (the next use writes the tables again)
void tilt_reset(fot_ctx* c);
// At the start of an entry point whose passes run on the caller's stream: once a caller has captured such
// a call, the table's writes are the caller's graphs' (now, or whenever one is replayed), so what the
// host remembers of earlier calls no longer holds.
void tilt_begin(fot_ctx* c);

}  // namespace fot
