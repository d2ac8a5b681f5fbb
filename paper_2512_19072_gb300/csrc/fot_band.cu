// Banded axis passes: the same contraction as the exact pass,
//     y[o][r] = log2 sum_m 2^( x[r][m]*scale - (o - m)^2 c ),   c = log2(e) / (2 eps),
// but each output only visits the terms that can matter, and where eps allows the inner sum is
// a matrix product instead of one exponential per term.  A pass is two kernels, the window plan
// (fot_plan.cuh) and the window sums (fot_window.cuh, which describes the arithmetic), or one that does
// both (fot_small.cuh).  This file has the plan's kernel and chooses between them.
#include "fot_small.cuh"

#include <math.h>

#include <algorithm>

namespace fot {

namespace {

template <int MAXP>
__global__ void __launch_bounds__(kPlanThreads) band_plan_kernel(const __grid_constant__ BandTable<MAXP> tab) {
  extern __shared__ __align__(16) float s_plan[];
  const int tid = threadIdx.x;
  const BandArgs& a = tab.p[find_prob<MAXP, 0>(tab, (int)blockIdx.x)];
  const int rg = (int)blockIdx.x - a.plan_base;           // row group of the problem
  const int T = a.n_tiles;
  // threads per row: a power of two (at least kPlanQ lanes of one warp serve a (row, tile))
  const int tpr = 1 << tab.plan_tpr_log2, rr = tid >> tab.plan_tpr_log2, ti = tid & (tpr - 1);
  const int row = kPlanRows * rg + rr;
  const bool live = row < a.n_rows;
  float* const mine = s_plan + (size_t)rr * tab.plan_row_floats;
  // per item (four tiles): the span of its windows
  int* const s_lo = reinterpret_cast<int*>(s_plan + (size_t)kPlanRows * tab.plan_row_floats);
  int* const s_hi = s_lo + tab.plan_items;
  for (int i = tid; i < a.items_row; i += blockDim.x) {
    s_lo[i] = 0x7fffffff;
    s_hi[i] = 0;
  }
  grid_wait();
  grid_launch_next();

  const float* const xr = a.x + (size_t)row * a.len;
  plan_stage(a, mine, ti, tpr, [&](int m0, float (&v)[8]) {
    if (live && (a.vec & 1) && m0 + 8 <= a.len) {
      const float4 p = __ldg(reinterpret_cast<const float4*>(xr + m0)), q = __ldg(reinterpret_cast<const float4*>(xr + m0) + 1);
      v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w;
      v[4] = q.x; v[5] = q.y; v[6] = q.z; v[7] = q.w;
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = live && m0 + u < a.len ? __ldg(xr + m0 + u) : -INFINITY;
    }
  });
  __syncthreads();

  // kPlanQ lanes per (row, tile)
  const size_t np = (size_t)a.plan_stride * T;
  int* const plan_i = reinterpret_cast<int*>(a.plan);
  const int q = ti & (kPlanQ - 1);
  // (lanes past the tiles or rows compute on a valid place and write nothing: the shuffles want
  // whole warps)
  for (int t0 = 0; t0 < T; t0 += tpr / kPlanQ) {
    const int t = min(t0 + ti / kPlanQ, T - 1);
    const PlanEntry e = plan_tile(a, mine, t, q);
    if (live && t0 + ti / kPlanQ < T && q == 0) {
      const size_t pi = (size_t)t * a.plan_stride + row;
      a.plan[pi] = e.alpha;
      plan_i[np + pi] = e.lo | ((e.hi - e.lo) << 16);
      plan_i[2 * np + pi] = e.mh;
      if (e.hi > e.lo) {
        atomicMin(&s_lo[t / kWinWarps], e.lo);
        atomicMax(&s_hi[t / kWinWarps], e.hi);
      }
    }
  }
  if (a.group != kPlanRows) return;                       // exact windows only: no item list
  __syncthreads();
  // the items of this row group: those with a wide span to the front of the list
  for (int i = tid; i < a.items_row; i += blockDim.x) {
    const int lo = s_hi[i] > 0 ? s_lo[i] : 0, hi = s_hi[i];
    const bool wide = hi - lo > a.wide_span;
    const int at = wide ? atomicAdd(&a.order[0], 1) : a.n_items - 1 - atomicAdd(&a.order[1], 1);
    a.items[at] = make_int4(rg, i, lo, hi);
  }
}

// BF16 operands are for rows that are 16-byte aligned (every side a multiple of 4); the others keep FP32
// operands.  Their errors, not their speed, set this line: 291 x 330 at eps 35 with FOT_BF16, rms 2.2e-6
// of the potential with BF16 rows and 2.5e-8 with FP32 ones.
bool aligned_rows(const BandArgs& a) { return (a.len & 3) == 0 && (reinterpret_cast<uintptr_t>(a.x) & 15u) == 0; }

// finish a table: chunk and tile counts, prefix sums
template <int MAXP>
void finish(BandTable<MAXP>& t, int* max_chunks) {
  int plans = 0, items = 0, pitch = 16, chunks = 1, items_row = 1;
  for (int q = 0; q < t.n; ++q) {
    BandArgs& a = t.p[q];
    a.n_chunks = (a.len + kCW - 1) / kCW;
    a.n_tiles = (a.n_out + a.tile_w - 1) / a.tile_w;
    a.plan_stride = (a.n_rows + 7) / 8 * 8;
    a.items_row = (a.n_tiles + kWinWarps - 1) / kWinWarps;
    a.vec = 0;
    if (aligned_rows(a)) a.vec |= 1;
    const uintptr_t outs = reinterpret_cast<uintptr_t>(a.y) | reinterpret_cast<uintptr_t>(a.lmarg) |
                           reinterpret_cast<uintptr_t>(a.logsum);
    if ((a.n_rows & 1) == 0 && (outs & 7u) == 0) a.vec |= 2;
    a.plan_base = plans;
    a.item_base = items;
    plans += (a.n_rows + kPlanRows - 1) / kPlanRows;
    a.n_items = (a.n_rows + a.group - 1) / a.group * a.items_row;
    items += a.n_items;
    items_row = std::max(items_row, a.items_row);
    chunks = std::max(chunks, a.n_chunks);
    pitch = std::max(pitch, stage_pitch(a.len));
  }
  t.plans = plans;
  t.items = items;
  t.plan_items = items_row;
  t.pitch_max = std::min(pitch, kPitchCap);
  t.plan_row_floats = plan_row_floats(chunks);
  *max_chunks = chunks;
}

}  // namespace

// Tile width for a problem with kernel constant c.  A row's operands stay in range while
// tile_w (D + mh - lo) c <= kRangeMax = 100, D the farthest window position from mh.  For a smooth
// potential the window W is about the tile plus the distance sqrt(kCut / c) on both sides at which
// the Gaussian has fallen by 2^-kCut, with mh in its middle: tile_w W c.  Real windows are longer
// where the transport map jumps, so a width is taken while that estimate leaves room (the wider
// tile shares each exponential, and each unit's set-up, between more outputs; units out of range
// are summed in segments).  32 ends at eps 101 (us per pass, 32-wide against 16-wide: split BF16 at 1024^2,
// eps 130 24.9 / 21.7, eps 80 31.2 / 22.8; FP32, eps 130 24.1 / 25.1, eps 80 26.1 / 25.1; 256^2, split BF16, eps 130
// 4.75 / 4.21, eps 80 5.14 / 4.20: 32 is right for FP32 operands and costs the others up to 15 % between eps
// 101 and 168).  16 ends at eps 12 (16-wide against exact, FP32: 1024^2 eps 11 37.7 / 32.7, eps 16 31.9 / 32.9, 2048^2 eps
// 11 111 / 105, eps 13 100 / 105; below 1024^2 exact sums stay the faster ones to eps 20 and beyond: 512^2 eps 16
// 14.3 / 10.7, 256^2 12.0 / 6.1).
int tile_width_for(float c) {
  const float reach = 2.f * sqrtf(kCut / c);
  auto need = [&](float w) { return w * (w + reach) * c; };
  if (need(32.f) <= 42.f) return 32;
  if (need(16.f) <= 64.f) return 16;
  return 0;
}

void band_set_eps(BandArgs& a, double eps) {
  a.c = (float)(1.4426950408889634 / (2.0 * eps));
  a.eps = (float)eps;
  const int tw = tile_width_for(a.c);
  a.tile_w = tw == 0 ? 16 : tw;
  a.group = tw == 0 ? 2 : 8;
  // (1.8 and 3.6 for 2.6: within 1 % at 1024^2 and 2048^2, eps 209 and 839)
  a.wide_span = kWinWarps * a.tile_w + (int)(2.6f * sqrtf(kCut / a.c));
  if (tw == 0) return;
  for (int i = 0; i <= 32; ++i) {
    const double e = 32.0 * (i - 16) * (double)a.c;
    a.step[i] = (float)exp2(e);
    a.step_err[i] = (float)((e - log2((double)a.step[i])) / 16.0);
  }
}

BandArgs band_args(fot_ctx* c, const float* x, int n_rows, int len, double eps, float x_scale) {
  BandArgs a{};
  a.x = x;
  a.plan = c->plan;
  a.err = c->err;
  a.terms = c->terms;
  a.items = c->items;
  a.order = c->order;
  a.x_scale = x_scale;
  a.n_rows = n_rows;
  a.len = len;
  a.n_out = len;
  band_set_eps(a, eps);
  return a;
}

template <int MAXP>
void plan_pass(cudaStream_t s, BandTable<MAXP>& t) {
  int chunks = 1;
  finish(t, &chunks);
  // plan: threads per row to the next power of two of the widest row's (tile, lane) pairs
  int tiles = 1;
  for (int q = 0; q < t.n; ++q) tiles = std::max(tiles, t.p[q].n_tiles);
  int tl = 2;                                             // (four threads stage a chunk together)
  while ((1 << tl) < tiles * kPlanQ && (kPlanRows << tl) < kPlanThreads) ++tl;
  t.plan_tpr_log2 = tl;
  const size_t plan_smem = (size_t)kPlanRows * t.plan_row_floats * sizeof(float) + 2 * t.plan_items * sizeof(int);
  ktimer_begin(s, kKPlan);
  launch_dependent(band_plan_kernel<MAXP>, dim3(t.plans), kPlanRows << tl, plan_smem, s, t);
  ktimer_end(s);
}

template void plan_pass<1>(cudaStream_t, BandTable<1>&);
template void plan_pass<2>(cudaStream_t, BandTable<2>&);
template void plan_pass<kMaxBatch>(cudaStream_t, BandTable<kMaxBatch>&);

namespace {

// Longest rows (inputs and outputs) of a one-kernel product, and its tiles per CTA.  us per pass, two kernels
// against one: 64^2 FP32 eps 60 4.9 / 3.2, 100^2 mixed eps 20 5.5 / 4.0, 256^2 mixed eps 64 6.1 / 4.2, eps
// 13 13.8 / 11.6, 257^2 FP32 eps 130 9.5 / 8.5, 512^2 mixed eps 64 9.9 / 7.8, eps 13 17.5 / 15.1; at
// 1024^2, where staging every row for each part costs more than the launch, 25.5 / 31.2 (eps 52) and
// 21.4 / 21.3 (eps 209).  Between them one kernel is still ahead at 640, the longest rows that could stay
// within 48 KB (576^2 mixed eps 60 14.7 / 12.0, 640^2 mixed eps 130 14.0 / 10.7).  16 tiles per CTA took 5.2
// us at 256^2 and 8.3 at 512^2 (eps 130; 7.1 with 8), 4 tiles 4.0 and 7.5.
constexpr int kSmallLen = 512;
constexpr int kSmallTiles = 8;

// Make a table that of a one-kernel pass: CTAs of `group` rows, a warp per tile (exact sums: up to 16 warps,
// the row's tiles among them).
template <int MAXP>
void small_table(BandTable<MAXP>& t) {
  int chunks = 1;
  finish(t, &chunks);
  const int group = t.p[0].group;
  int ctas = 0, tiles = 1, pitch = 16;
  for (int q = 0; q < t.n; ++q) {
    BandArgs& a = t.p[q];
    int share = a.n_tiles;
    a.parts = 1;
    if (group == 8) {
      a.parts = (a.n_tiles + kSmallTiles - 1) / kSmallTiles;
      share = (a.n_tiles + a.parts - 1) / a.parts;
      a.parts = (a.n_tiles + share - 1) / share;          // (no empty part)
    }
    a.plan_base = ctas;
    ctas += (a.n_rows + group - 1) / group * a.parts;
    tiles = std::max(tiles, share);
    pitch = std::max(pitch, stage_pitch(t.p[q].len));
  }
  int warps = 4;
  while (warps < tiles && warps < kSmallWarps) warps *= 2;
  t.plans = ctas;
  t.plan_items = tiles;
  t.pitch_max = pitch;
  t.plan_tpr_log2 = 0;
  while ((group << t.plan_tpr_log2) < 32 * warps) ++t.plan_tpr_log2;
}

template <int MODE, int MAXP>
void exact_pass(cudaStream_t s, BandTable<MAXP>& t) {
  small_table(t);
  ktimer_begin(s, kKPlan);
  small_exact_launch<MODE, MAXP>(s, t);
  ktimer_end(s);
}

}  // namespace

template <int MODE, int MAXP>
int band_pass(cudaStream_t s, BandTable<MAXP>& t, int form) {
  bool exact = true, small = MAXP <= 2;
  for (int q = 0; q < t.n; ++q) {
    exact = exact && t.p[q].group == 2;
    small = small && t.p[q].group == 8 && std::max(t.p[q].len, t.p[q].n_out) <= kSmallLen;
  }
  // Exact sums: one kernel at every size (us per pass against plan and sums apart: 64^2 3.4 / 5.7, 256^2
  // 6.4 / 11.1, 512^2 13.7 / 21.8, 1024^2 37 / 56, 2048^2 132 / 204, all at eps 1).  A batch's pass is
  // two launches whatever its eps: half of the problems each.
  if (exact) {
    if (MAXP <= 2 || t.n == 1) {
      exact_pass<MODE>(s, t);
      return 1;
    }
    size_t all = 0, head = 0;
    for (int q = 0; q < t.n; ++q) all += (size_t)t.p[q].n_rows * t.p[q].n_out;
    int cut = 0;
    while (cut < t.n - 1 && (cut == 0 || 2 * head < all)) head += (size_t)t.p[cut].n_rows * t.p[cut].n_out, ++cut;
    BandTable<MAXP> rest = t;
    rest.n = t.n - cut;
    std::copy(t.p + cut, t.p + t.n, rest.p);
    t.n = cut;
    exact_pass<MODE>(s, t);
    exact_pass<MODE>(s, rest);
    t.n += rest.n;
    return 2;
  }
  if (form != kFormFp32) {
    const int aligned = (int)std::count_if(t.p, t.p + t.n, aligned_rows);
    if (aligned == 0) form = kFormFp32;
    if (aligned > 0 && aligned < t.n) {                   // (a batch: each kind by itself)
      BandTable<MAXP> rest = t;
      t.n = (int)(std::copy_if(rest.p, rest.p + rest.n, t.p, aligned_rows) - t.p);
      int k = band_pass<MODE>(s, t, form);
      t.n = (int)(std::remove_copy_if(rest.p, rest.p + rest.n, t.p, aligned_rows) - t.p);
      k += band_pass<MODE>(s, t, kFormFp32);
      t = rest;
      return k;
    }
  }
  if constexpr (MAXP <= 2) {
    if (small) {
      small_table(t);
      ktimer_begin(s, kKPlan);
      if (form == kFormFp32)
        small_launch<MODE, kFormFp32, MAXP>(s, t);
      else if (form == kFormSplit)
        small_launch<MODE, kFormSplit, MAXP>(s, t);
      else
        small_launch<MODE, kFormSingle, MAXP>(s, t);
      ktimer_end(s);
      return 1;
    }
  }
  plan_pass(s, t);
  ktimer_begin(s, form == kFormFp32 ? kKBand : kKTensor);
  if (form == kFormFp32)
    window_launch<MODE, kFormFp32, MAXP>(s, t);
  else if (form == kFormSplit)
    window_launch<MODE, kFormSplit, MAXP>(s, t);
  else
    window_launch<MODE, kFormSingle, MAXP>(s, t);
  ktimer_end(s);
  return 2;
}

template int band_pass<0, 1>(cudaStream_t, BandTable<1>&, int);
template int band_pass<1, 1>(cudaStream_t, BandTable<1>&, int);
template int band_pass<0, 2>(cudaStream_t, BandTable<2>&, int);
template int band_pass<1, 2>(cudaStream_t, BandTable<2>&, int);
template int band_pass<0, kMaxBatch>(cudaStream_t, BandTable<kMaxBatch>&, int);
template int band_pass<1, kMaxBatch>(cudaStream_t, BandTable<kMaxBatch>&, int);

// Kernel attributes for rows of up to `longest`: more than the default 48 KB of dynamic shared memory, which
// the plan kernel (eight rows) takes from rows of 1152 on, the exact one (two rows) from about 2350.
// The one-kernel products stay below it.
cudaError_t plan_configure(int longest) {
  constexpr size_t kDefault = 48 * 1024;
  constexpr int kMaxLen = 4096;
  const int chunks = (longest + kCW - 1) / kCW;
  cudaError_t e = cudaSuccess;
  if (kPlanRows * plan_row_floats(chunks) * sizeof(float) + 2 * 256 * sizeof(int) > kDefault) {
    const int lim = (int)(kPlanRows * plan_row_floats(kMaxLen / kCW) * sizeof(float)) + 2 * 256 * (int)sizeof(int);
    e = cudaFuncSetAttribute(band_plan_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(band_plan_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    if (e == cudaSuccess) e = cudaFuncSetAttribute(band_plan_kernel<kMaxBatch>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  }
  if (e == cudaSuccess && small_smem(2, stage_pitch(longest), plan_row_floats(chunks), (longest + 15) / 16) > kDefault)
    e = small_exact_configure((int)small_smem(2, stage_pitch(kMaxLen), plan_row_floats(kMaxLen / kCW), (kMaxLen + 15) / 16));
  return e;
}
static_assert((16 + 8 * ((kSmallLen + 15) / 32 * 32 + 16 + 2 * (kSmallLen / 32 + 3) + kSmallLen / 32 * 40) +
               3 * 8 * kSmallTiles) * sizeof(float) <= 48 * 1024, "one-kernel products");

int default_wait_limit() { return kSpinDefault; }

int form_of(const fot_ctx* c) {
  return c->precision == FOT_MIXED ? kFormSplit : c->precision == FOT_BF16 ? kFormSingle : kFormFp32;
}

// ---- tilt tables of the BF16 forms ---------------------------------------------------------

namespace {

struct TiltArgs {
  uint4* out;
  int tw[kTiltTables / 4];                    // four 8-bit tile widths per word
  float c[kTiltTables];
};

// One table: fragments of T[kap][p] = 2^(2 kap p c), kap = row - tw/2, split into BF16 hi and lo
// parts in the register order of mma.m16n8k16's A operand, with the columns permuted as the
// window kernel produces them (lane q of a quad owns positions 4q .. 4q + 3).
__global__ void tilt_table_kernel(const __grid_constant__ TiltArgs t) {
  const int i = blockIdx.x, mt = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tw = (t.tw[i >> 2] >> (8 * (i & 3))) & 255;
  if (16 * mt >= tw) return;
  uint32_t hi[4], lo[4];
  tilt_fragments_bf16(t.c[i], 16 * mt - tw / 2, lane, hi, lo);
  uint4* o = t.out + (size_t)i * kTiltWords + (size_t)mt * 64 + lane;
  o[0] = make_uint4(hi[0], hi[1], hi[2], hi[3]);
  o[32] = make_uint4(lo[0], lo[1], lo[2], lo[3]);
}

}  // namespace

size_t tilt_bytes() { return (size_t)kTiltTables * kTiltWords * sizeof(uint4); }

void tilt_reset(fot_ctx* c) { c->tilt_eps.clear(); }

void tilt_begin(fot_ctx* c) {
  if (!c->tilt) return;
  cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(c->stream, &st) != cudaSuccess) cudaGetLastError();
  c->captured = c->captured || st != cudaStreamCaptureStatusNone;
  if (c->captured) tilt_reset(c);
}

void tilt_prepare(fot_ctx* c, const double* eps, int n, int64_t* launches) {
  if (!c->tilt) return;
  TiltArgs t{};
  t.out = c->tilt;
  c->tilt_eps.clear();
  for (int i = 0; i < n && (int)c->tilt_eps.size() < kTiltTables; ++i) {
    if (!c->tilt_eps.empty() && c->tilt_eps.back() == eps[i]) continue;
    const float cc = (float)(1.4426950408889634 / (2.0 * eps[i]));
    const int tw = tile_width_for(cc);
    if (tw == 0) continue;                    // exact windows: no table
    const int k = (int)c->tilt_eps.size();
    t.c[k] = cc;
    t.tw[k >> 2] |= tw << (8 * (k & 3));
    c->tilt_eps.push_back(eps[i]);
  }
  if (c->tilt_eps.empty()) return;
  ktimer_begin(c->stream, kKPlan);            // timed with the plans (set-up of the passes)
  tilt_table_kernel<<<(unsigned)c->tilt_eps.size(), 64, 0, c->stream>>>(t);
  ktimer_end(c->stream);
  ++*launches;
}

const uint4* tilt_for(fot_ctx* c, double eps, int tile_w, int64_t* launches) {
  if (!c->tilt || tile_w == 0) return nullptr;
  for (size_t i = 0; i < c->tilt_eps.size(); ++i)
    if (c->tilt_eps[i] == eps) return c->tilt + i * kTiltWords;
  tilt_prepare(c, &eps, 1, launches);
  return c->tilt;
}

// One half-step with banded passes: pot_out = eps (lmarg - log(Lambda exp(pot_in/eps) Lambda)).
void half_step_band(fot_ctx* c, const float* pot_in, const float* lmarg, double eps, float* pot_out,
                    float* logsum) {
  const int form = form_of(c);
  BandTable<1> t{};
  t.n = 1;
  t.spin_limit = c->spin;
  int64_t k = 0;
  // pass over the contiguous axis: rows of pot_in, outputs along cols, written [k][L]
  t.p[0] = band_args(c, pot_in, c->rows, c->cols, eps, (float)(1.4426950408889634 / eps));
  t.p[0].y = c->R;
  const uint4* tilt = tilt_for(c, eps, t.p[0].group == 8 ? t.p[0].tile_w : 0, &k);
  t.p[0].tilt = tilt;
  k += band_pass<0>(c->stream, t, form);
  // pass over the row axis (input R[k][L], log2 units) with the fused potential update
  t.p[0] = band_args(c, c->R, c->cols, c->rows, eps, 1.f);
  t.p[0].tilt = tilt;
  t.p[0].y = pot_out;
  t.p[0].lmarg = lmarg;
  t.p[0].logsum = logsum;
  k += band_pass<1>(c->stream, t, form);
  c->launches += k;
}

// Two half-steps of one context in the same launches (2 per pass).
void half_step_band_pair(fot_ctx* c, const float* inA, const float* inB, const float* lmarg, double eps, float* outA,
                         float* outB, float* logsumA, float* logsumB, const PairSpace& second) {
  const int form = form_of(c);
  BandTable<2> t{};
  t.n = 2;
  t.spin_limit = c->spin;
  int64_t k = 0;
  const uint4* tilt = nullptr;
  for (int pass = 0; pass < 2; ++pass) {
    for (int q = 0; q < 2; ++q) {
      BandArgs& a = t.p[q];
      float* R = q == 0 ? c->R : second.R;
      a = pass == 0 ? band_args(c, q == 0 ? inA : inB, c->rows, c->cols, eps, (float)(1.4426950408889634 / eps))
                    : band_args(c, R, c->cols, c->rows, eps, 1.f);
      if (pass == 0 && q == 0) tilt = tilt_for(c, eps, a.group == 8 ? a.tile_w : 0, &k);
      a.tilt = tilt;
      if (q == 1) {
        a.plan = second.plan;
        a.items = second.items;
        a.order = second.order;
      }
      a.y = pass == 0 ? R : q == 0 ? outA : outB;
      if (pass == 1) {
        a.lmarg = lmarg;
        a.logsum = q == 0 ? logsumA : logsumB;
      }
    }
    k += pass == 0 ? band_pass<0>(c->stream, t, form) : band_pass<1>(c->stream, t, form);
  }
  c->launches += k;
}

}  // namespace fot
