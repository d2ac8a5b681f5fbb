// Banded axis passes: the same contraction as the exact pass,
//     y[o][r] = log2 sum_m 2^( x[r][m]*scale - (o - m)^2 c ),   c = log2(e) / (2 eps),
// but each output only visits the terms that can matter, and where eps allows the inner sum is
// a matrix product instead of one exponential per term.  A pass is two kernels: the window plan
// (this file) and the window sums (fot_window.cuh, which describes the arithmetic).
//
// The plan leaves, per (row, tile of tile_w outputs), an offset alpha, the position mh it was
// taken at and a window [lo, lo + wl):
//
// 1. alpha = e(mh, kc), e(m, o) = x[m] scale - (o - m)^2 c, at the tile centre kc: the maximum
//    over the 32-wide chunk whose own maximum gives the best term there.  It may lie below the
//    exact maximum, which only raises the operands 2^(e - alpha) of the window sums (a sum that
//    leaves the range of FP32 is done again there).
// 2. A provable window: every o in the tile has max_m e(m, o) >= LB = min over the tile's two
//    ends of e(mh, o) (e(mh, .) is concave).  A block of 8 positions whose bound (its maximum
//    at its nearest distance to the tile) lies below LB - kCut holds only terms below 2^-kCut
//    of every output of the tile; the window is the hull of the remaining blocks (found per
//    32-wide chunk first, then narrowed from both ends).
// Arg-maxima carry the index in the low mantissa bits of the value they compare (5 bits for a
// position, 7 for a chunk): one maximum instead of a compare and two selects; a chunk's maximum
// is rounded by 2^-18 of itself that way, far inside the margin of kCut.
//
// What bounds it: latency and issue slots (4 MB of input at 1024^2, in L2).  Two lanes serve a
// (row, tile): each takes every other pair of chunks (packed FP32 pairs), half of the scanned
// chunk and one end of the window.  Chunks are padded to 36 words: lanes on different chunks read
// different banks, lanes on the same chunk broadcast.
#include "fot_window.cuh"

#include <math.h>

#include <algorithm>

namespace fot {

namespace {

constexpr int kPlanRows = 8;                  // rows of a CTA: one row group of the window kernel
constexpr int kPlanThreads = 512;
constexpr int kPlanQ = 2;                     // lanes per (row, tile)
constexpr int kZS = kCW + 4;                  // words of a staged chunk

// shared memory of one row (floats): chunk maxima and minus their positions (rounded up to four
// chunks each), block maxima [n_chunks * 4], z [n_chunks * kZS]
__host__ __device__ inline int plan_row_floats(int n_chunks) { return 2 * ((n_chunks + 3) & ~3) + n_chunks * (4 + kZS); }

// v with its low mantissa bits replaced by an index (-inf becomes a NaN, which fmaxf drops)
template <int BITS>
__device__ __forceinline__ float tagged(float v, int index) {
  return __uint_as_float((__float_as_uint(v) & ~((1u << BITS) - 1u)) | (uint32_t)index);
}
template <int BITS>
__device__ __forceinline__ int tag_of(float v) { return (int)(__float_as_uint(v) & ((1u << BITS) - 1u)); }

template <int MAXP>
__global__ void __launch_bounds__(kPlanThreads) band_plan_kernel(const __grid_constant__ BandTable<MAXP> tab) {
  extern __shared__ __align__(16) float s_plan[];
  const int tid = threadIdx.x;
  const BandArgs& a = tab.p[find_prob<MAXP, 0>(tab, (int)blockIdx.x)];
  const int rg = (int)blockIdx.x - a.plan_base;           // row group of the problem
  const int T = a.n_tiles, len = a.len, nch = a.n_chunks, tw = a.tile_w;
  const float c = a.c, sc = a.x_scale;
  // threads per row: a power of two (at least kPlanQ lanes of one warp serve a (row, tile))
  const int tpr = 1 << tab.plan_tpr_log2, rr = tid >> tab.plan_tpr_log2, ti = tid & (tpr - 1);
  const int row = kPlanRows * rg + rr;
  const bool live = row < a.n_rows;
  float* const cm = s_plan + (size_t)rr * tab.plan_row_floats;
  const int nchp = (nch + 3) & ~3;
  float* const np_ = cm + nchp;                           // minus the maxima's positions
  float* const bm = np_ + nchp;
  float* const z = bm + 4 * nch;
  // per item (four tiles): the span of its windows
  int* const s_lo = reinterpret_cast<int*>(s_plan + (size_t)kPlanRows * tab.plan_row_floats);
  int* const s_hi = s_lo + tab.plan_items;
  for (int i = tid; i < a.items_row; i += blockDim.x) {
    s_lo[i] = 0x7fffffff;
    s_hi[i] = 0;
  }
  grid_wait();
  grid_launch_next();

  // ---- stage: blocks of 8 positions, a thread each; four neighbouring threads share a chunk
  {
    const float* xr = a.x + (size_t)row * len;
    const bool vec = (a.vec & 1) != 0;
    const f32x2 sc2 = pack2(sc, sc);
    for (int b = ti; b < nchp * 4; b += tpr) {
      const int m0 = b * 8, j = b >> 2, u0 = (b & 3) * 8;
      float v[8];
      if (live && vec && m0 + 8 <= len) {
        const float4 p = __ldg(reinterpret_cast<const float4*>(xr + m0)), q = __ldg(reinterpret_cast<const float4*>(xr + m0) + 1);
        v[0] = p.x; v[1] = p.y; v[2] = p.z; v[3] = p.w;
        v[4] = q.x; v[5] = q.y; v[6] = q.z; v[7] = q.w;
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = live && m0 + u < len ? __ldg(xr + m0 + u) : -INFINITY;
      }
      float best = -INFINITY, top = -INFINITY;            // block maximum; the same with its position
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        unpack2(mul2(pack2(v[u], v[u + 1]), sc2), v[u], v[u + 1]);
        best = fmaxf(best, fmaxf(v[u], v[u + 1]));
        top = fmaxf(top, fmaxf(tagged<5>(v[u], u0 + u), tagged<5>(v[u + 1], u0 + u + 1)));
      }
      if (j < nch) {
        float4* const zb = reinterpret_cast<float4*>(z + j * kZS + u0);
        zb[0] = make_float4(v[0], v[1], v[2], v[3]);
        zb[1] = make_float4(v[4], v[5], v[6], v[7]);
        bm[b] = best;
      }
      // (the four threads of a chunk are neighbours and take this iteration together)
      const unsigned quad = 0xfu << (tid & 28);
      top = fmaxf(top, __shfl_xor_sync(quad, top, 1));
      top = fmaxf(top, __shfl_xor_sync(quad, top, 2));
      best = fmaxf(best, __shfl_xor_sync(quad, best, 1));
      best = fmaxf(best, __shfl_xor_sync(quad, best, 2));
      if (u0 == 0) {
        cm[j] = best;
        np_[j] = -(float)(j * kCW + tag_of<5>(top));
      }
    }
  }
  __syncthreads();

  // ---- kPlanQ lanes per (row, tile)
  const size_t np = (size_t)a.plan_stride * T;
  int* const plan_i = reinterpret_cast<int*>(a.plan);
  const int q = ti & (kPlanQ - 1);
  const f32x2 nc2 = pack2(-c, -c);
  // (lanes past the tiles or rows compute on a valid place and write nothing: the shuffles below
  // want whole warps)
  for (int t0 = 0; t0 < T; t0 += tpr / kPlanQ) {
    const int t = min(t0 + ti / kPlanQ, T - 1);
    const bool has = live && t0 + ti / kPlanQ < T;
    const float f0 = (float)(t * tw) + a.shift;            // the tile's ends and centre
    const float f1 = (float)(min((t + 1) * tw, a.n_out) - 1) + a.shift;
    const float fkc = (float)(t * tw + tw / 2) + a.shift;

    // the chunk whose maximum gives the best term at kc
    float vb = -INFINITY;
    const f32x2 kc2 = pack2(fkc, fkc);
#pragma unroll 4
    for (int j = 2 * q; j < nchp; j += 2 * kPlanQ) {
      const float2 m = *reinterpret_cast<const float2*>(cm + j), p = *reinterpret_cast<const float2*>(np_ + j);
      const f32x2 d = add2(kc2, pack2(p.x, p.y));
      float v0, v1;
      unpack2(fma2(mul2(d, d), nc2, pack2(m.x, m.y)), v0, v1);
      vb = fmaxf(vb, fmaxf(tagged<7>(v0, j), tagged<7>(v1, j + 1)));
    }
#pragma unroll
    for (int d = 1; d < kPlanQ; d <<= 1) vb = fmaxf(vb, __shfl_xor_sync(0xffffffffu, vb, d));
    const bool any = vb != -INFINITY;                     // some term is finite
    const int jb = any ? tag_of<7>(vb) : 0;

    // the maximum over that chunk (half of it for each lane)
    float sb = -INFINITY;
    {
      constexpr int kShare = kCW / kPlanQ;
      const float* zj = z + jb * kZS + q * kShare;
      const float d0 = fkc - (float)(jb * kCW + q * kShare);
      f32x2 d01 = pack2(d0, d0 - 1.f);
      const f32x2 dn2 = pack2(-2.f, -2.f);
#pragma unroll
      for (int u = 0; u < kShare; u += 4) {
        const float4 x = *reinterpret_cast<const float4*>(zj + u);
        float v0, v1, v2, v3;
        unpack2(fma2(mul2(d01, d01), nc2, pack2(x.x, x.y)), v0, v1);
        d01 = add2(d01, dn2);
        unpack2(fma2(mul2(d01, d01), nc2, pack2(x.z, x.w)), v2, v3);
        d01 = add2(d01, dn2);
        const int i = q * kShare + u;
        sb = fmaxf(sb, fmaxf(tagged<5>(v0, i), tagged<5>(v1, i + 1)));
        sb = fmaxf(sb, fmaxf(tagged<5>(v2, i + 2), tagged<5>(v3, i + 3)));
      }
    }
#pragma unroll
    for (int d = 1; d < kPlanQ; d <<= 1) sb = fmaxf(sb, __shfl_xor_sync(0xffffffffu, sb, d));
    const int ub = tag_of<5>(sb);
    const float zm = z[jb * kZS + ub];
    int mh = jb * kCW + ub;
    const float fm = (float)mh;
    const float dk = fkc - fm, da = f0 - fm, db = f1 - fm;
    const float alpha = fmaf(-dk * dk, c, zm);
    const float lb = fminf(fmaf(-da * da, c, zm), fmaf(-db * db, c, zm)) - kCut;

    // the window in chunks
    int wlo = 0x7fffffff, whi = -1;
    {
      const float c0 = (float)(2 * q * kCW);
      f32x2 e0 = pack2(f0 - c0 - (float)(kCW - 1), f0 - c0 - (float)(2 * kCW - 1));   // f0 - chunk's last
      f32x2 e1 = pack2(c0 - f1, c0 + (float)kCW - f1);                                // chunk's first - f1
      const f32x2 up = pack2((float)(2 * kPlanQ * kCW), (float)(2 * kPlanQ * kCW));
      const f32x2 dn = pack2(-(float)(2 * kPlanQ * kCW), -(float)(2 * kPlanQ * kCW));
#pragma unroll 4
      for (int j = 2 * q; j < nchp; j += 2 * kPlanQ) {
        const float2 m = *reinterpret_cast<const float2*>(cm + j);
        float a0, a1, b0, b1, v0, v1;
        unpack2(e0, a0, a1);
        unpack2(e1, b0, b1);
        const f32x2 d = pack2(fmaxf(fmaxf(a0, b0), 0.f), fmaxf(fmaxf(a1, b1), 0.f));
        e0 = add2(e0, dn);
        e1 = add2(e1, up);
        unpack2(fma2(mul2(d, d), nc2, pack2(m.x, m.y)), v0, v1);
        if (v0 >= lb) {
          wlo = min(wlo, j);
          whi = j;
        }
        if (v1 >= lb) {
          wlo = min(wlo, j + 1);
          whi = j + 1;
        }
      }
    }
#pragma unroll
    for (int d = 1; d < kPlanQ; d <<= 1) {
      wlo = min(wlo, __shfl_xor_sync(0xffffffffu, wlo, d));
      whi = max(whi, __shfl_xor_sync(0xffffffffu, whi, d));
    }
    // narrow the hull block by block, chunk by chunk: lane 0 from its start, lane 1 from its end
    // (it holds mh's block, whose bound reaches LB)
    const bool win = any && whi >= 0;
    int j = win ? (q == 0 ? wlo : whi) : 0, edge = 0;
    const int jend = win ? (q == 0 ? whi : wlo) : 0, jstep = q == 0 ? 1 : -1;
    for (;;) {
      const float4 m = *reinterpret_cast<const float4*>(bm + 4 * j);
      const float ms[4] = {m.x, m.y, m.z, m.w};
      const float a0 = f0 - (float)(j * kCW) - 7.f, b0 = (float)(j * kCW) - f1;
      int mask = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float d = fmaxf(fmaxf(a0 - 8.f * i, b0 + 8.f * i), 0.f);
        if (fmaf(-d * d, c, ms[i]) >= lb) mask |= 1 << i;
      }
      edge = 4 * j + (q == 0 ? (mask ? __ffs(mask) - 1 : 0) : (mask ? 32 - __clz(mask) : 4));
      if (mask != 0 || j == jend) break;
      j += jstep;
    }
    const int other = __shfl_xor_sync(0xffffffffu, edge, 1);
    if (has && q == 0) {
      const int lo = win ? edge * 8 : 0, hi = win ? min(other * 8, len) : 0;
      mh = max(lo, min(mh, hi - 1));
      const size_t pi = (size_t)t * a.plan_stride + row;
      a.plan[pi] = any ? alpha : -INFINITY;
      plan_i[np + pi] = lo | ((hi - lo) << 16);
      plan_i[2 * np + pi] = mh;
      if (hi > lo) {
        atomicMin(&s_lo[t / kWinWarps], lo);
        atomicMax(&s_hi[t / kWinWarps], hi);
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
    if ((a.len & 3) == 0 && (reinterpret_cast<uintptr_t>(a.x) & 15u) == 0) a.vec |= 1;
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
// are summed in segments).  8 ends where exact sums become the faster ones (at 256^2, per pass:
// eps 7 12.7 against 23.5 us, eps 5 13.0 against 10.3).
int tile_width_for(float c) {
  const float reach = 2.f * sqrtf(kCut / c);
  auto need = [&](float w) { return w * (w + reach) * c; };
  if (need(32.f) <= 42.f) return 32;
  if (need(16.f) <= 64.f) return 16;
  if (need(8.f) <= 45.f) return 8;
  return 0;
}

void band_set_eps(BandArgs& a, double eps) {
  a.c = (float)(1.4426950408889634 / (2.0 * eps));
  a.eps = (float)eps;
  const int tw = tile_width_for(a.c);
  a.tile_w = tw == 0 ? 16 : tw;
  a.group = tw == 0 ? 2 : 8;
  a.wide_span = kWinWarps * a.tile_w + (int)(2.6f * sqrtf(kCut / a.c));
  if (tw != 0)
    for (int i = 0; i <= 32; ++i) a.step[i] = (float)exp2(32.0 * (i - 16) * (double)a.c);
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

template <int MODE, int MAXP>
void band_pass(cudaStream_t s, BandTable<MAXP>& t, int form) {
  plan_pass(s, t);
  ktimer_begin(s, form == kFormFp32 ? kKBand : kKTensor);
  bool exact = true;
  for (int q = 0; q < t.n; ++q) exact = exact && t.p[q].group == 2;
  if (exact)
    exact_launch<MODE, MAXP>(s, t);
  else if (form == kFormFp32)
    window_launch<MODE, kFormFp32, MAXP>(s, t);
  else if (form == kFormSplit)
    window_launch<MODE, kFormSplit, MAXP>(s, t);
  else
    window_launch<MODE, kFormSingle, MAXP>(s, t);
  ktimer_end(s);
}

template void band_pass<0, 1>(cudaStream_t, BandTable<1>&, int);
template void band_pass<1, 1>(cudaStream_t, BandTable<1>&, int);
template void band_pass<0, 2>(cudaStream_t, BandTable<2>&, int);
template void band_pass<1, 2>(cudaStream_t, BandTable<2>&, int);
template void band_pass<0, kMaxBatch>(cudaStream_t, BandTable<kMaxBatch>&, int);
template void band_pass<1, kMaxBatch>(cudaStream_t, BandTable<kMaxBatch>&, int);

// the plan kernel stages eight rows: more than the default 48 KB from rows of 1152 on
cudaError_t plan_configure() {
  const int lim = (int)(kPlanRows * plan_row_floats(4096 / kCW) * sizeof(float)) + 2 * 256 * (int)sizeof(int);
  cudaError_t e = cudaFuncSetAttribute(band_plan_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(band_plan_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(band_plan_kernel<kMaxBatch>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
  return e;
}

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

void tilt_prepare(fot_ctx* c, const double* eps, int n, int64_t* launches) {
  if (!c->tilt) return;
  TiltArgs t{};
  t.out = c->tilt;
  c->tilt_eps.clear();
  for (int i = 0; i < n && (int)c->tilt_eps.size() < kTiltTables; ++i) {
    if (!c->tilt_eps.empty() && c->tilt_eps.back() == eps[i]) continue;
    const float cc = (float)(1.4426950408889634 / (2.0 * eps[i]));
    const int tw = tile_width_for(cc);
    if (tw < 16) continue;                    // narrow tiles, exact windows: no table
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
  if (!c->tilt || tile_w < 16) return nullptr;
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
  int64_t k = 2 * 2;
  // pass over the contiguous axis: rows of pot_in, outputs along cols, written [k][L]
  t.p[0] = band_args(c, pot_in, c->rows, c->cols, eps, (float)(1.4426950408889634 / eps));
  t.p[0].y = c->R;
  const uint4* tilt = tilt_for(c, eps, t.p[0].group == 8 ? t.p[0].tile_w : 0, &k);
  t.p[0].tilt = tilt;
  band_pass<0>(c->stream, t, form);
  // pass over the row axis (input R[k][L], log2 units) with the fused potential update
  t.p[0] = band_args(c, c->R, c->cols, c->rows, eps, 1.f);
  t.p[0].tilt = tilt;
  t.p[0].y = pot_out;
  t.p[0].lmarg = lmarg;
  t.p[0].logsum = logsum;
  band_pass<1>(c->stream, t, form);
  c->launches += k;
}

// Two half-steps of one context in the same launches (2 per pass).
void half_step_band_pair(fot_ctx* c, const float* inA, const float* inB, const float* lmarg, double eps, float* outA,
                         float* outB, float* logsumA, float* logsumB, const PairSpace& second) {
  const int form = form_of(c);
  BandTable<2> t{};
  t.n = 2;
  t.spin_limit = c->spin;
  int64_t k = 2 * 2;
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
    if (pass == 0)
      band_pass<0>(c->stream, t, form);
    else
      band_pass<1>(c->stream, t, form);
  }
  c->launches += k;
}

}  // namespace fot
