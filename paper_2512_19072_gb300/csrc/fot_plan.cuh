// Window plan of a banded pass, device code: used by the plan kernel (fot_band.cu) and by the
// one-kernel passes of small problems (fot_small.cuh).
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
// A row with a NaN or +inf in it is not to pass for one without: its blocks' maxima keep either (as
// kWild), every one of its windows is the whole row and its offsets are NaN, so that the sums
// come out as NaN (or are taken exactly, should the row hold values beyond kWild / 3).
//
// Arg-maxima carry the index in the low mantissa bits of the value they compare (5 bits for a
// position, 7 for a chunk): one maximum instead of a compare and two selects; a chunk's maximum
// is rounded by up to 2^-16 of itself that way.  An offset that this takes from a lesser chunk (where the
// values differ by less than that) only widens the window, and raises the operands: sums beyond
// the range of FP32 are done again in segments or exactly.
//
// What bounds it: latency and issue slots (4 MB of input at 1024^2, in L2).  Two lanes serve a
// (row, tile): each takes every other pair of chunks (packed FP32 pairs), half of the scanned
// chunk and one end of the window.  Chunks are padded to 36 words: lanes on different chunks read
// different banks, lanes on the same chunk broadcast.
#pragma once

#include "fot_window.cuh"

namespace fot {

constexpr int kPlanRows = 8;                  // rows of a CTA: one row group of the window kernel
constexpr int kPlanThreads = 512;
constexpr int kPlanQ = 2;                     // lanes per (row, tile)
constexpr int kZS = kCW + 4;                  // words of a staged chunk
constexpr float kWild = 3e38f;                // block maximum that stands for NaN and +inf

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

// the larger of two values, NaN when either is
__device__ __forceinline__ float max_nan(float a, float b) {
  float m;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
  return m;
}

// Stage one row: blocks of 8 positions, a thread each (ti of tpr threads); four neighbouring threads
// share a chunk.  load(m0, v): positions m0 .. m0 + 7, -inf outside the row.
template <typename F>
__device__ __forceinline__ void plan_stage(const BandArgs& a, float* row_smem, int ti, int tpr, F load) {
  const int nch = a.n_chunks, nchp = (nch + 3) & ~3;
  float* const cm = row_smem;
  float* const np_ = cm + nchp;                           // minus the maxima's positions
  float* const bm = np_ + nchp;
  float* const z = bm + 4 * nch;
  const f32x2 sc2 = pack2(a.x_scale, a.x_scale);
  for (int b = ti; b < nchp * 4; b += tpr) {
    const int m0 = b * 8, j = b >> 2, u0 = (b & 3) * 8;
    float v[8];
    load(m0, v);
    float best = -INFINITY, top = -INFINITY;              // block maximum; the same with its position
#pragma unroll
    for (int u = 0; u < 8; u += 2) {
      unpack2(mul2(pack2(v[u], v[u + 1]), sc2), v[u], v[u + 1]);
      best = max_nan(best, max_nan(v[u], v[u + 1]));
      top = fmaxf(top, fmaxf(tagged<5>(v[u], u0 + u), tagged<5>(v[u + 1], u0 + u + 1)));
    }
    if (!(best <= kWild)) best = kWild;
    if (j < nch) {
      float4* const zb = reinterpret_cast<float4*>(z + j * kZS + u0);
      zb[0] = make_float4(v[0], v[1], v[2], v[3]);
      zb[1] = make_float4(v[4], v[5], v[6], v[7]);
      bm[b] = best;
    }
    // (the four threads of a chunk are neighbours and take this iteration together)
    const unsigned quad = 0xfu << (threadIdx.x & 28);
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

// One (row, tile): offset, window [lo, hi) and mh, on lane q = 0 of the kPlanQ that serve it (whole warps
// call this).  alpha is -inf for a row without a finite term.
struct PlanEntry {
  float alpha;
  int lo, hi, mh;
};
__device__ __forceinline__ PlanEntry plan_tile(const BandArgs& a, const float* row_smem, int t, int q) {
  const int nch = a.n_chunks, nchp = (nch + 3) & ~3, tw = a.tile_w;
  const float c = a.c;
  const float* const cm = row_smem;
  const float* const np_ = cm + nchp;
  const float* const bm = np_ + nchp;
  const float* const z = bm + 4 * nch;
  const f32x2 nc2 = pack2(-c, -c);
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
  const bool wild = vb > kWild / 3.f;
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
  PlanEntry e;
  e.lo = win && !wild ? edge * 8 : 0;
  e.hi = wild ? a.len : win ? min(other * 8, a.len) : 0;
  e.mh = max(e.lo, min(mh, e.hi - 1));
  e.alpha = wild ? NAN : any ? alpha : -INFINITY;
  return e;
}

}  // namespace fot
