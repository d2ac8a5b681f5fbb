// Window sums of a banded pass (plan: fot_band.cu).
//
// A unit is a group of 8 rows r and a tile of TN = 16 or 32 consecutive outputs o = kc + kap
// around the tile centre kc, one warp each.  An item, one CTA, is four neighbouring tiles of a row
// group, whose windows overlap: the part of the rows they need is staged in shared memory by one
// bulk copy per row (one copy per tile would read 2.5 times as much from L2).  Nothing but the
// staged rows is shared between the warps.
//
// Windows differ (13 steps on average at 1024^2, up to 45 where the transport map jumps), so the
// plan hands over the items with the long ones first: started last, they ran alone for a third of
// the pass.
//
// Tilt identity.  With m = lo_r + p (p a position in row r's window, W the unit's longest window)
// and any reference position M_r,
//     e(m, o) = [x_r[m] - (kc - m)^2 c - alpha_r] + 2 kap (m - M_r) c
//               + alpha_r + (2 kap (M_r - kc) - kap^2) c,
// so  y[kc + kap][r] = alpha_r + (2 kap (M_r - kc) - kap^2) c + log2 sum_p T[kap][p] X[p][r],
// X[p][r] = 2^(e(m, kc) - alpha_r) (one exponential per row and position, shared by the tile's
// outputs) and T[kap][p] = 2^(2 kap (p - p0) c) the same for every row: a matrix product with
// M = outputs, N = rows, K = positions (the per-row max-offsets of the paper's Toeplitz
// contraction, Sec. 3.1).
//
// mma.sync rather than tcgen05.  A unit is 32 x 8 x ~250: its X has to be computed by the CUDA
// cores, position by position, and a lane of an m16n8k16 B operand owns exactly the positions of
// one row that it has computed, in registers; nothing passes through shared memory and no warp
// waits for another.  The tcgen05 form of this pass (128-row units, X written to shared memory,
// five barriers per 32 positions, one CTA per SM) took 34 us per pass at 1024^2 with the tensor
// pipe 3 % busy; it also summed the union of 128 rows' windows, 1.4 times the terms of 8-row units.
//
// Horner over 16-position steps.  T[kap][p + 16] = T[kap][p] 2^(32 kap c): moving the reference
// by one step scales row kap by a constant.  So the operand fragments of T for one step stay in
// registers for the whole window, which is walked from its end to its start; the sums D become
// D G + (the step's products), G = 2^(32 kap c), and end up referred to lo_r.  The products start
// from zero and are added by the CUDA cores: the tensor core truncates what it accumulates, and
// a chain of steps through it added up to 1e-5 of a sum.  Two steps per turn of the loop, their
// products added a turn later, so that the exponentials of one turn run while the tensor core
// works on the last: a long window is one warp's chain (45 steps at 1024^2 where the mean is 13).
//
// Operands.  kFormSplit: BF16 hi + lo parts, hi*hi + hi*lo + lo*hi (2^-16 relative per product);
// kFormSingle: hi*hi; kFormFp32: TF32 hi + lo parts (2^-21), two m16n8k8 per step and product.
//
// Range.  With kmax = TN/2 and D the farthest window position from mh: a term that matters to
// output kap has X >= 2^-(2 kmax D c) (alpha is e(mh, kc); the largest term at kap is at least
// mh's), and referring the sum to lo_r instead of mh moves it by at most 2 kmax (mh - lo_r) c.  A
// row is in range while the first is <= kTiltMax and both together are <= kRangeMax: what flushes
// to zero below 2^-126 is then less than W 2^-30 of a sum, and sums stay below 2^(100 + 9) times
// 2^(how far the offset lies below the maximum).  An offset that lies too far below shows as an
// output that is not finite; such a unit is summed again exactly.
//
// Units outside that bound: a 32-wide tile is cut in two 16-wide ones that take their own
// offsets; what fails again (or a problem whose eps is too small for any unit) is summed exactly:
// one exponential per term and output, lanes on 2 rows x 16 outputs, offset e(mh, o).
//
// What bounds it: issue slots and latency.  A split-BF16 step at TN = 32 is about 40 instructions
// and 6 MMAs (48 tensor cycles per SM quarter), a unit's set-up and outputs about 450.  A loop of
// 200 iterations at 1024^2 (800 passes, plan and launch gaps included): split BF16 31.9 -> 16.6 ms,
// FP32 45.7 -> 18.4 ms (it was FFMA with the operands through shared memory); 100 iterations at
// 2048^2, split BF16: 39.8 -> 20.9 ms; 64^2 at eps 1 (exact windows), 200 iterations: 14.5 -> 4.5 ms.
#pragma once

#include "fot_band.cuh"

namespace fot {

constexpr int kCW = 32;              // chunk width of the plan
constexpr float kCut = 40.f;         // window cut-off, log2 units
constexpr float kTiltMax = 96.f;
constexpr float kRangeMax = 100.f;
constexpr int kWinWarps = 4;
constexpr int kWinThreads = 32 * kWinWarps;
constexpr int kPitchCap = 40 * 32 + 16;   // floats staged per row at most (41 KB of 8 rows: five CTAs fit
                                          // an SM); wider spans are read from global memory
constexpr int kSpinDefault = 1 << 20;     // polls of a bounded wait
constexpr int kTiltWords = 2 * 2 * 32;    // uint4 words of a tilt table: 2 row tiles x (hi, lo) x lanes

// staged row pitch for a span of n floats: a multiple of 16 that is 16 mod 32, so that the two
// rows a quarter warp reads together lie on different banks
__host__ __device__ inline int stage_pitch(int n) { return (n + 15) / 32 * 32 + 16; }

// ---- small device pieces ------------------------------------------------------------------

// Programmatic dependent launch: wait for the kernel before this one (no-op when launched
// without the attribute); let the next one be set up.
__device__ __forceinline__ void grid_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

typedef unsigned long long f32x2;    // two packed FP32 values
__device__ __forceinline__ f32x2 pack2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}

// BF16 hi and lo parts of two values (a in the low half)
__device__ __forceinline__ void split_bf16(float a, float b, uint32_t& hi, uint32_t& lo) {
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(hi) : "f"(b), "f"(a));
  const float ra = a - __uint_as_float(hi << 16), rb = b - __uint_as_float(hi & 0xffff0000u);
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(lo) : "f"(rb), "f"(ra));
}
// TF32 hi and lo parts (the tensor core reads the upper 19 bits of each)
__device__ __forceinline__ void split_tf32(float a, uint32_t& hi, uint32_t& lo) {
  hi = __float_as_uint(a) & 0xffffe000u;
  lo = __float_as_uint(a - __uint_as_float(hi));
}

// d = a b + (zero or d); FP32 operands: one m16n8k8 half, BF16: m16n8k16
__device__ __forceinline__ void mma_bf16_0(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void mma_bf16(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void mma_tf32_0(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%10,%10,%10};"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(0.f));
}
__device__ __forceinline__ void mma_tf32(float* d, const uint32_t* a, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

template <int FORM>
__device__ __forceinline__ void mma(float* d, const uint32_t* a, uint32_t b0, uint32_t b1, bool zero) {
  if (FORM == kFormFp32) {
    if (zero) mma_tf32_0(d, a, b0, b1);
    else mma_tf32(d, a, b0, b1);
  } else {
    if (zero) mma_bf16_0(d, a, b0, b1);
    else mma_bf16(d, a, b0, b1);
  }
}

// T[kap][p], exponent clamped (only units that are never accepted reach the clamp)
__device__ __forceinline__ float tilt_value(float kap, float p, float c) {
  return ex2(fminf(fmaxf(2.f * kap * p * c, -126.f), 126.f));
}
// A-operand fragments of 16 rows kap0 .. kap0 + 15 of T for one step.  Lane (g, q) holds rows g
// and g + 8; the columns of q are positions 4q .. 4q + 3 (the K index permuted alike in X).
__device__ __forceinline__ void tilt_fragments_bf16(float c, int kap0, int lane, uint32_t* hi, uint32_t* lo) {
  const float ka = (float)(kap0 + (lane >> 2)), kb = ka + 8.f, p = (float)(4 * (lane & 3));
  split_bf16(tilt_value(ka, p, c), tilt_value(ka, p + 1.f, c), hi[0], lo[0]);
  split_bf16(tilt_value(kb, p, c), tilt_value(kb, p + 1.f, c), hi[1], lo[1]);
  split_bf16(tilt_value(ka, p + 2.f, c), tilt_value(ka, p + 3.f, c), hi[2], lo[2]);
  split_bf16(tilt_value(kb, p + 2.f, c), tilt_value(kb, p + 3.f, c), hi[3], lo[3]);
}
// m16n8k8 half h: positions 4q + 2h (k = q) and 4q + 2h + 1 (k = q + 4)
__device__ __forceinline__ void tilt_fragments_tf32(float c, int kap0, int h, int lane, uint32_t* hi, uint32_t* lo) {
  const float ka = (float)(kap0 + (lane >> 2)), kb = ka + 8.f, p = (float)(4 * (lane & 3) + 2 * h);
  split_tf32(tilt_value(ka, p, c), hi[0], lo[0]);
  split_tf32(tilt_value(kb, p, c), hi[1], lo[1]);
  split_tf32(tilt_value(ka, p + 1.f, c), hi[2], lo[2]);
  split_tf32(tilt_value(kb, p + 1.f, c), hi[3], lo[3]);
}

// ---- mbarrier and bulk copy ---------------------------------------------------------------

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" :: "r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_test(uint32_t bar, uint32_t parity) {   // returns at once
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {    // may suspend for a while
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
               : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait for the staged rows: limit - 1 polls.  A limit below the default (the test setting)
// polls without suspending; the shortest does not poll at all, since the rows have usually arrived
// by the time a warp waits for them.  On time-out FOT_ETIMEOUT is latched and the copies are waited
// for with the full limit; false when they still have not arrived.
__device__ __forceinline__ bool stage_wait(uint32_t bar, uint32_t parity, int limit, int* err) {
  const bool quick = limit < kSpinDefault;
  for (int i = 1; i < limit; ++i)
    if (quick ? mbar_test(bar, parity) : mbar_try(bar, parity)) return true;
  raise_error(err, FOT_ETIMEOUT);
  for (int i = 0; i < kSpinDefault; ++i)
    if (mbar_try(bar, parity)) return true;
  return false;
}
// 1-D bulk copy global -> shared (16-byte aligned addresses, size a multiple of 16)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               :: "r"(dst), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// ---- one output ----------------------------------------------------------------------------

// S (log2 units) -> the pass's output: the value itself, or f = eps (log marginal - S)
template <int MODE>
__device__ __forceinline__ float finish_output(const BandArgs& a, float s2, float lm, float& s, bool& bad) {
  if (MODE == 0) return s2;
  s = __fmul_rn(s2, kLn2);
  if (lm == -INFINITY) return -INFINITY;
  const float pot = __fmul_rn(a.eps, __fsub_rn(lm, s));
  bad |= !isfinite(pot);
  return pot;
}

// four positions m .. m + 3 of a row (p of them are inside the window: -inf elsewhere)
__device__ __forceinline__ float4 fetch4(const float* xp, int m, int left, bool vec) {
  if (left <= 0) return make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  if (vec) return *reinterpret_cast<const float4*>(xp + m);   // window ends are multiples of 4
  return make_float4(xp[m], left > 1 ? xp[m + 1] : -INFINITY, left > 2 ? xp[m + 2] : -INFINITY,
                     left > 3 ? xp[m + 3] : -INFINITY);
}
__device__ __forceinline__ float4 lds4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}

// exponents of four positions: x sc - alpha - (d - j)^2 c, j = 0 .. 3 (d01 = (d, d - 1), d the
// first one's distance).  x sc - alpha is formed first: near the window's maximum it cancels, so
// that the rounding error is that of the small difference and not of the offset.
__device__ __forceinline__ void exponents4(const float4& x, f32x2 sc2, f32x2 na2, f32x2 nc2, f32x2 d01, float* e) {
  const f32x2 d23 = add2(d01, pack2(-2.f, -2.f));
  const f32x2 u01 = fma2(pack2(x.x, x.y), sc2, na2), u23 = fma2(pack2(x.z, x.w), sc2, na2);
  unpack2(fma2(mul2(d01, d01), nc2, u01), e[0], e[1]);
  unpack2(fma2(mul2(d23, d23), nc2, u23), e[2], e[3]);
}

// One row of a unit as a lane sees it: offset, window [lo, lo + wl), position mh, and where its
// positions are: row[m] in shared or global memory, saddr the shared address of row[0] (staged
// rows; minf is a shared address that holds four -inf).
struct RowView {
  float alpha;
  int lo, wl, mh;
  const float* row;
  uint32_t saddr, minf;
  bool staged, vec;
};

// What a warp keeps of one problem: the operand fragments of T for (c, TN), hi and lo parts of
// each row tile (FP32 operands: of both m16n8k8 halves), and the step scales G.
template <int FORM>
struct Tilt {
  static constexpr int NH = FORM == kFormFp32 ? 2 : 1;
  uint32_t hi[2][4 * NH], lo[2][4 * NH];
  f32x2 G[2][2];
  // tw = 16 (first row tile only) or 32; table: a.tilt holds the fragments (BF16 forms)
  __device__ __forceinline__ void load(const BandArgs& a, int tw, bool table) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      if (16 * t >= tw) break;
      const int kap0 = 16 * t - tw / 2;
      if (FORM == kFormFp32) {
#pragma unroll
        for (int h = 0; h < NH; ++h) tilt_fragments_tf32(a.c, kap0, h, lane, hi[t] + 4 * h, lo[t] + 4 * h);
      } else if (table) {
        const uint4 h4 = __ldg(a.tilt + t * 64 + lane), l4 = __ldg(a.tilt + t * 64 + 32 + lane);
        hi[t][0] = h4.x; hi[t][1] = h4.y; hi[t][2] = h4.z; hi[t][3] = h4.w;
        lo[t][0] = l4.x; lo[t][1] = l4.y; lo[t][2] = l4.z; lo[t][3] = l4.w;
      } else {
        tilt_fragments_bf16(a.c, kap0, lane, hi[t], lo[t]);
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float v = a.step[kap0 + (lane >> 2) + 8 * h + 16];
        G[t][h] = pack2(v, v);
      }
    }
  }
};

// The tilted matrix product of one unit (see the top).  Lane (g = lane / 4, q = lane % 4) owns row
// r0 + g (rv) for X, and outputs kap g and g + 8 of each row tile of columns r0 + 2q, + 1.
// Returns false, with nothing written, when a sum left the range of FP32 (warp-uniform).
template <int MODE, int FORM, int TN, bool STAGED>
__device__ __forceinline__ bool gemm_unit(const BandArgs& a, int r0, int k0, float kc, const RowView& rv, int W,
                                          const Tilt<FORM>& tilt, bool skip) {
  constexpr int MT = TN / 16;
  constexpr int NH = Tilt<FORM>::NH;
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const float c = a.c;
  const float sc = a.x_scale;
  const f32x2 sc2 = pack2(sc, sc), nc2 = pack2(-c, -c);
  const float na = rv.wl == 0 ? 0.f : -rv.alpha;
  const f32x2 na2 = pack2(na, na);
  f32x2 D[MT][2];                                         // (columns 2q, 2q + 1) of rows g and g + 8
  float P[2][MT][4];                                      // the last turn's products
#pragma unroll
  for (int t = 0; t < MT; ++t) {
    D[t][0] = D[t][1] = pack2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 4; ++u) P[0][t][u] = P[1][t][u] = 0.f;
  }
  const int turns = (W + 31) >> 5;
  int pos = rv.lo + 32 * turns - 16 + 4 * q;              // this lane's first position of the step
  int left = rv.wl - 32 * turns + 16 - 4 * q;             // of it and after it in the window
  uint32_t addr = rv.saddr + 4u * (uint32_t)pos;
  const float d0 = kc - (float)pos;
  f32x2 d01 = pack2(d0, d0 - 1.f);
  const f32x2 d16 = pack2(16.f, 16.f);
  auto fetch = [&]() {
    float4 v;
    if (STAGED)
      v = lds4(left > 0 ? addr : rv.minf);
    else
      v = fetch4(rv.row, pos, left, rv.vec);
    addr -= 64u;
    pos -= 16;
    left += 16;
    return v;
  };
  auto absorb = [&]() {                                   // D <- (D G + P0) G + P1
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int t = 0; t < MT; ++t) {
        D[t][0] = fma2(D[t][0], tilt.G[t][0], pack2(P[i][t][0], P[i][t][1]));
        D[t][1] = fma2(D[t][1], tilt.G[t][1], pack2(P[i][t][2], P[i][t][3]));
      }
  };
  float4 xn[2];
  if (turns > 0) {
    xn[0] = fetch();
    xn[1] = fetch();
  }
#pragma unroll 1
  for (int i = 0; i < turns; ++i) {
    const float4 xv[2] = {xn[0], xn[1]};
    if (i + 1 < turns) {
      xn[0] = fetch();
      xn[1] = fetch();
    }
    uint32_t xh[2][2 * NH], xl[2][2 * NH];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      float e[4];
      exponents4(xv[v], sc2, na2, nc2, d01, e);
      d01 = add2(d01, d16);
#pragma unroll
      for (int u = 0; u < 4; ++u) e[u] = ex2(e[u]);
      if (FORM == kFormFp32) {
#pragma unroll
        for (int u = 0; u < 4; ++u) split_tf32(e[u], xh[v][u % (2 * NH)], xl[v][u % (2 * NH)]);
      } else {
        split_bf16(e[0], e[1], xh[v][0], xl[v][0]);
        split_bf16(e[2], e[3], xh[v][1], xl[v][1]);
      }
    }
    absorb();
    // the small products first, then hi * hi
#pragma unroll
    for (int part = FORM == kFormSingle ? 2 : 0; part < 3; ++part)
#pragma unroll
      for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int t = 0; t < MT; ++t) {
            const uint32_t* A = (part == 0 ? tilt.lo[t] : tilt.hi[t]) + 4 * h;
            const uint32_t* Bm = (part == 1 ? xl[v] : xh[v]) + (NH == 2 ? 2 * h : 0);
            const bool first = part == (FORM == kFormSingle ? 2 : 0) && h == 0;
            mma<FORM>(P[v][t], A, Bm[0], Bm[1], first);
          }
  }
  absorb();

  // outputs of columns rA = r0 + 2q and rA + 1; an empty row (alpha = -inf) has sums 0: log -inf
  const int rA = r0 + 2 * q;
  const float al[2] = {__shfl_sync(0xffffffffu, rv.alpha, 8 * q), __shfl_sync(0xffffffffu, rv.alpha, 8 * q + 4)};
  const float mr[2] = {(float)__shfl_sync(0xffffffffu, rv.lo, 8 * q) - kc,
                       (float)__shfl_sync(0xffffffffu, rv.lo, 8 * q + 4) - kc};   // reference - kc
  const size_t y0 = (size_t)(k0 + g) * a.n_rows + rA;
  const size_t ystep = (size_t)8 * a.n_rows;
  const bool full = (a.vec & 2) && k0 + TN <= a.n_out && r0 + 8 <= a.n_rows;   // warp-uniform
  float lm[2 * MT][2];
  if (MODE == 1) {
#pragma unroll
    for (int i = 0; i < 2 * MT; ++i) {
      const float* p = a.lmarg + y0 + i * ystep;
      if (full) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(p));
        lm[i][0] = v.x;
        lm[i][1] = v.y;
      } else {
        const bool in = k0 + g + 8 * i < a.n_out;
        lm[i][0] = in && rA < a.n_rows ? __ldg(p) : -INFINITY;
        lm[i][1] = in && rA + 1 < a.n_rows ? __ldg(p + 1) : -INFINITY;
      }
    }
  }
  float s2[2 * MT][2], chk[2] = {0.f, 0.f};               // chk: NaN after a non-finite log-sum
#pragma unroll
  for (int i = 0; i < 2 * MT; ++i) {
    const float kap = (float)(8 * i - TN / 2 + g);
    float v[2];
    unpack2(D[i >> 1][i & 1], v[0], v[1]);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float l2 = FORM == kFormFp32 ? log2f(v[u]) : lg2(v[u]);
      s2[i][u] = __fadd_rn(al[u], fmaf(fmaf(2.f * kap, mr[u], -kap * kap), c, l2));
      chk[u] = fmaf(s2[i][u], 0.f, chk[u]);
    }
  }
  if (__any_sync(0xffffffffu, (chk[0] != 0.f && al[0] != -INFINITY) || (chk[1] != 0.f && al[1] != -INFINITY)))
    return false;
  if (skip) return true;
  bool bad = false;
#pragma unroll
  for (int i = 0; i < 2 * MT; ++i) {
    float out[2], sv[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) out[u] = finish_output<MODE>(a, s2[i][u], MODE == 1 ? lm[i][u] : 0.f, sv[u], bad);
    const size_t yi = y0 + i * ystep;
    if (full) {
      *reinterpret_cast<float2*>(a.y + yi) = make_float2(out[0], out[1]);
      if (MODE == 1 && a.logsum) *reinterpret_cast<float2*>(a.logsum + yi) = make_float2(sv[0], sv[1]);
    } else if (k0 + g + 8 * i < a.n_out) {
#pragma unroll
      for (int u = 0; u < 2; ++u)
        if (rA + u < a.n_rows) {
          a.y[yi + u] = out[u];
          if (MODE == 1 && a.logsum) a.logsum[yi + u] = sv[u];
        }
    }
  }
  if (bad) raise_error(a.err, FOT_ENONFINITE);            // (outputs outside the image have lm = -inf)
  return true;
}

// Exact window sums of 2 rows x 16 outputs: lane (half, i) owns output k0 + i of its half's row,
// window [lo, lo + wl), xp[m] that row's position m.  Terms are taken relative to e(mh, o), which
// is within the range of FP32 of the maximum unless the maximum moves far from mh within the
// tile; a sum that overflows is done again from its exact maximum.
template <int MODE>
__device__ __forceinline__ void exact_pair(const BandArgs& a, int row, int k0, int lo, int wl, int mh, const float* xp,
                                           bool vec, bool skip) {
  const int o = k0 + (threadIdx.x & 15);
  const float fo = (float)o + a.shift, sc = a.x_scale, nc = -a.c;
  float out = -INFINITY;
  if (wl > 0) {
    const float dm = fo - (float)mh;
    float off = fmaf(dm * dm, nc, xp[mh] * sc);
    const f32x2 sc2 = pack2(sc, sc), nc2 = pack2(nc, nc), dn4 = pack2(-4.f, -4.f);
    const float d0 = fo - (float)lo;
    for (int pass = 0; pass < 2; ++pass) {
      const f32x2 no2 = pack2(-off, -off);
      f32x2 d01 = pack2(d0, d0 - 1.f);
      float s0 = 0.f, s1 = 0.f;
#pragma unroll 2
      for (int p = 0; p < wl; p += 4) {
        float e[4];
        exponents4(fetch4(xp, lo + p, wl - p, vec), sc2, no2, nc2, d01, e);
        d01 = add2(d01, dn4);
        s0 += ex2(e[0]) + ex2(e[1]);
        s1 += ex2(e[2]) + ex2(e[3]);
      }
      const float sum = s0 + s1;
      out = __fadd_rn(off, log2f(sum));
      if (sum <= 3.4e38f) break;
      // (a NaN ends here too and stays one)
      off = -INFINITY;
      d01 = pack2(d0, d0 - 1.f);
      for (int p = 0; p < wl; p += 4) {
        float e[4];
        exponents4(fetch4(xp, lo + p, wl - p, vec), sc2, pack2(0.f, 0.f), nc2, d01, e);
        d01 = add2(d01, dn4);
        off = fmaxf(fmaxf(off, fmaxf(e[0], e[1])), fmaxf(e[2], e[3]));
      }
    }
  }
  if (row >= a.n_rows || o >= a.n_out || skip) return;
  const size_t yi = (size_t)o * a.n_rows + row;
  float s = 0.f;
  bool bad = false;
  a.y[yi] = finish_output<MODE>(a, out, MODE == 1 ? __ldg(a.lmarg + yi) : 0.f, s, bad);
  if (MODE == 1 && a.logsum) a.logsum[yi] = s;
  if (bad) raise_error(a.err, FOT_ENONFINITE);
}

// the rows of a unit outside the tilted product, two at a time
template <int MODE>
__device__ __forceinline__ void exact_unit(const BandArgs& a, int r0, int k0, RowView rv, bool skip) {
  const int half = (threadIdx.x & 31) >> 4;
  for (int p = 0; p < 4; ++p) {
    const int src = 4 * (2 * p + half);
    const int l = __shfl_sync(0xffffffffu, rv.lo, src), w = __shfl_sync(0xffffffffu, rv.wl, src);
    const int m = __shfl_sync(0xffffffffu, rv.mh, src);
    const float* xr = (const float*)__shfl_sync(0xffffffffu, (unsigned long long)rv.row, src);
    exact_pair<MODE>(a, r0 + 2 * p + half, k0, l, w, m, xr, rv.vec, skip);
  }
}

// whether a row's operands stay in range of the tilted product (the top)
__device__ __forceinline__ bool row_in_range(float kmax, int lo, int hi, int mh, float c) {
  const float t = 2.f * kmax * c, far = t * (float)max(mh - lo, hi - mh);
  return far <= kTiltMax && far + t * (float)(mh - lo) <= kRangeMax;
}

// a 32-wide unit outside the bound: two 16-wide ones with the rows' exact maxima at their own
// centres, over the same windows (which cover theirs)
template <int MODE, int FORM>
__device__ __forceinline__ void split_unit(const BandArgs& a, int r0, int k0, RowView rv, int W, bool skip,
                                        unsigned long long* terms) {
  const int lane = threadIdx.x & 31, q = lane & 3;
  const float c = a.c, sc = a.x_scale;
  for (int sub = 0; sub < 2; ++sub) {
    const int ks = k0 + 16 * sub;
    if (ks >= a.n_out) break;
    const float kc = (float)(ks + 8) + a.shift;
    RowView r = rv;
    r.alpha = -INFINITY;
    for (int p = 4 * q; p < rv.wl; p += 16) {
      const float4 x = fetch4(rv.row, rv.lo + p, rv.wl - p, rv.vec);
      const float xs[4] = {x.x, x.y, x.z, x.w};
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const float d = kc - (float)(rv.lo + p + u);
        const float e = fmaf(-d * d, c, xs[u] * sc);
        if (e > r.alpha) {
          r.alpha = e;
          r.mh = rv.lo + p + u;
        }
      }
    }
#pragma unroll
    for (int d = 1; d < 4; d <<= 1) {
      const float oa = __shfl_xor_sync(0xffffffffu, r.alpha, d);
      const int om = __shfl_xor_sync(0xffffffffu, r.mh, d);
      if (oa > r.alpha || (oa == r.alpha && om < r.mh)) {
        r.alpha = oa;
        r.mh = om;
      }
    }
    if (__all_sync(0xffffffffu, r.wl == 0 || row_in_range(8.f, r.lo, r.lo + r.wl, r.mh, c))) {
      if (lane == 0) atomicAdd(terms + (FORM == kFormFp32 ? 0 : 2), (unsigned long long)W * 16 * 8);
      Tilt<FORM> tilt;
      tilt.load(a, 16, false);
      if (gemm_unit<MODE, FORM, 16, false>(a, r0, ks, kc, r, W, tilt, skip)) continue;
    }
    if (q == 0) atomicAdd(terms + 1, (unsigned long long)r.wl * 16);
    exact_unit<MODE>(a, r0, ks, r, skip);
  }
}

// a unit whose rows are not staged, or that is outside the bound, or whose sums left the range of
// FP32 (try_product false)
template <int MODE, int FORM>
__device__ __noinline__ void other_unit(const BandArgs& a, int r0, int k0, RowView rv, int W, bool try_product, bool skip,
                                        unsigned long long* terms) {
  if (try_product) {
    Tilt<FORM> tilt;
    tilt.load(a, a.tile_w, true);
    const float kc = (float)(k0 + (a.tile_w >> 1)) + a.shift;
    if (a.tile_w == 32 ? gemm_unit<MODE, FORM, 32, false>(a, r0, k0, kc, rv, W, tilt, skip)
                       : gemm_unit<MODE, FORM, 16, false>(a, r0, k0, kc, rv, W, tilt, skip))
      return;
  }
  if (a.tile_w == 32) {
    split_unit<MODE, FORM>(a, r0, k0, rv, W, skip, terms);
  } else {
    if ((threadIdx.x & 3) == 0) atomicAdd(terms + 1, (unsigned long long)rv.wl * 16);
    exact_unit<MODE>(a, r0, k0, rv, skip);
  }
}

// A warp's unit of the item that its CTA was launched for.
struct Unit {
  RowView rv;
  int r0, k0, row;                                        // first row and output, this lane's row
  bool pairs, out_of_range, skip;
};

// The start of a window CTA: read the item and this warp's plan entries, stage the rows; `meanwhile`
// runs while they are on their way.  s_x: four -inf (padded to 64 bytes), then the rows.  False: the
// warp has nothing to do.
template <int MAXP, typename F>
__device__ __forceinline__ bool open_unit(const BandTable<MAXP>& tab, const BandArgs& a, float* s_x, uint64_t* s_bar, Unit& u,
                                          F meanwhile) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  u.pairs = a.group == 2;
  if (tid == 0) {
    mbar_init(smem_addr(s_bar), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 4) s_x[tid] = -INFINITY;
  float* const rows = s_x + 16;
  grid_wait();
  grid_launch_next();
  if (tid < 2 && (int)blockIdx.x == a.item_base) a.order[tid] = 0;   // for the next pass's plan
  u.skip = error_latched(a.err);                          // an error is latched: write nothing
  // the item: row group, four tiles, and the span of the rows that they read
  int rg, tg, base, top;
  if (u.pairs) {
    const int local = (int)blockIdx.x - a.item_base;
    rg = local / a.items_row;
    tg = local - rg * a.items_row;
    base = 0;
    top = a.len;
  } else {
    const int4 it = a.items[(int)blockIdx.x - a.item_base];
    rg = it.x;
    tg = it.y;
    base = it.z;
    top = it.w;
  }
  const int r0 = a.group * rg;
  const int pitch = stage_pitch(top - base);
  const bool staged = top > base && pitch <= tab.pitch_max;
  const bool bulk = staged && (a.vec & 1);
  const int nr = min(a.group, a.n_rows - r0);
  if (bulk && warp == 0) {
    const uint32_t bytes = (uint32_t)(top - base) * 4u;   // the ends are multiples of 4 here
    __syncwarp();
    if (lane == 0) mbar_expect(smem_addr(s_bar), bytes * nr);
    __syncwarp();
    if (lane < nr)
      bulk_load(smem_addr(rows + lane * pitch), a.x + (size_t)(r0 + lane) * a.len + base, bytes, smem_addr(s_bar));
  }
  // the plan entry of this lane's row, for its warp's tile
  const int tile = tg * kWinWarps + warp;
  const int lr = u.pairs ? lane >> 4 : lane >> 2;
  u.r0 = r0;
  u.k0 = tile * a.tile_w;
  u.row = r0 + lr;
  RowView& rv = u.rv;
  rv.alpha = -INFINITY;
  int w1 = 0, w2 = 0;
  if (tile < a.n_tiles && u.row < a.n_rows) {
    const size_t np = (size_t)a.plan_stride * a.n_tiles, pi = (size_t)tile * a.plan_stride + u.row;
    rv.alpha = a.plan[pi];
    w1 = reinterpret_cast<const int*>(a.plan)[np + pi];
    w2 = reinterpret_cast<const int*>(a.plan)[2 * np + pi];
  }
  meanwhile();
  rv.lo = w1 & 0xffff;
  rv.wl = w1 >> 16;
  rv.mh = w2 & 0xffff;
  u.out_of_range = (w2 >> 16) != 0;
  rv.staged = staged;
  rv.vec = staged || (a.vec & 1);
  rv.row = staged ? rows + lr * pitch - base : a.x + (size_t)min(u.row, a.n_rows - 1) * a.len;
  rv.saddr = smem_addr(rows + lr * pitch) - 4u * (uint32_t)base;
  rv.minf = smem_addr(s_x);
  if (staged && !bulk) {
    // rows that are not 16-byte aligned: plain loads, -inf up to the next multiple of 4
    const int n4 = (top - base + 3) & ~3;
    const float* src = a.x + (size_t)r0 * a.len + base;
    for (int r = warp; r < nr; r += kWinWarps)
      for (int i = lane; i < n4; i += 32)
        rows[r * pitch + i] = base + i < a.len ? __ldg(src + (size_t)r * a.len + i) : -INFINITY;
  }
  __syncthreads();                                        // (the barrier's initialisation, the -inf, plain rows)
  const bool ok = !bulk || stage_wait(smem_addr(s_bar), 0, tab.spin_limit, a.err);
  return __all_sync(0xffffffffu, ok) && tile < a.n_tiles;
}

template <int MODE, int FORM, int MAXP>
__global__ void __launch_bounds__(kWinThreads, FORM == kFormFp32 ? 4 : 5) window_pass_kernel(const __grid_constant__ BandTable<MAXP> tab) {
  extern __shared__ __align__(128) float s_x[];
  __shared__ __align__(8) uint64_t s_bar;
  const int lane = threadIdx.x & 31;
  const BandArgs& a = tab.p[find_prob<MAXP, 1>(tab, (int)blockIdx.x)];
  Unit u;
  Tilt<FORM> tilt;
  if (!open_unit(tab, a, s_x, &s_bar, u, [&]() {
        if (a.group != 2) tilt.load(a, a.tile_w, true);
      }))
    return;
  unsigned long long* terms = a.terms + 4 * (blockIdx.x & (kTermSlots - 1));
  const RowView& rv = u.rv;
  if (u.pairs) {
    if ((lane & 15) == 0 && rv.wl > 0) atomicAdd(terms + 1, (unsigned long long)rv.wl * 16);
    exact_pair<MODE>(a, u.row, u.k0, rv.lo, rv.wl, rv.mh, rv.row, rv.vec, u.skip);
    return;
  }
  const int W = __reduce_max_sync(0xffffffffu, rv.wl);
  const bool in_range = !__any_sync(0xffffffffu, u.out_of_range);
  if (in_range && lane == 0 && W > 0)
    atomicAdd(terms + (FORM == kFormFp32 ? 0 : 2), (unsigned long long)W * a.tile_w * 8);
  const bool here = in_range && (rv.staged || W == 0);
  if (here) {
    const float kc = (float)(u.k0 + (a.tile_w >> 1)) + a.shift;
    if (a.tile_w == 32 ? gemm_unit<MODE, FORM, 32, true>(a, u.r0, u.k0, kc, rv, W, tilt, u.skip)
                       : gemm_unit<MODE, FORM, 16, true>(a, u.r0, u.k0, kc, rv, W, tilt, u.skip))
      return;
  }
  other_unit<MODE, FORM>(a, u.r0, u.k0, rv, W, in_range && !here, u.skip, terms);
}

// launch with programmatic dependence on the kernel before it in the stream: its set-up (and
// everything up to grid_wait) overlaps that kernel's end
template <typename K, typename T>
void launch_dependent(K kernel, dim3 grid, int threads, size_t smem, cudaStream_t s, const T& args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, kernel, args);
}

// dynamic shared memory of the window kernel: four -inf, eight rows (within the default 48 KB)
__host__ __device__ inline size_t window_smem(int pitch) { return (size_t)(16 + 8 * pitch) * sizeof(float); }

template <int MODE, int FORM, int MAXP>
void window_launch(cudaStream_t s, const BandTable<MAXP>& t);

}  // namespace fot
