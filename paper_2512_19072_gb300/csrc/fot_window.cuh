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
// registers for the whole window, which is walked down to its start or up to its end; the sums D
// become D G + (the step's products), G = 2^(+-32 kap c), and end up referred to the first position
// of the last step walked.  The products start from zero and are added by the CUDA cores: the
// tensor core truncates what it accumulates, and a chain of steps through it added up to 1e-5 of a
// sum.  Two steps per turn of the loop, their products added a turn later, so that the exponentials
// of one turn run while the tensor core works on the last: a long window is one warp's chain (45
// steps at 1024^2 where the mean is 13).
//
// Operands.  kFormSplit: BF16 hi + lo parts, hi*hi + hi*lo + lo*hi (2^-16 relative per product);
// kFormSingle: X in one part, T in both (T is the same in every step of a window, so that its rounding would not
// average out as X's does: with hi*hi alone an update was 1.5 times as far from 64 bits as with the operands of
// a longer table); kFormFp32: TF32 hi + lo parts (2^-21), two m16n8k8 per step and product.
//
// Range.  With kmax = TN/2 and D the farthest window position from mh: a term that matters to
// output kap has X >= 2^-(2 kmax D c) (alpha is e(mh, kc); the largest term at kap is at least
// mh's), and referring the sum to position r instead of mh moves it by at most 2 kmax |mh - r| c.  A
// row is in range while the first is <= kTiltMax and both together are <= kRangeMax: what flushes
// to zero below 2^-126 is then less than W 2^-30 of a sum, and sums stay below 2^(100 + 9) times
// 2^(how far the offset lies below the maximum).  The walk ends at the start of the window where
// every row is in range that way, else at its end (mh sits at one end of most windows that span a
// gap).  An offset that lies too far below the maximum shows as an output that is not finite; such a
// unit is summed again in segments.
//
// Small eps.  The range shrinks with the tile: where eps is too small for 16 outputs (below about 12) every
// output is summed exactly, one exponential per term, relative to e(mh, o), plan and sums in one kernel
// (fot_small.cuh): the windows are a few blocks long.  Products of 8-wide tiles, with half of T's rows
// zero, were slower (us per pass, FP32, eps 7 / 11: 256^2 9.6 / 8.0 against 6.8 / 6.0 exact, 1024^2 46 / 44 against
// 32 / 33) and twice as far from 64 bits (log-sums at eps 8: 2.5e-7 and 1.1e-7 rms).
//
// Segments.  A unit outside the bound (a window that spans the gap between two parts of a target,
// mostly) is summed with FP32 operands in segments of its window short enough to be in range by
// themselves, each with its rows' maxima as offsets; the segments' sums are added as logarithms, and a segment in
// which no row has a term within 2^-kCut of its output's largest is passed over.  (Exact sums for
// these units, one in twenty, made a pass at 256^2 and eps 15 three times as long: 18.6 us, 13.4 with
// segments.)  What fails even then is summed exactly.
//
// What bounds it: issue slots and latency.  A split-BF16 step at TN = 32 is about 40 instructions
// and 6 MMAs (48 tensor cycles per SM quarter), a unit's set-up and outputs about 450.  A loop of
// 200 iterations at 1024^2 (800 passes, plan and launch gaps included) went from 31.9 to 14.5 ms with
// split BF16 and from 45.7 to 16.5 ms with FP32 operands (FFMA with the operands through shared memory
// before; 17.2 with the operands' parts rounded); 100 iterations at 2048^2, split BF16, from 39.8 to 21.2 ms (21.9 with
// the step scale's rounding made up for); 256^2 annealed from eps 64 to 1 over 300 iterations from 41.7 to 11.7
// ms (8.6 with the one-kernel passes of fot_small.cuh); 64^2 at eps 1, 200 iterations, from 14.5 to 4.6 ms (2.7).
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
                                          // (2048^2, split BF16, a half-step: eps 6000, most
                                          // items staged, 172 us, eps 7000, none, 180)
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
// TF32 hi and lo parts, hi rounded to nearest.  The tensor core reads the upper 19 bits of each and cuts the
// rest off: with hi cut as well, lo and what is lost of it are never negative, and neither is lo * lo,
// which the three products leave out: 2^-21 on average and all one way (log-sums were 3e-7 per pass too
// low).  Rounded, lo has either sign and at most 12 bits, of which 11 are read: 2^-23 is lost.  (A NaN
// stays one in lo.)
__device__ __forceinline__ void split_tf32(float a, uint32_t& hi, uint32_t& lo) {
  hi = (__float_as_uint(a) + 0x1000u) & 0xffffe000u;
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

// 4-byte asynchronous copies for rows that are not 16-byte aligned: as many in flight as a thread has
// (plain loads went a few at a time: a pair of half-steps at 257x201 41.8 us, 36.4 with these; 30 iterations
// between 300x257 and 385x212 1.09 and 0.88 ms)
__device__ __forceinline__ void async_load4(uint32_t dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" :: "r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void async_loads_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }
// n values of each of nr rows (src, stride len) to dst (pitch floats, shared), -inf up to the next multiple
// of 4; thread i of count (a power of two, at least a warp).  Complete after async_loads_done and a barrier.
__device__ __forceinline__ void stage_unaligned(float* dst, int pitch, const float* src, int len, int n, int nr, int i, int count) {
  const int n4 = (n + 3) & ~3;
  for (int r = i >> 5; r < nr; r += count >> 5) {
    const uint32_t to = smem_addr(dst + r * pitch);
    const float* const from = src + (size_t)r * len;
    for (int k = i & 31; k < n; k += 32) async_load4(to + 4u * k, from + k);
    if ((i & 31) < n4 - n) dst[r * pitch + n + (i & 31)] = -INFINITY;
  }
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
  // tw: outputs of the tile (16: first row tile only); BF16 forms take a.tilt's fragments
  __device__ __forceinline__ void load(const BandArgs& a, int tw) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      if (16 * t >= tw) break;
      const int kap0 = 16 * t - tw / 2;
      if (FORM == kFormFp32) {
#pragma unroll
        for (int h = 0; h < NH; ++h) {
          tilt_fragments_tf32(a.c, kap0, h, lane, hi[t] + 4 * h, lo[t] + 4 * h);
        }
      } else {
        const uint4 h4 = __ldg(a.tilt + t * 64 + lane), l4 = __ldg(a.tilt + t * 64 + 32 + lane);
        hi[t][0] = h4.x; hi[t][1] = h4.y; hi[t][2] = h4.z; hi[t][3] = h4.w;
        lo[t][0] = l4.x; lo[t][1] = l4.y; lo[t][2] = l4.z; lo[t][3] = l4.w;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float v = a.step[kap0 + (lane >> 2) + 8 * h + 16];
        G[t][h] = pack2(v, v);
      }
    }
  }
};

// The window sums D of one unit (see the top), referred to each row's lo (up: to the first position
// of the last step, lo + walk_end(W)).  Lane (g = lane / 4, q = lane % 4) owns row g of the unit (rv)
// for X, and outputs kap g and g + 8 of each row tile of columns 2q, 2q + 1.
// So much longer than a smooth potential's (about 210) that it is likely to span a gap.  (us per pass, split
// BF16, line at 450 / 900 / 1800: 1024^2 eps 209 19.3 / 18.7 / 18.1, 2048^2 eps 839 58.4 / 56.7 / 56.6, 576^2 eps 60
// 14.8 / 14.7 / 13.5: a little high does no harm.)
__device__ __forceinline__ bool long_window(int W, float c) { return (float)W * (float)W * c > 900.f; }
__device__ __forceinline__ int walk_end(int W) { return ((W + 31) >> 5) * 32 - 16; }
// PLAIN: the common case, rows staged, walking down, no look for empty turns (fewer registers).
template <int FORM, int TN, bool PLAIN>
__device__ __forceinline__ void window_product(const BandArgs& a, float kc, const RowView& rv, int W, bool up_,
                                               const Tilt<FORM>& tilt, f32x2 (&D)[TN / 16][2]) {
  constexpr int MT = TN / 16;
  constexpr int NH = Tilt<FORM>::NH;
  const int q = threadIdx.x & 3;
  const float c = a.c;
  const float sc = a.x_scale;
  const f32x2 sc2 = pack2(sc, sc), nc2 = pack2(-c, -c);
  const float na = rv.wl == 0 ? 0.f : -rv.alpha;
  const f32x2 na2 = pack2(na, na);
  float P[2][MT][4];                                      // the last turn's products
#pragma unroll
  for (int t = 0; t < MT; ++t) {
    D[t][0] = D[t][1] = pack2(0.f, 0.f);
#pragma unroll
    for (int u = 0; u < 4; ++u) P[0][t][u] = P[1][t][u] = 0.f;
  }
  const bool up = !PLAIN && up_;
  const int turns = (W + 31) >> 5;
  const int first = up ? 0 : walk_end(W), by = up ? 16 : -16;
  int pos = rv.lo + first + 4 * q;                        // this lane's first position of the step
  int left = rv.wl - first - 4 * q;                       // of it and after it in the window
  uint32_t addr = rv.saddr + 4u * (uint32_t)pos;
  const float d0 = kc - (float)pos;
  f32x2 d01 = pack2(d0, d0 - 1.f);
  const f32x2 d16 = pack2((float)-by, (float)-by);
  f32x2 G[MT][2];
#pragma unroll
  for (int t = 0; t < MT; ++t)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      G[t][h] = tilt.G[t][h];
      if (up) {
        const float v = a.step[16 - (16 * t - TN / 2 + (int)((threadIdx.x & 31) >> 2) + 8 * h)];
        G[t][h] = pack2(v, v);
      }
    }
  const bool gaps = !PLAIN && long_window(W, c);
  auto fetch = [&]() {
    float4 v;
    if (PLAIN)
      v = lds4(left > 0 ? addr : rv.minf);
    else
      v = fetch4(rv.row, pos, left, rv.vec);
    addr += (uint32_t)(4 * by);
    pos += by;
    left -= by;
    return v;
  };
  auto absorb = [&]() {                                   // D <- (D G + P0) G + P1
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int t = 0; t < MT; ++t) {
        D[t][0] = fma2(D[t][0], G[t][0], pack2(P[i][t][0], P[i][t][1]));
        D[t][1] = fma2(D[t][1], G[t][1], pack2(P[i][t][2], P[i][t][3]));
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
    float e[2][4];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      exponents4(xv[v], sc2, na2, nc2, d01, e[v]);
      d01 = add2(d01, d16);
    }
    if (gaps) {
      // a turn whose operands are all zero (ex2 flushes below 2^-126).  As unsigned words, the
      // numbers below -126 are those above its own (a NaN of the arithmetic, 0x7fffffff, is not:
      // it takes the products)
      uint32_t least = 0xffffffffu;
#pragma unroll
      for (int v = 0; v < 2; ++v)
#pragma unroll
        for (int u = 0; u < 4; ++u) least = min(least, __float_as_uint(e[v][u]));
      if (__all_sync(0xffffffffu, least > 0xc2fc0000u)) {
        absorb();
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int t = 0; t < MT; ++t)
#pragma unroll
            for (int u = 0; u < 4; ++u) P[v][t][u] = 0.f;
        continue;
      }
    }
    uint32_t xh[2][2 * NH], xl[2][2 * NH];
#pragma unroll
    for (int v = 0; v < 2; ++v) {
#pragma unroll
      for (int u = 0; u < 4; ++u) e[v][u] = ex2(e[v][u]);
      if (FORM == kFormFp32) {
#pragma unroll
        for (int u = 0; u < 4; ++u) split_tf32(e[v][u], xh[v][u % (2 * NH)], xl[v][u % (2 * NH)]);
      } else {
        split_bf16(e[v][0], e[v][1], xh[v][0], xl[v][0]);
        split_bf16(e[v][2], e[v][3], xh[v][1], xl[v][1]);
      }
    }
    absorb();
    // the small products first, then hi * hi
#pragma unroll
    for (int part = 0; part < 3; part += FORM == kFormSingle ? 2 : 1)
#pragma unroll
      for (int h = 0; h < NH; ++h)
#pragma unroll
        for (int v = 0; v < 2; ++v)
#pragma unroll
          for (int t = 0; t < MT; ++t) {
            const uint32_t* A = (part == 0 ? tilt.lo[t] : tilt.hi[t]) + 4 * h;
            const uint32_t* Bm = (part == 1 ? xl[v] : xh[v]) + (NH == 2 ? 2 * h : 0);
            const bool first = part == 0 && h == 0;
            mma<FORM>(P[v][t], A, Bm[0], Bm[1], first);
          }
  }
  absorb();
}

// Outputs of a unit: the log-sum of output group i (kap = 8 i - TN/2 + g) and column u is
// al[u] + t[i][u].  False, with nothing written, when one is not finite where its row has mass
// (warp-uniform).
template <int MODE, int TN>
__device__ __forceinline__ bool write_unit(const BandArgs& a, int r0, int k0, const float (&al)[TN / 8][2],
                                           const float (&t)[TN / 8][2], bool skip) {
  constexpr int NO = TN / 8;                // groups of 8 outputs
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const int rA = r0 + 2 * q;
  const size_t y0 = (size_t)(k0 + g) * a.n_rows + rA;
  const size_t ystep = (size_t)8 * a.n_rows;
  const bool full = (a.vec & 2) && k0 + TN <= a.n_out && r0 + 8 <= a.n_rows;   // warp-uniform
  auto inside = [&](int i) { return k0 + g + 8 * i < a.n_out; };
  float lm[NO][2];
  if (MODE == 1) {
#pragma unroll
    for (int i = 0; i < NO; ++i) {
      const float* p = a.lmarg + y0 + i * ystep;
      if (full) {
        const float2 v = __ldg(reinterpret_cast<const float2*>(p));
        lm[i][0] = v.x;
        lm[i][1] = v.y;
      } else {
        const bool in = inside(i);
        lm[i][0] = in && rA < a.n_rows ? __ldg(p) : -INFINITY;
        lm[i][1] = in && rA + 1 < a.n_rows ? __ldg(p + 1) : -INFINITY;
      }
    }
  }
  float s2[NO][2], chk[2] = {0.f, 0.f};                   // chk: NaN after a non-finite log-sum
#pragma unroll
  for (int i = 0; i < NO; ++i)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      s2[i][u] = __fadd_rn(al[i][u], t[i][u]);
      chk[u] = fmaf(s2[i][u], 0.f, chk[u]);
    }
  if (__any_sync(0xffffffffu, (chk[0] != 0.f && al[0][0] != -INFINITY) || (chk[1] != 0.f && al[0][1] != -INFINITY)))
    return false;
  if (skip) return true;
  bool bad = false;
#pragma unroll
  for (int i = 0; i < NO; ++i) {
    float out[2], sv[2];
#pragma unroll
    for (int u = 0; u < 2; ++u) out[u] = finish_output<MODE>(a, s2[i][u], MODE == 1 ? lm[i][u] : 0.f, sv[u], bad);
    const size_t yi = y0 + i * ystep;
    if (full) {
      *reinterpret_cast<float2*>(a.y + yi) = make_float2(out[0], out[1]);
      if (MODE == 1 && a.logsum) *reinterpret_cast<float2*>(a.logsum + yi) = make_float2(sv[0], sv[1]);
    } else if (inside(i)) {
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

// Windows from which on outputs get back what the rounding of the step scale G took from their sums: up to
// 2^-25 per step (a.step_err, log2 per position), over the steps between the reference and the row's largest
// term.  Below, it is no more than the FP32 error of the rest (log-sums at 1500 x 1400, FP32 form, rms: eps 369
// 4.7e-7 without and 3.2e-7 with it; eps 5900 1.4e-6 and 3.8e-7), and a solve at 1024^2 and eps 209 takes
// longer with it (with a lane's entries read from the constant bank one by one, 5 %; 100 iterations at 2048^2,
// split BF16, 20.9 ms without, 21.9 that way, 21.1 with one read and shuffles).
constexpr int kLongWalk = 320;

// log-sums of the sums D (referred to lo, or up: lo + walk_end(W)): offset and rest of every output
template <int FORM, int TN>
__device__ __forceinline__ void log_sums(const BandArgs& a, float kc, const RowView& rv, int W, bool up,
                                         const f32x2 (&D)[TN / 16][2], float (&al)[TN / 8][2],
                                         float (&t)[TN / 8][2]) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const float alpha = __shfl_sync(0xffffffffu, rv.alpha, 8 * q + 4 * u);
    const int at = __shfl_sync(0xffffffffu, rv.lo, 8 * q + 4 * u) + (up ? walk_end(W) : 0);
    const float mr = (float)at - kc;                      // reference - kc
#pragma unroll
    for (int i = 0; i < TN / 8; ++i) {
      const float kap = (float)(8 * i - TN / 2 + g);
      float v[2];
      unpack2(D[i >> 1][i & 1], v[0], v[1]);
      const float l2 = FORM == kFormFp32 ? log2f(v[u]) : lg2(v[u]);
      al[i][u] = alpha;
      t[i][u] = fmaf(fmaf(2.f * kap, mr, -kap * kap), a.c, l2);
    }
  }
  if (W > kLongWalk) {
    // each lane reads one entry (the constant bank answers one address at a time), shuffles bring the others
    const float err = a.step_err[up ? 32 - lane : lane];  // of kap = lane - 16
    const float walk = up ? (float)(rv.lo + walk_end(W) - rv.mh) : (float)(rv.mh - rv.lo);
    const float w0 = __shfl_sync(0xffffffffu, walk, 8 * q), w1 = __shfl_sync(0xffffffffu, walk, 8 * q + 4);
#pragma unroll
    for (int i = 0; i < TN / 8; ++i) {
      const float e = __shfl_sync(0xffffffffu, err, 8 * i + g + 16 - TN / 2);
      t[i][0] = fmaf(e, w0, t[i][0]);
      t[i][1] = fmaf(e, w1, t[i][1]);
    }
  }
}

// One unit by the tilted product.  False, with nothing written, when a sum left the range of FP32
// (warp-uniform).
template <int MODE, int FORM, int TN, bool PLAIN>
__device__ __forceinline__ bool gemm_unit(const BandArgs& a, int r0, int k0, float kc, const RowView& rv, int W, bool up,
                                          const Tilt<FORM>& tilt, bool skip) {
  f32x2 D[TN / 16][2];
  window_product<FORM, TN, PLAIN>(a, kc, rv, W, up, tilt, D);
  float al[TN / 8][2], t[TN / 8][2];   // (an empty row has sums 0: log -inf)
  log_sums<FORM, TN>(a, kc, rv, W, !PLAIN && up, D, al, t);
  return write_unit<MODE, TN>(a, r0, k0, al, t, skip);
}

// Exact window sum of one lane's output o of `row`, window [lo, lo + wl), xp[m] that row's position
// m.  Terms are taken relative to e(mh, o), which is within the range of FP32 of the maximum unless
// the maximum moves far from mh within the tile, or exponents are so large (beyond 2^30) that their
// rounding alone is; a sum out of range is done again from its exact maximum, and should that fail,
// of terms rounded as the maximum is.
template <int MODE>
__device__ __forceinline__ void exact_output(const BandArgs& a, int row, int o, int lo, int wl, int mh, const float* xp,
                                             bool vec, bool skip) {
  const float fo = (float)o + a.shift, sc = a.x_scale, nc = -a.c;
  float out = -INFINITY;
  if (wl > 0) {
    const float dm = fo - (float)mh;
    float off = fmaf(dm * dm, nc, xp[mh] * sc);
    const f32x2 sc2 = pack2(sc, sc), nc2 = pack2(nc, nc), dn4 = pack2(-4.f, -4.f);
    const float d0 = fo - (float)lo;
    float s0, s1;
    auto in_range = [&]() { return s0 + s1 >= 1e-24f && s0 + s1 <= 3.4e38f; };   // (a NaN is not, and stays one)
    for (int pass = 0; pass < 2; ++pass) {
      const f32x2 no2 = pack2(-off, -off);
      f32x2 d01 = pack2(d0, d0 - 1.f);
      s0 = s1 = 0.f;
#pragma unroll 2
      for (int p = 0; p < wl; p += 4) {
        float e[4];
        exponents4(fetch4(xp, lo + p, wl - p, vec), sc2, no2, nc2, d01, e);
        d01 = add2(d01, dn4);
        s0 += ex2(e[0]) + ex2(e[1]);
        s1 += ex2(e[2]) + ex2(e[3]);
      }
      if (in_range()) break;
      // its exact maximum; then (the second time) terms rounded as that is
      if (pass == 0) off = -INFINITY;
      s0 = s1 = 0.f;
      d01 = pack2(d0, d0 - 1.f);
      for (int p = 0; p < wl; p += 4) {
        float e[4];
        exponents4(fetch4(xp, lo + p, wl - p, vec), sc2, pack2(0.f, 0.f), nc2, d01, e);
        d01 = add2(d01, dn4);
        if (pass == 0) {
          off = fmaxf(fmaxf(off, fmaxf(e[0], e[1])), fmaxf(e[2], e[3]));
        } else {
          s0 += ex2(e[0] - off) + ex2(e[1] - off);
          s1 += ex2(e[2] - off) + ex2(e[3] - off);
        }
      }
    }
    out = __fadd_rn(off, log2f(s0 + s1));
  }
  if (row >= a.n_rows || o >= a.n_out || skip) return;
  const size_t yi = (size_t)o * a.n_rows + row;
  float s = 0.f;
  bool bad = false;
  a.y[yi] = finish_output<MODE>(a, out, MODE == 1 ? __ldg(a.lmarg + yi) : 0.f, s, bad);
  if (MODE == 1 && a.logsum) a.logsum[yi] = s;
  if (bad) raise_error(a.err, FOT_ENONFINITE);
}

// How a unit's rows stay in range of the tilted product (the top): 0 walking down, 1 walking up,
// 2 not at all (warp-uniform)
__device__ __forceinline__ int unit_walk(float kmax, const RowView& rv, int W, float c) {
  const float t = 2.f * kmax * c, far = t * (float)max(rv.mh - rv.lo, rv.lo + rv.wl - rv.mh);
  const bool none = rv.wl == 0, in = far <= kTiltMax;
  if (__all_sync(0xffffffffu, none || (in && far + t * (float)(rv.mh - rv.lo) <= kRangeMax))) return 0;
  return __all_sync(0xffffffffu, none || (in && far + t * (float)abs(rv.lo + walk_end(W) - rv.mh) <= kRangeMax)) ? 1 : 2;
}

// every row's exact maximum over its window at centre kc, and where it is reached
__device__ __forceinline__ RowView recentred(const BandArgs& a, const RowView& rv, float kc) {
  const int q = threadIdx.x & 3;
  const float c = a.c, sc = a.x_scale;
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
  return r;
}

// A unit outside the bound, in segments of its window (the top).  False, with nothing written, when
// it cannot be done that way (warp-uniform).
template <int MODE, int TN>
__device__ __noinline__ bool segmented_unit(const BandArgs& a, int r0, int k0, const RowView& rv, int W, bool skip,
                                            unsigned long long* terms) {
  constexpr int NO = TN / 8;
  const float kc = (float)(k0 + TN / 2) + a.shift, c = a.c;
  const int L = min((int)(kRangeMax / (2.f * TN * c)) & ~15, 4096);   // TN (D + mh - lo) c <= TN 2 L c
  if (L < 16 || __any_sync(0xffffffffu, isnan(rv.alpha))) return false;   // (a row for exact sums: fot_plan.cuh)
  Tilt<kFormFp32> tilt;
  tilt.load(a, TN);
  float A[NO][2], T[NO][2];                               // the sums so far: offset and rest
#pragma unroll
  for (int i = 0; i < NO; ++i)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      A[i][u] = -INFINITY;
      T[i][u] = 0.f;
    }
  for (int s0 = 0; s0 < W; s0 += L) {
    RowView r = rv;
    r.lo = rv.lo + s0;
    r.wl = max(0, min(rv.wl - s0, L));
    r = recentred(a, r, kc);
    if (r.alpha == -INFINITY) r.wl = 0;
    // against mh's term, a term m of the segment gains at most TN |m - mh| c at the tile's ends
    const float gain = (float)TN * c * (float)max(abs(r.lo - rv.mh), abs(r.lo + r.wl - rv.mh));
    if (!__any_sync(0xffffffffu, r.wl > 0 && r.alpha + gain >= rv.alpha - kCut)) continue;
    const int Ws = __reduce_max_sync(0xffffffffu, r.wl);
    if ((threadIdx.x & 31) == 0) atomicAdd(terms, (unsigned long long)Ws * TN * 8);
    f32x2 D[TN / 16][2];
    window_product<kFormFp32, TN, false>(a, kc, r, Ws, false, tilt, D);
    float al[NO][2], t[NO][2];
    log_sums<kFormFp32, TN>(a, kc, r, Ws, false, D, al, t);
#pragma unroll
    for (int i = 0; i < NO; ++i)
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        // (A, T) <- log2(2^(A + T) + 2^(al + t)); the offsets are subtracted first
        if (al[i][u] == -INFINITY) continue;
        const float d = (al[i][u] - A[i][u]) + (t[i][u] - T[i][u]);
        const bool up = !(d < 0.f);                       // the new one is the larger (or the first)
        const float more = log2f(1.f + ex2(up ? -d : d));
        A[i][u] = up ? al[i][u] : A[i][u];
        T[i][u] = (up ? t[i][u] : T[i][u]) + more;
      }
  }
  return write_unit<MODE, TN>(a, r0, k0, A, T, skip);
}

// a unit that is not the common case: rows not staged, a long window, walking up,
// outside the bound or with sums that left the range of FP32 (walk 2: no product)
template <int MODE, int FORM, int TN>
__device__ __forceinline__ void other_unit_of(const BandArgs& a, int r0, int k0, const RowView& rv, int W, int walk,
                                              bool skip, unsigned long long* terms) {
  if (walk != 2) {
    Tilt<FORM> tilt;
    tilt.load(a, TN);
    if (gemm_unit<MODE, FORM, TN, false>(a, r0, k0, (float)(k0 + TN / 2) + a.shift, rv, W, walk == 1, tilt, skip)) return;
  }
  if (segmented_unit<MODE, TN>(a, r0, k0, rv, W, skip, terms)) return;
  const int lane = threadIdx.x & 31;
  if ((lane & 3) == 0) atomicAdd(terms + 1, (unsigned long long)rv.wl * TN);
  for (int k = k0; k < k0 + TN; k += 4)
    exact_output<MODE>(a, r0 + (lane >> 2), k + (lane & 3), rv.lo, rv.wl, rv.mh, rv.row, rv.vec, skip);
}
template <int MODE, int FORM>
__device__ __noinline__ void other_unit(const BandArgs& a, int r0, int k0, RowView rv, int W, int walk, bool skip,
                                        unsigned long long* terms) {
  if (a.tile_w == 32)
    other_unit_of<MODE, FORM, 32>(a, r0, k0, rv, W, walk, skip, terms);
  else
    other_unit_of<MODE, FORM, 16>(a, r0, k0, rv, W, walk, skip, terms);
}

// A warp's unit of the item that its CTA was launched for.
struct Unit {
  RowView rv;
  int r0, k0, row;                                        // first row and output, this lane's row
  bool pairs, skip;
};

// The sums of a unit, once its rows are staged: 2 rows x 16 exact outputs, or a product of 8 rows
// (tilt is loaded for tiles of 16 and 32).
template <int MODE>
__device__ __forceinline__ void exact_unit(const BandArgs& a, const Unit& u, unsigned long long* terms) {
  const int lane = threadIdx.x & 31;
  const RowView& rv = u.rv;
  if ((lane & 15) == 0 && rv.wl > 0) atomicAdd(terms + 1, (unsigned long long)rv.wl * 16);
  exact_output<MODE>(a, u.row, u.k0 + (lane & 15), rv.lo, rv.wl, rv.mh, rv.row, rv.vec, u.skip);
}
template <int MODE, int FORM>
__device__ __forceinline__ void product_unit(const BandArgs& a, const Unit& u, const Tilt<FORM>& tilt, unsigned long long* terms) {
  const int lane = threadIdx.x & 31;
  const RowView& rv = u.rv;
  const int W = __reduce_max_sync(0xffffffffu, rv.wl);
  const int walk = unit_walk(0.5f * (float)a.tile_w, rv, W, a.c);
  if (walk != 2 && lane == 0 && W > 0)
    atomicAdd(terms + (FORM == kFormFp32 ? 0 : 2), (unsigned long long)W * a.tile_w * 8);
  const bool plain = walk == 0 && (rv.staged || W == 0) && !long_window(W, a.c);
  if (plain) {
    const float kc = (float)(u.k0 + (a.tile_w >> 1)) + a.shift;
    if (a.tile_w == 32 ? gemm_unit<MODE, FORM, 32, true>(a, u.r0, u.k0, kc, rv, W, false, tilt, u.skip)
                       : gemm_unit<MODE, FORM, 16, true>(a, u.r0, u.k0, kc, rv, W, false, tilt, u.skip))
      return;
  }
  other_unit<MODE, FORM>(a, u.r0, u.k0, rv, W, plain ? 2 : walk, u.skip, terms);
}

// The start of a window CTA: read the item and this warp's plan entries, stage the rows; `meanwhile`
// runs while they are on their way.  s_x: four -inf (padded to 64 bytes), then the rows.  False: the
// warp has nothing to do.
template <int MAXP, typename F>
__device__ __forceinline__ bool open_unit(const BandTable<MAXP>& tab, const BandArgs& a, float* s_x, uint64_t* s_bar, bool pairs,
                                          Unit& u, F meanwhile) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  u.pairs = pairs;
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
  rv.mh = w2;
  rv.staged = staged;
  rv.vec = staged || (a.vec & 1);
  rv.row = staged ? rows + lr * pitch - base : a.x + (size_t)min(u.row, a.n_rows - 1) * a.len;
  rv.saddr = smem_addr(rows + lr * pitch) - 4u * (uint32_t)base;
  rv.minf = smem_addr(s_x);
  if (staged && !bulk) {
    // (top may be the row's end: what lies past it is -inf)
    stage_unaligned(rows, pitch, a.x + (size_t)r0 * a.len + base, a.len, min(top, a.len) - base, nr, tid, kWinThreads);
    async_loads_done();
  }
  __syncthreads();                                        // (the barrier's initialisation, the -inf, plain rows)
  const bool ok = !bulk || stage_wait(smem_addr(s_bar), 0, tab.spin_limit, a.err);
  return __all_sync(0xffffffffu, ok) && tile < a.n_tiles;
}

template <int MODE, int FORM, int MAXP>
__global__ void __launch_bounds__(kWinThreads, FORM == kFormFp32 ? 4 : 5) window_pass_kernel(const __grid_constant__ BandTable<MAXP> tab) {
  extern __shared__ __align__(128) float s_x[];
  __shared__ __align__(8) uint64_t s_bar;
  const BandArgs& a = tab.p[find_prob<MAXP, 1>(tab, (int)blockIdx.x)];
  Unit u;
  Tilt<FORM> tilt;
  const bool pairs = MAXP > 2 && a.group == 2;            // (a batch with problems of both kinds)
  if (!open_unit(tab, a, s_x, &s_bar, pairs, u, [&]() {
        if (!pairs) tilt.load(a, a.tile_w);
      }))
    return;
  unsigned long long* terms = a.terms + 4 * (blockIdx.x & (kTermSlots - 1));
  if (u.pairs)
    exact_unit<MODE>(a, u, terms);
  else
    product_unit<MODE, FORM>(a, u, tilt, terms);
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

// one-kernel passes (fot_small.cuh): products of one operand form, exact sums and their dynamic shared
// memory limit
template <int MODE, int FORM, int MAXP>
void small_launch(cudaStream_t s, const BandTable<MAXP>& t);
template <int MODE, int MAXP>
void small_exact_launch(cudaStream_t s, const BandTable<MAXP>& t);
cudaError_t small_exact_configure(int bytes);

}  // namespace fot
