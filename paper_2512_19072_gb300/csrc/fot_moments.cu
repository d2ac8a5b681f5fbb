// The phase step's moments (Eqs. 9-10 in ratio form) with banded passes.
//
// With u/g^2 = e^-S (S the kernel sum of the last u-update) the moments are
//     Dx_jk = e^-S_jk sum_L X_L 2^(R[k][L] - (j - L)^2 c),   Dy_jk = e^-S_jk sum_L E[k][L] 2^(...),
// R[k][L] the row pass's log-sums of psi and E[k][L] the mean of Y_M under the row pass's terms: two
// passes over the same windows as a half-step (plan: fot_band.cu), each with weighted sums beside
// the plain one.  Terms outside a window are below 2^-40 of an output's largest; the weights are
// coordinates, at most the image across, so the bound on what is left out grows by that factor.
//
// The weighted sums are more right-hand sides of the tilted product (fot_window.cuh): X v for the
// weight v, accumulated with the same T, G and step order.  The coordinate is linear in m, so its
// weight is the position in the row's window, p = m - lo: sums of small numbers, and the mean
// position is added to lo at the end.  FP32 operands (TF32 hi + lo), 16-wide tiles; problems or
// units outside the bound take exact sums, one exponential per term and output.
//
// Both passes took dense exact kernels before (two sweeps over every term, one exponential each):
// 340 us per pass at 1024^2 against about 36 and 54 us for plan and sums now.
#include "fot_window.cuh"

namespace fot {

namespace {

enum MomentMode : int { kRowMean = 0, kMoment = 1 };      // row pass (R, E), column pass (Dx, Dy)

// one output: plain sum s0 relative to 2^ref (log2), weighted means p (position) and w
template <int MODE>
__device__ __forceinline__ void moment_output(const BandArgs& a, size_t yi, bool some, float alpha, float rest, int lo,
                                              float p, float w) {
  const float cm = fmaf((float)lo + p, a.coord_step, a.coord0);
  if (MODE == kRowMean) {
    a.y[yi] = some ? alpha + rest : -INFINITY;
    a.y2[yi] = some ? cm : 0.f;
  } else {
    // total weight e^-S sum 2^...: the offset and S cancel first
    const float t = some ? ex2(fmaf(-a.off[yi], kLog2e, alpha) + rest) : 0.f;
    a.y[yi] = some ? cm * t : 0.f;
    a.y2[yi] = some ? w * t : 0.f;
  }
}

// exact sums of 2 rows x 16 outputs
template <int MODE>
__device__ __forceinline__ void exact_moments(const BandArgs& a, int row, int k0, int lo, int wl, int mh, const float* xp,
                                              bool skip) {
  const int o = k0 + (threadIdx.x & 15);
  if (row >= a.n_rows || o >= a.n_out || skip) return;
  const float fo = (float)o + a.shift, sc = a.x_scale, c = a.c;
  const float* wr = MODE == kMoment ? a.w + (size_t)row * a.len : nullptr;
  float off = -INFINITY, s0 = 0.f, s1 = 0.f, s2 = 0.f;
  if (wl > 0) {
    const float dm = fo - (float)mh;
    off = fmaf(-dm * dm, c, xp[mh] * sc);
    for (int pass = 0; pass < 2; ++pass) {
      s0 = s1 = s2 = 0.f;
      float top = -INFINITY;
      for (int p = 0; p < wl; ++p) {
        const float d = fo - (float)(lo + p);
        const float e = fmaf(-d * d, c, xp[lo + p] * sc);
        top = fmaxf(top, e);
        const float v = ex2(e - off);
        s0 += v;
        s1 = fmaf(v, (float)p, s1);
        if (MODE == kMoment) s2 = fmaf(v, wr[lo + p], s2);
      }
      // out of range (s2 as well: its weights are as large as 1 / the pixel pitch): again from the exact
      // maximum
      if (s0 <= 3.4e38f && fabsf(s1) <= 3.4e38f && fabsf(s2) <= 3.4e38f) break;
      off = top;
    }
  }
  const bool some = wl > 0 && (off != -INFINITY || isnan(s0));
  moment_output<MODE>(a, (size_t)o * a.n_rows + row, some, off, log2f(s0), lo, s1 / s0, s2 / s0);
}

template <int MODE>
__device__ __noinline__ void exact_moment_unit(const BandArgs& a, int r0, int k0, RowView rv, bool skip) {
  const int half = (threadIdx.x & 31) >> 4;
  for (int p = 0; p < 4; ++p) {
    const int src = 4 * (2 * p + half);
    const int l = __shfl_sync(0xffffffffu, rv.lo, src), w = __shfl_sync(0xffffffffu, rv.wl, src);
    const int m = __shfl_sync(0xffffffffu, rv.mh, src);
    const float* xr = (const float*)__shfl_sync(0xffffffffu, (unsigned long long)rv.row, src);
    exact_moments<MODE>(a, r0 + 2 * p + half, k0, l, w, m, xr, skip);
  }
}

// the tilted product of 8 rows x 16 outputs with 1 + NV right-hand sides; false as gemm_unit
template <int MODE>
__device__ __forceinline__ bool moment_unit(const BandArgs& a, int r0, int k0, float kc, const RowView& rv, int row, int W,
                                            const Tilt<kFormFp32>& tilt, bool skip) {
  constexpr int NV = MODE == kMoment ? 2 : 1;             // weights: position, then w
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const float c = a.c, sc = a.x_scale;
  const f32x2 sc2 = pack2(sc, sc), nc2 = pack2(-c, -c);
  const float na = rv.wl == 0 ? 0.f : -rv.alpha;
  const f32x2 na2 = pack2(na, na);
  const float* wr = MODE == kMoment ? a.w + (size_t)min(row, a.n_rows - 1) * a.len : nullptr;
  const bool wvec = MODE == kMoment && (a.len & 3) == 0 && (reinterpret_cast<unsigned long long>(a.w) & 15ull) == 0;
  f32x2 D[1 + NV][2];
#pragma unroll
  for (int v = 0; v <= NV; ++v) D[v][0] = D[v][1] = pack2(0.f, 0.f);
  const int S = (W + 15) >> 4;
  int pos = rv.lo + 16 * (S - 1) + 4 * q, left = rv.wl - 16 * (S - 1) - 4 * q;
  const float d0 = kc - (float)pos;
  f32x2 d01 = pack2(d0, d0 - 1.f);
  const f32x2 d16 = pack2(16.f, 16.f);
  auto weights = [&]() {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (MODE == kMoment && left > 0) {
      if (wvec) return __ldg(reinterpret_cast<const float4*>(wr + pos));
      v.x = __ldg(wr + pos);
      if (left > 1) v.y = __ldg(wr + pos + 1);
      if (left > 2) v.z = __ldg(wr + pos + 2);
      if (left > 3) v.w = __ldg(wr + pos + 3);
    }
    return v;
  };
  float4 xn = make_float4(0.f, 0.f, 0.f, 0.f), wn = xn;
  if (S > 0) {
    xn = fetch4(rv.row, pos, left, rv.vec);
    wn = weights();
  }
#pragma unroll 1
  for (int s = S - 1; s >= 0; --s) {
    const float4 xv = xn, wv = wn;
    const float fp = (float)(pos - rv.lo);
    pos -= 16;
    left += 16;
    if (s > 0) {
      xn = fetch4(rv.row, pos, left, rv.vec);
      wn = weights();
    }
    float e[1 + NV][4];
    exponents4(xv, sc2, na2, nc2, d01, e[0]);
    d01 = add2(d01, d16);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      e[0][u] = ex2(e[0][u]);
      e[1][u] = e[0][u] * (fp + (float)u);
      if (NV == 2) e[NV][u] = e[0][u] * (u == 0 ? wv.x : u == 1 ? wv.y : u == 2 ? wv.z : wv.w);
    }
    float P[1 + NV][4];
    uint32_t xh[1 + NV][4], xl[1 + NV][4];
#pragma unroll
    for (int v = 0; v <= NV; ++v)
#pragma unroll
      for (int u = 0; u < 4; ++u) split_tf32(e[v][u], xh[v][u], xl[v][u]);
    // the small products first, then hi * hi (as gemm_unit)
#pragma unroll
    for (int part = 0; part < 3; ++part)
#pragma unroll
      for (int h = 0; h < 2; ++h)
#pragma unroll
        for (int v = 0; v <= NV; ++v)
          mma<kFormFp32>(P[v], (part == 0 ? tilt.lo[0] : tilt.hi[0]) + 4 * h, (part == 1 ? xl[v] : xh[v])[2 * h],
                         (part == 1 ? xl[v] : xh[v])[2 * h + 1], part == 0 && h == 0);
#pragma unroll
    for (int v = 0; v <= NV; ++v) {
      D[v][0] = fma2(D[v][0], tilt.G[0][0], pack2(P[v][0], P[v][1]));
      D[v][1] = fma2(D[v][1], tilt.G[0][1], pack2(P[v][2], P[v][3]));
    }
  }
  const int rA = r0 + 2 * q;
  const float al[2] = {__shfl_sync(0xffffffffu, rv.alpha, 8 * q), __shfl_sync(0xffffffffu, rv.alpha, 8 * q + 4)};
  const int lo[2] = {__shfl_sync(0xffffffffu, rv.lo, 8 * q), __shfl_sync(0xffffffffu, rv.lo, 8 * q + 4)};
  float rest[2][2], mean[2][2], wm[2][2];
  bool bad = false;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const float kap = (float)(8 * i - 8 + g);
    float s[1 + NV][2];
#pragma unroll
    for (int v = 0; v <= NV; ++v) unpack2(D[v][i], s[v][0], s[v][1]);
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float ref = (float)lo[u] - kc;
      rest[i][u] = fmaf(fmaf(2.f * kap, ref, -kap * kap), c, log2f(s[0][u]));
      mean[i][u] = s[1][u] / s[0][u];
      wm[i][u] = NV == 2 ? s[NV][u] / s[0][u] : 0.f;
      bad |= al[u] != -INFINITY && !(isfinite(rest[i][u]) && isfinite(mean[i][u]) && isfinite(wm[i][u]));
    }
  }
  if (__any_sync(0xffffffffu, bad)) return false;
  if (W > kLongWalk) {
    const float err = a.step_err[lane], walk = (float)(rv.mh - rv.lo);   // (as log_sums)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const float w = __shfl_sync(0xffffffffu, walk, 8 * q + 4 * u);
#pragma unroll
      for (int i = 0; i < 2; ++i) rest[i][u] = fmaf(__shfl_sync(0xffffffffu, err, 8 * i + 8 + g), w, rest[i][u]);
    }
  }
  if (skip) return true;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int o = k0 + 8 * i + g;
    if (o >= a.n_out) continue;
#pragma unroll
    for (int u = 0; u < 2; ++u)
      if (rA + u < a.n_rows)
        moment_output<MODE>(a, (size_t)o * a.n_rows + rA + u, al[u] != -INFINITY, al[u], rest[i][u], lo[u], mean[i][u],
                            wm[i][u]);
  }
  return true;
}

template <int MODE>
__global__ void __launch_bounds__(kWinThreads, 4) moment_pass_kernel(const __grid_constant__ BandTable<1> tab) {
  extern __shared__ __align__(128) float s_x[];
  __shared__ __align__(8) uint64_t s_bar;
  const int lane = threadIdx.x & 31;
  const BandArgs& a = tab.p[0];
  Unit u;
  Tilt<kFormFp32> tilt;
  if (!open_unit(tab, a, s_x, &s_bar, a.group == 2, u, [&]() {
        if (a.group != 2) tilt.load(a, 16);
      }))
    return;
  unsigned long long* terms = a.terms + 4 * (blockIdx.x & (kTermSlots - 1));
  const RowView& rv = u.rv;
  if (u.pairs) {
    if ((lane & 15) == 0 && rv.wl > 0) atomicAdd(terms + 1, (unsigned long long)rv.wl * 16);
    exact_moments<MODE>(a, u.row, u.k0, rv.lo, rv.wl, rv.mh, rv.row, u.skip);
    return;
  }
  const int W = __reduce_max_sync(0xffffffffu, rv.wl);
  if (unit_walk(8.f, rv, W, a.c) == 0) {
    if (lane == 0 && W > 0) atomicAdd(terms, (unsigned long long)W * 16 * 8);
    if (moment_unit<MODE>(a, u.r0, u.k0, (float)(u.k0 + 8) + a.shift, rv, u.row, W, tilt, u.skip)) return;
  }
  if ((lane & 3) == 0) atomicAdd(terms + 1, (unsigned long long)rv.wl * 16);
  exact_moment_unit<MODE>(a, u.r0, u.k0, rv, u.skip);
}

template <int MODE>
void moment_pass(fot_ctx* c, BandTable<1>& t) {
  const float reach = 2.f * sqrtf(kCut / t.p[0].c);
  t.p[0].tile_w = 16;
  t.p[0].group = 16.f * (16.f + reach) * t.p[0].c <= 64.f ? 8 : 2;
  t.p[0].wide_span = kWinWarps * 16 + (int)(2.6f * sqrtf(kCut / t.p[0].c));
  plan_pass(c->stream, t);
  launch_dependent(moment_pass_kernel<MODE>, dim3(t.items), kWinThreads, window_smem(t.pitch_max), c->stream, t);
  c->launches += 2;
}

}  // namespace

void moments_band(fot_ctx* c, const float* psi, const float* S, double eps, double dx, float* Dx, float* Dy) {
  const int rows = c->rows, cols = c->cols;
  BandTable<1> t{};
  t.n = 1;
  t.spin_limit = c->spin;
  t.p[0] = band_args(c, psi, rows, cols, eps, (float)(1.4426950408889634 / eps));
  t.p[0].y = c->R;
  t.p[0].y2 = c->R2;
  t.p[0].coord0 = (float)(-(double)(cols / 2) / (cols * dx));
  t.p[0].coord_step = (float)(1.0 / (cols * dx));
  moment_pass<kRowMean>(c, t);
  t.p[0] = band_args(c, c->R, cols, rows, eps, 1.f);
  t.p[0].w = c->R2;
  t.p[0].off = S;
  t.p[0].y = Dx;
  t.p[0].y2 = Dy;
  t.p[0].coord0 = (float)(-(double)(rows / 2) / (rows * dx));
  t.p[0].coord_step = (float)(1.0 / (rows * dx));
  moment_pass<kMoment>(c, t);
}

}  // namespace fot
