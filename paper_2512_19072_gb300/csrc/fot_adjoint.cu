// Adjoint (reverse mode) of the FOT solve: gradients of a scalar loss of the phase and/or the
// final potentials with respect to the input and target amplitudes g and G, through every
// unrolled iteration (Eqs. 7-8), the moments (Eqs. 9-10), the trapezoid integration and the
// marginal normalisation a = g^2 / sum g^2, b = G^2 / sum G^2.
//
// Half-step VJPs.  f = eps (log a - S(psi)), S_jk = log sum_LM exp(psi_LM/eps - C_jkLM/eps):
//     dL/dlog a += eps fbar,   psibar_LM -= sum_jk fbar_jk exp(psi_LM/eps - C/eps - S_jk),
// and likewise for psi = eps (log b - T(f)).  The sum is a Gaussian-kernel application to
// the signed weights z_jk = fbar_jk e^{-S_jk}; it is evaluated in the log domain by the same
// separable axis passes as the forward solve, once on the positive and once on the negative
// part:  sum_jk z e^{-C/eps} = e^{L+} - e^{L-},  L+- = log(Lambda e^{log z+-} Lambda).
//
// Moments: with W_jk,LM = exp((f_jk + psi_LM - C)/eps - log a_jk) (the plan over g^2),
// Dx_jk = sum_LM X_L W, Dy_jk = sum_LM Y_M W, so
//     psibar_LM += (1/eps) e^{psi_LM/eps} [X_L K(Dxbar e^{-S}) + Y_M K(Dybar e^{-S})]_LM,
//     fbar_jk += (Dxbar Dx + Dybar Dy)_jk / eps,   dL/dlog a_jk -= (Dxbar Dx + Dybar Dy)_jk.
// Trapezoid: the transpose of the linear integration map (suffix / prefix sums).
// Normalisation: log a = 2 log g - log sum g^2, so dL/dg = 2 (abar - a sum abar) / g (0 where
// g = 0), abar = dL/dlog a.
//
// Memory: the forward is recomputed from potentials checkpointed every k iterations; one
// segment of k iterations (psi_t, S_t, f_t+1, T_t) is held at a time (the last one is kept as the
// forward runs through it).
//
// At 256^2 a step is a few microseconds of latency whatever it does, so the number of launches
// decides: the applications to z+ and z- are one two-problem pass each, and everything
// elementwise between two applications is one kernel (vjp_step_kernel): 10 launches per iteration
// of the reverse sweep instead of 24, 6 where passes are one kernel.  A training step at 256^2 with 30
// iterations went from 8.5 to 5.4 ms with two-kernel passes, and is 4.3 ms with one-kernel ones.
#include <math.h>

#include "fot_band.cuh"

namespace fot {
void half_step_dispatch(fot_ctx* c, const float* pot_in, const float* lmarg, double eps, float* pot_out,
                        float* logsum);
void half_step_simt(fot_ctx* c, const float* pot_in, const float* lmarg, double eps,
                    float* pot_out, float* logsum, float* tmp);
void moments(fot_ctx* c, const float* psi, const float* S, double eps, double dx, float* Dx, float* Dy);
void set_problem_simt(fot_ctx* c, const float* g, const float* G, float* psi0, float psi0_val);
void fill(fot_ctx* c, float* p, size_t N, float v);
}  // namespace fot

using namespace fot;

namespace {

// log-domain parts of a signed weight v: pos = eps (log v+ - off), neg = eps (log v- - off); -inf
// where that part is zero
__device__ __forceinline__ void split_value(float v, float o, float eps, float& pos, float& neg) {
  const bool fin = isfinite(o);
  pos = (v > 0.f && fin) ? eps * (logf(v) - o) : -INFINITY;
  neg = (v < 0.f && fin) ? eps * (logf(-v) - o) : -INFINITY;
}

__global__ void split_kernel(const float* __restrict__ z, const float* __restrict__ off, float eps, size_t N,
                             float* __restrict__ pos, float* __restrict__ neg) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x)
    split_value(z[i], off[i], eps, pos[i], neg[i]);
}

// Between two applications of the reverse sweep.  v = prev - (e^{base/ep + Lp} - e^{base/ep + Ln})
// (base = null: v = prev; base = -inf contributes 0; prev = null: 0) is the adjoint that the last
// application gives.  Then, each when asked for: acc += e v (dL/dlog marginal), the split of v
// against off at e for the next application, v itself.
__global__ void vjp_step_kernel(const float* __restrict__ prev, const float* __restrict__ base, float inv_ep,
                                const float* __restrict__ Lp, const float* __restrict__ Ln, float e,
                                float* __restrict__ acc, const float* __restrict__ off, float* __restrict__ pos,
                                float* __restrict__ neg, float* __restrict__ v_out, size_t N) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    float v = prev ? prev[i] : 0.f;
    if (base) {
      const float b = base[i];
      if (b != -INFINITY) {
        const float x = b * inv_ep, lp = Lp[i], ln = Ln[i];
        v -= (lp == -INFINITY ? 0.f : expf(x + lp)) - (ln == -INFINITY ? 0.f : expf(x + ln));
      }
    }
    if (acc) acc[i] += e * v;
    if (pos) split_value(v, off[i], e, pos[i], neg[i]);
    if (v_out) v_out[i] = v;
  }
}

__global__ void axpy_kernel(float* __restrict__ y, const float* __restrict__ x, float s, size_t N) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x)
    y[i] += s * x[i];
}

// moments VJP, elementwise part: fbar += (Dxbar Dx + Dybar Dy)/eps; abar -= (Dxbar Dx +
// Dybar Dy).  (The kernel applications to Dxbar e^{-S}, Dybar e^{-S} take S as the log
// offset of split_kernel: e^{-S} alone overflows FP32 where S is very negative.)
__global__ void moments_vjp_pre(const float* __restrict__ Dxb, const float* __restrict__ Dyb,
                                const float* __restrict__ Dx, const float* __restrict__ Dy, float inv_eps,
                                size_t N, float* __restrict__ fbar, float* __restrict__ abar) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    const float d = Dxb[i] * Dx[i] + Dyb[i] * Dy[i];
    fbar[i] += d * inv_eps;
    abar[i] -= d;
  }
}

// psibar_LM += (1/eps) e^{psi/eps} [X_L (e^{Lx+} - e^{Lx-}) + Y_M (e^{Ly+} - e^{Ly-})]
__global__ void moments_vjp_post(const float* __restrict__ psi, float inv_eps, const float* __restrict__ Lxp,
                                 const float* __restrict__ Lxn, const float* __restrict__ Lyp,
                                 const float* __restrict__ Lyn, int rows, int cols, float dX, float dY,
                                 float* __restrict__ psibar) {
  const size_t N = (size_t)rows * cols;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    if (psi[i] == -INFINITY) continue;
    const int L = (int)(i / cols), M = (int)(i % cols);
    const float X = (float)(L - rows / 2) * dX, Y = (float)(M - cols / 2) * dY;
    const float x = psi[i] * inv_eps;
    const float kx = (Lxp[i] == -INFINITY ? 0.f : expf(x + Lxp[i])) - (Lxn[i] == -INFINITY ? 0.f : expf(x + Lxn[i]));
    const float ky = (Lyp[i] == -INFINITY ? 0.f : expf(x + Lyp[i])) - (Lyn[i] == -INFINITY ? 0.f : expf(x + Lyn[i]));
    psibar[i] += inv_eps * (X * kx + Y * ky);
  }
}

// Transpose of the trapezoid integration along a line of n values p[i * stride], centre c: with S the
// sum of p from the outer end of the half that q lies in up to q (inclusive), and S' without q,
//     d[q] = +- h/2 (S + S')  (+ above the centre),   d[c] = h/2 (sum above - sum below).
// One warp per half line, from the outer end inwards, the loads of eight chunks in flight (one
// thread per row, a dependent load at a time, took 102 us at 256^2).  Returns the half's sum.
constexpr int kVjpChunks = 8;
__device__ float trapezoid_vjp_half(const float* __restrict__ p, size_t stride, int n, int c, float h, float* __restrict__ d,
                                    size_t dstride, bool up) {
  const int lane = threadIdx.x & 31;
  const int count = up ? n - 1 - c : c;
  const float s = up ? 0.5f * h : -0.5f * h;
  float carry = 0.f;
  for (int i0 = 0; i0 < count; i0 += 32 * kVjpChunks) {
    float v[kVjpChunks];
#pragma unroll
    for (int u = 0; u < kVjpChunks; ++u) {
      const int i = i0 + 32 * u + lane, q = up ? n - 1 - i : i;
      v[u] = i < count ? p[(size_t)q * stride] : 0.f;
    }
#pragma unroll
    for (int u = 0; u < kVjpChunks; ++u) {
      const int i = i0 + 32 * u + lane, q = up ? n - 1 - i : i;
      float t = v[u];
#pragma unroll
      for (int k = 1; k < 32; k <<= 1) {
        const float o = __shfl_up_sync(0xffffffffu, t, k);
        if (lane >= k) t += o;
      }
      t += carry;
      float before = __shfl_up_sync(0xffffffffu, t, 1);
      if (lane == 0) before = carry;
      if (i < count) d[(size_t)q * dstride] = s * (t + before);
      carry = __shfl_sync(0xffffffffu, t, 31);
    }
  }
  return carry;
}
// lines of n values, two warps each (8 warps per CTA): d as above, total[line] = sum of the line
__global__ void __launch_bounds__(256) trapezoid_vjp_kernel(const float* __restrict__ p, int lines, int n, size_t stride,
                                                            size_t line_step, float h, float* __restrict__ d,
                                                            size_t dstride, size_t dline_step, float* __restrict__ total) {
  __shared__ float s_half[8];
  const int w = threadIdx.x >> 5, line = blockIdx.x * 4 + (w >> 1), c = n / 2;
  const bool in = line < lines;
  const float* pl = p + (size_t)(in ? line : 0) * line_step;
  float* dl = d + (size_t)(in ? line : 0) * dline_step;
  float sum = 0.f;
  if (in) sum = trapezoid_vjp_half(pl, stride, n, c, h, dl, dstride, (w & 1) == 0);
  if ((threadIdx.x & 31) == 0) s_half[w] = sum;
  __syncthreads();
  if (in && (threadIdx.x & 63) == 0) {
    const float up = s_half[w], down = s_half[w + 1];
    dl[(size_t)c * dstride] = 0.5f * h * (up - down);
    if (total) total[line] = up + down + pl[(size_t)c * stride];
  }
}

// Through the normalisation a = g^2 / sum g^2 (of g and of G): parts of sum abar and sum amp^2 in
// FP64, then (every CTA adds the same parts in the same order) grad = 2 (abar - a sum abar) / amp.
// One CTA for all of it took 540 us per image at 256^2.
constexpr int kGradParts = 128;
struct GradArgs {
  const float* abar[2];
  const float* amp[2];
  float* grad[2];
  double* parts;      // [2][kGradParts][2]
  int which;          // finishing: 0 = g, 1 = G (one after the other: dL_dG may lie over g)
  size_t N;
};
template <bool FINISH>
__global__ void __launch_bounds__(256) grad_from_logmarg(GradArgs a) {
  __shared__ double s1[256], s2[256];
  const int y = FINISH ? a.which : blockIdx.y, tid = threadIdx.x;
  const float* const abar = a.abar[y];
  const float* const amp = a.amp[y];
  double t1 = 0.0, t2 = 0.0;
  if (FINISH) {
    if (tid < kGradParts) {
      t1 = a.parts[(y * kGradParts + tid) * 2];
      t2 = a.parts[(y * kGradParts + tid) * 2 + 1];
    }
  } else {
    for (size_t i = blockIdx.x * (size_t)blockDim.x + tid; i < a.N; i += (size_t)gridDim.x * blockDim.x) {
      t1 += (double)abar[i];
      t2 += (double)amp[i] * amp[i];
    }
  }
  s1[tid] = t1;
  s2[tid] = t2;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (tid < w) {
      s1[tid] += s1[tid + w];
      s2[tid] += s2[tid + w];
    }
    __syncthreads();
  }
  if (!FINISH) {
    if (tid == 0) {
      a.parts[(y * kGradParts + blockIdx.x) * 2] = s1[0];
      a.parts[(y * kGradParts + blockIdx.x) * 2 + 1] = s2[0];
    }
    return;
  }
  const double r = s1[0] / s2[0];
  for (size_t i = blockIdx.x * (size_t)blockDim.x + tid; i < a.N; i += (size_t)gridDim.x * blockDim.x) {
    const float x = amp[i];
    a.grad[y][i] = x > 0.f ? (float)(2.0 * ((double)abar[i] - (double)x * x * r) / x) : 0.f;
  }
}

inline dim3 grid_for(size_t N) {
  size_t b = (N + 255) / 256;
  return dim3((unsigned)(b < 2048 ? (b < 1 ? 1 : b) : 2048));
}

}  // namespace

extern "C" fot_status fot_backward(fot_ctx* c, const float* g, const float* G, const float* dL_dphi,
                                   const float* dL_df, const float* dL_dpsi, int checkpoint_every,
                                   float* dL_dg, float* dL_dG) {
  if (!c || !g || !G || !dL_dg || !dL_dG || checkpoint_every < 1) return FOT_EINVAL;
  if (!c->have_solution || c->sched.empty()) return FOT_ESTATE;
  if (cudaSetDevice(c->device) != cudaSuccess) return FOT_ECUDA;
  const int T = (int)c->sched.size();
  const int K = checkpoint_every;
  const int nseg = (T + K - 1) / K;
  const size_t N = (size_t)c->rows * c->cols;
  const size_t B = N * sizeof(float);
  cudaStream_t s = c->stream;
  const bool dense = c->precision == FOT_FP32_DENSE;
  // device memory of the backward, one allocation: checkpoints, one segment, adjoints and
  // temporaries, and the second problem's work space of the two-problem passes
  const size_t n_items = band_items(c->rows, c->cols), plan_words = band_plan_words(c->rows, c->cols);
  size_t need = 0;
  auto part = [&](size_t bytes) {
    const size_t at = need;
    need += (bytes + 255) / 256 * 256;
    return at;
  };
  const size_t at_ckpt = part(B * nseg);                 // psi at t = 0, K, 2K, ...
  const size_t at_psi = part(B * K), at_S = part(B * K), at_f = part(B * K), at_T = part(B * K);
  const size_t at_zero = need;                           // cleared: adjoints, counters
  const size_t at_psib = part(B), at_fb = part(B), at_ab = part(B), at_bb = part(B);
  const size_t at_order = part(2 * sizeof(int));
  const size_t zero_bytes = need - at_zero;
  size_t at_buf[15];
  for (size_t& at : at_buf) at = part(B);
  const size_t at_plan = part(plan_words * sizeof(float)), at_items = part(n_items * sizeof(int4));
  const size_t at_parts = part(4 * kGradParts * sizeof(double));
  unsigned char* mem = nullptr;
  if (cudaMalloc((void**)&mem, need) != cudaSuccess) {
    cudaGetLastError();
    return FOT_ENOMEM;
  }
  auto img = [&](size_t at) { return (float*)(mem + at); };
  float *ckpt = img(at_ckpt), *seg_psi = img(at_psi), *seg_S = img(at_S), *seg_f = img(at_f), *seg_T = img(at_T);
  float *psib = img(at_psib), *fb = img(at_fb), *ab = img(at_ab), *bb = img(at_bb);
  float *neg_inf = img(at_buf[0]), *tA = img(at_buf[1]), *tB = img(at_buf[2]), *Lp = img(at_buf[3]), *Ln = img(at_buf[4]);
  float *scratch = img(at_buf[5]), *psi_cur = img(at_buf[6]), *f_cur = img(at_buf[7]);
  float *lxp = img(at_buf[8]), *lxn = img(at_buf[9]), *lyp = img(at_buf[10]), *lyn = img(at_buf[11]);
  float *pp = img(at_buf[12]), *pn = img(at_buf[13]), *R2 = img(at_buf[14]);
  const dim3 gN = grid_for(N);
  tilt_begin(c);
  fill(c, neg_inf, N, -INFINITY);
  cudaMemsetAsync(mem + at_zero, 0, zero_bytes, s);
  // log(Lambda e^{in/eps} Lambda) of two inputs
  auto apply_pair = [&](const float* inA, const float* inB, double eps, float* LA, float* LB) {
    if (dense) {
      half_step_simt(c, inA, neg_inf, eps, scratch, LA, c->R);
      half_step_simt(c, inB, neg_inf, eps, scratch, LB, c->R);
      return;
    }
    PairSpace second{img(at_plan), (int4*)(mem + at_items), (int*)(mem + at_order), R2};
    half_step_band_pair(c, inA, inB, neg_inf, eps, scratch, f_cur, LA, LB, second);
  };
  // iteration t from psi_cur, its intermediate results kept as entry q of the segment
  auto forward_kept = [&](int t, int q) {
    cudaMemcpyAsync(seg_psi + (size_t)q * N, psi_cur, B, cudaMemcpyDeviceToDevice, s);
    half_step_dispatch(c, psi_cur, c->la, c->sched[t], seg_f + (size_t)q * N, seg_S + (size_t)q * N);
    half_step_dispatch(c, seg_f + (size_t)q * N, c->lb, c->sched[t], psi_cur, seg_T + (size_t)q * N);
  };
  // 1. forward with checkpoints (bitwise the solve: same kernels, same order)
  const double e0 = c->sched[0];
  fill(c, psi_cur, N, (float)(e0 * log(1.0 / (double)N)));
  for (int t = 0; t < T; ++t) {
    if (t % K == 0) cudaMemcpyAsync(ckpt + (size_t)(t / K) * N, psi_cur, B, cudaMemcpyDeviceToDevice, s);
    if (t >= (nseg - 1) * K) {
      forward_kept(t, t - (nseg - 1) * K);
    } else {
      half_step_dispatch(c, psi_cur, c->la, c->sched[t], f_cur, nullptr);
      half_step_dispatch(c, f_cur, c->lb, c->sched[t], psi_cur, nullptr);
    }
  }
  // 2. seeds at the end of the solve: psi_T = psi_cur, f_T, S_{T-1} = c->S_last
  const double eT = c->sched[T - 1];
  if (dL_dpsi) axpy_kernel<<<gN, 256, 0, s>>>(psib, dL_dpsi, 1.f, N);
  if (dL_df) axpy_kernel<<<gN, 256, 0, s>>>(fb, dL_df, 1.f, N);
  if (dL_dphi) {
    float* Dxb = tA;
    float* Dyb = tB;
    float* colb = scratch;
    cudaMemsetAsync(Dxb, 0, B, s);
    // the rows (sums into colb), then the centre column
    trapezoid_vjp_kernel<<<(c->rows + 3) / 4, 256, 0, s>>>(dL_dphi, c->rows, c->cols, 1, c->cols, (float)c->dx, Dyb, 1,
                                                           c->cols, colb);
    trapezoid_vjp_kernel<<<1, 64, 0, s>>>(colb, 1, c->rows, 1, 0, (float)c->dx, Dxb + c->cols / 2, c->cols, 0, nullptr);
    float* Dx = Lp;
    float* Dy = Ln;
    moments(c, psi_cur, c->S_last, eT, c->dx, Dx, Dy);
    moments_vjp_pre<<<gN, 256, 0, s>>>(Dxb, Dyb, Dx, Dy, (float)(1.0 / eT), N, fb, ab);
    // K(Dxbar e^{-S}), K(Dybar e^{-S}) on the target grid (log-domain applications)
    split_kernel<<<gN, 256, 0, s>>>(Dxb, c->S_last, (float)eT, N, pp, pn);
    apply_pair(pp, pn, eT, lxp, lxn);
    split_kernel<<<gN, 256, 0, s>>>(Dyb, c->S_last, (float)eT, N, pp, pn);
    apply_pair(pp, pn, eT, lyp, lyn);
    moments_vjp_post<<<gN, 256, 0, s>>>(psi_cur, (float)(1.0 / eT), lxp, lxn, lyp, lyn, c->rows, c->cols,
                                        (float)(1.0 / (c->rows * c->dx)), (float)(1.0 / (c->cols * c->dx)), psib);
  }
  // 3. reverse sweep, one recomputed segment at a time; psib holds the adjoint of psi_{t+1} at its
  // start, fb the seed of f_T (then zero)
  const float* f_seed = fb;
  for (int sg = nseg - 1; sg >= 0; --sg) {
    const int t0 = sg * K, t1 = t0 + K < T ? t0 + K : T;
    if (sg < nseg - 1) {
      cudaMemcpyAsync(psi_cur, ckpt + (size_t)sg * N, B, cudaMemcpyDeviceToDevice, s);
      for (int t = t0; t < t1; ++t) forward_kept(t, t - t0);
    }
    for (int t = t1 - 1; t >= t0; --t) {
      const int q = t - t0;
      const double e = c->sched[t];
      const float ie = (float)(1.0 / e), fe = (float)e;
      const float* f1 = seg_f + (size_t)q * N;
      // V-half: psi_{t+1} = eps (log b - T_t(f_{t+1})); the segment's first step starts from psib,
      // the others were split by the U-half before
      if (t == t1 - 1)
        vjp_step_kernel<<<gN, 256, 0, s>>>(psib, nullptr, 0.f, nullptr, nullptr, fe, bb, seg_T + (size_t)q * N, tA, tB,
                                           nullptr, N);
      apply_pair(tA, tB, e, Lp, Ln);
      // U-half: f_{t+1} = eps (log a - S_t(psi_t))
      vjp_step_kernel<<<gN, 256, 0, s>>>(f_seed, f1, ie, Lp, Ln, fe, ab, seg_S + (size_t)q * N, tA, tB, nullptr, N);
      f_seed = nullptr;
      apply_pair(tA, tB, e, Lp, Ln);
      // the adjoint of psi_t: split for the iteration before, or kept across the recomputation
      const bool last = t == t0;
      const float fp = last ? 0.f : (float)c->sched[t - 1];
      vjp_step_kernel<<<gN, 256, 0, s>>>(nullptr, seg_psi + (size_t)q * N, ie, Lp, Ln, fp, last ? nullptr : bb,
                                         last ? nullptr : seg_T + (size_t)(q - 1) * N, last ? nullptr : tA, tB,
                                         last ? psib : nullptr, N);
    }
  }
  // 4. through the normalisation to the amplitudes
  GradArgs ga{{ab, bb}, {g, G}, {dL_dg, dL_dG}, (double*)(mem + at_parts), 0, N};
  grad_from_logmarg<false><<<dim3(kGradParts, 2), 256, 0, s>>>(ga);
  for (ga.which = 0; ga.which < 2; ++ga.which) grad_from_logmarg<true><<<kGradParts, 256, 0, s>>>(ga);
  c->launches += 8;
  const cudaError_t le = cudaGetLastError();
  cudaStreamSynchronize(s);
  cudaFree(mem);
  if (le != cudaSuccess) return FOT_ECUDA;
  int e = 0;
  if (cudaMemcpy(&e, c->err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return FOT_ECUDA;
  return (fot_status)e;
}
