// Far-field intensity and the L1 intensity loss of a phase solution (Sec. 5).
//
//   I = |F[g e^{2 pi i phi}]|^2,   loss = sum_LM | I_LM / sum I - b_LM |,
//
// F the 2-D DFT between the centred grids of Sec. 2 (x_j = (j - floor(n/2)) dx, X_L =
// (L - floor(n/2)) dX, dx dX = 1/n).  The centring multiplies each output of the plain DFT by a
// unit-modulus factor that depends on the output index alone, so I at (L, M) is the squared
// modulus of the plain DFT at ((L - c_r) mod n_r, (M - c_c) mod n_c): the kernels compute plain
// DFTs and write each intensity at its shifted position.  The amplitude is sqrt(a) = e^{log a / 2}
// (a = g^2 / sum g^2; the overall scale cancels in I / sum I).
//
// One kernel, launched twice (power-of-two lengths up to 4096; fot_fft.cuh): pass 0 transforms the
// rows of the field and writes the spectrum transposed as split real / imaginary planes; pass 1
// transforms those lines (the columns), writes |.|^2 at the shifted position and the CTA's part of
// the total power.  A last pass divides by the total (every CTA adds the same parts in the same
// order) and sums |I / P - b|; b = e^{log b} and the difference are formed in pairs of FP32 numbers
// and summed that way per thread (2^-37 relative: a double exponential per pixel took
// 33 us at 1024^2, the GPU's FP64 rate being 1/64 of its FP32 rate), across threads in FP64.
#include "fot_fft.cuh"

#include <algorithm>

namespace fot {
namespace {

// lines shorter than 8 (2, 4) are done as direct sums by their single thread
__device__ __forceinline__ void small_dft(float (&re)[8], float (&im)[8], int len) {
  float xr[4], xi[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    xr[k] = xi[k] = 0.f;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      if (j < len && k < len) {
        float s, c;
        sincospif(-2.f * (float)((j * k) % len) / (float)len, &s, &c);
        xr[k] += re[j] * c - im[j] * s;
        xi[k] += re[j] * s + im[j] * c;
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    re[k] = xr[k];
    im[k] = xi[k];
  }
}

// (ah, al) += t, the rounding error of the sum kept in al (Knuth's two-sum)
__device__ __forceinline__ void pair_add(float& ah, float& al, float t) {
  const float sum = ah + t, z = sum - ah;
  al += (ah - (sum - z)) + (t - z);
  ah = sum;
}

template <int PASS>
__global__ void __launch_bounds__(512) fft_line_kernel(
    const float* __restrict__ la, const float* __restrict__ phi,       // pass 0: [n_lines][len]
    const float* __restrict__ re_in, const float* __restrict__ im_in,  // pass 1: [n_lines][len]
    float* __restrict__ re_out, float* __restrict__ im_out,            // pass 0: [len][n_lines]
    float* __restrict__ inten, double* __restrict__ part,               // pass 1: [len][n_lines], CTA parts
    const float2* __restrict__ roots, int n_lines, int len, int lg, int lpc, int c_len, int c_line) {
  extern __shared__ float s_fft[];
  const int tpl = max(len >> 3, 1);                       // threads per line
  // neighbouring threads take the lines of the CTA in turn, so that the transposed stores of a
  // warp fill segments of lpc floats
  const int li = threadIdx.x % lpc, t = threadIdx.x / lpc;
  const int line = blockIdx.x * lpc + li;
  const bool in = line < n_lines && t < tpl;
  const size_t base = (size_t)min(line, n_lines - 1) * len;
  float re[8], im[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int i = len >= 8 ? t + j * tpl : j;
    re[j] = im[j] = 0.f;
    if (!in || i >= len) continue;
    if (PASS == 0) {
      const float amp = expf(0.5f * la[base + i]);        // log a = -inf -> 0
      float sn, cs;
      sincospif(2.f * phi[base + i], &sn, &cs);           // e^{2 pi i phi}, phi in cycles
      re[j] = amp * cs;
      im[j] = amp * sn;
    } else {
      re[j] = re_in[base + i];
      im[j] = im_in[base + i];
    }
  }
  if (len >= 8)
    fft_line<false>(re, im, lg, t, roots, s_fft + li * fft_line_stride(len, lpc));
  else
    small_dft(re, im, len);
  float ah = 0.f, al = 0.f;                               // this thread's power as a pair
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    if (!in || (len < 8 && j >= len)) continue;
    const int f = len >= 8 ? (int)(__brev((unsigned)(8 * t + j)) >> (32 - lg)) : j;   // frequency
    if (PASS == 0) {
      re_out[(size_t)f * n_lines + line] = re[j];
      im_out[(size_t)f * n_lines + line] = im[j];
    } else {
      // line = spectral column index, f = spectral row index
      const int L = (f + c_len) & (len - 1), M = (line + c_line) & (n_lines - 1);
      const float v = re[j] * re[j] + im[j] * im[j];
      inten[(size_t)L * n_lines + M] = v;
      pair_add(ah, al, v);
    }
  }
  if (PASS == 1) {
    __shared__ double s_sum[16];
    double acc = (double)ah + (double)al;
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
    if ((threadIdx.x & 31) == 0) s_sum[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x == 0) {
      for (int w = 1; w < (int)(blockDim.x >> 5); ++w) acc += s_sum[w];
      part[blockIdx.x] = acc;
    }
  }
}

// sum of n doubles by a CTA of 256 threads, in a fixed order; every thread gets it
__device__ double cta_sum(const double* __restrict__ v, int n, double* s) {
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc += v[i];
  s[threadIdx.x] = acc;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
    __syncthreads();
  }
  acc = s[0];
  __syncthreads();
  return acc;
}

// e^l as hi + lo, relative error below 2^-37; l <= 0 or a little above; tab: 2^(j/8) as hi + lo.  By table and
// polynomial (Tang, "Table-driven implementation of the exponential function in IEEE floating-point
// arithmetic", 1989): l = n ln(2) / 8 + r, e^l = 2^(n / 8) e^r, the product n ln(2) / 8 in three parts
// of which the first is exact (Cody and Waite), |r| <= 0.044 as a pair.
__device__ __forceinline__ void exp_pair(float l, const float2* tab, float& hi, float& lo) {
  constexpr double kStep = 0.69314718055994530942 / 8.0;
  const float n = rintf(l * (8.f * kLog2e));
  constexpr float kL1 = 2839.f / 32768.f;                 // 12 bits of the step: n kL1 is exact
  constexpr float kL2 = (float)(kStep - (double)kL1), kL3 = (float)(kStep - (double)kL1 - (double)kL2);
  const float r0 = fmaf(-n, kL1, l);                      // exact
  const float p = -n * kL2;
  const float pe = fmaf(-n, kL2, -p) - n * kL3;
  const float rh = r0 + p, z = rh - r0;                   // r = rh + rl (Knuth's two-sum)
  const float rl = ((r0 - (rh - z)) + (p - z)) + pe;
  // 1 + r + r^2 / 2 in pairs (Dekker's fast two-sum), r^3 (1/6 + r/24 + ...), 2^-16 of the sum, in FP32
  const float q = rh * rh, qe = fmaf(rh, rh, -q) + 2.f * rh * rl;
  float c = 1.f / 720.f;
  c = fmaf(c, rh, 1.f / 120.f);
  c = fmaf(c, rh, 1.f / 24.f);
  c = fmaf(c, rh, 1.f / 6.f);
  const float s1 = 1.f + rh, e1 = (rh - (s1 - 1.f)) + rl;
  const float h = 0.5f * q;
  const float s2 = s1 + h, e2 = h - (s2 - s1);
  const float tail = e1 + e2 + fmaf(c * rh, q, 0.5f * qe);
  const float eh = s2 + tail, el = tail - (eh - s2);
  const int ni = (int)fminf(fmaxf(n, -2400.f), 960.f);    // below 2^-126 the result fades to zero
  const float2 t = tab[ni & 7];
  const float vh = eh * t.x, vl = fmaf(eh, t.x, -vh) + fmaf(eh, t.y, el * t.x);
  const int k = ni >> 3;
  const float sa = exp2f((float)(k / 2)), sb = exp2f((float)(k - k / 2));
  hi = vh + vl;
  lo = (vl - (hi - vh)) * sa * sb;
  hi = hi * sa * sb;
}
// 2^(j/8), j = 0 .. 7
__device__ __forceinline__ double eighth_power(int j) {
  return j == 0 ? 1.0 : j == 1 ? 1.0905077326652576592 : j == 2 ? 1.1892071150027210667 : j == 3 ? 1.2968395546510096659
       : j == 4 ? 1.4142135623730950488 : j == 5 ? 1.5422108254079408236 : j == 6 ? 1.6817928305074290861
                : 1.8340080864093424635;
}

// with P the total of the n_parts parts: v <- v / P in place and out[b] = sum |v / P - e^{lb}|
__global__ void __launch_bounds__(256) intensity_loss_kernel(float* __restrict__ v, const float* __restrict__ lb,
                                                             const double* __restrict__ parts, int n_parts, size_t N,
                                                             double* __restrict__ out) {
  __shared__ double s[256];
  __shared__ float s_inv[2];
  __shared__ float2 s_pow[8];
  if (threadIdx.x < 8) {
    const double v2 = eighth_power(threadIdx.x);
    const float vh = (float)v2;
    s_pow[threadIdx.x] = make_float2(vh, (float)(v2 - (double)vh));
  }
  const double total = cta_sum(parts, n_parts, s);
  if (threadIdx.x == 0) {                                 // (FP64 division: once per CTA)
    const double inv = 1.0 / total;
    s_inv[0] = (float)inv;
    s_inv[1] = (float)(inv - (double)s_inv[0]);
  }
  __syncthreads();
  const float ih = s_inv[0], il = s_inv[1];
  float ah = 0.f, al = 0.f;                               // this thread's sum as a pair
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    const float x = v[i], l = lb[i];
    const float qh = x * ih, ql = fmaf(x, ih, -qh) + x * il;
    v[i] = qh + ql;
    float bh = 0.f, bl = 0.f;
    if (l != -INFINITY) exp_pair(l, s_pow, bh, bl);
    const float d = qh - bh, bb = qh - d, de = (bb - bh) + (qh - (d + bb));   // qh - bh = d + de
    const float w = de + (ql - bl), th = d + w, tz = th - d;
    const float tl = (d - (th - tz)) + (w - tz);          // |difference| = |th + tl|
    pair_add(ah, al, fabsf(th));
    al += th < 0.f ? -tl : tl;
  }
  s[threadIdx.x] = (double)ah + (double)al;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = s[0];
}

__global__ void __launch_bounds__(256) sum_parts_kernel(const double* __restrict__ part, int n, double* out) {
  __shared__ double s[256];
  const double t = cta_sum(part, n, s);
  if (threadIdx.x == 0) *out = t;
}

__global__ void fft_roots_kernel(float2* __restrict__ roots, double* __restrict__ cosines) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  double s, c;
  sincospi(-2.0 * (double)k / (double)kFftMax, &s, &c);
  roots[k] = make_float2((float)c, (float)s);
  cosines[k] = c;
}

int log2_exact(int n) {
  int l = 0;
  while ((1 << l) < n) ++l;
  return (1 << l) == n ? l : -1;
}

}  // namespace

bool intensity_supported(int rows, int cols) {
  return rows >= 2 && cols >= 2 && rows <= kFftMax && cols <= kFftMax && log2_exact(rows) > 0 &&
         log2_exact(cols) > 0;
}

// one line of 4096, or eight of 512, stay within the default limit
static_assert(fft_line_floats(kFftMax) * sizeof(float) + 8 * 16 <= 48 * 1024, "shared memory of a CTA's lines");

fot_status fft_tables(fot_ctx* c) {
  if (c->roots) return FOT_OK;
  if (!c->cap && cudaStreamCreateWithFlags(&c->cap, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    c->cap = nullptr;
    return FOT_ECUDA;
  }
  unsigned char* p = nullptr;
  constexpr size_t kRoots = kFftMax * sizeof(float2), kCos = kFftMax * sizeof(double);
  if (cudaMalloc((void**)&p, kRoots + kCos + 2 * kFftMax * sizeof(double)) != cudaSuccess) {
    cudaGetLastError();
    return FOT_ENOMEM;
  }
  // on the context's own stream, waited for: later calls may be on another stream, and the caller's may
  // have work before it or be under capture
  fft_roots_kernel<<<kFftMax / 256, 256, 0, c->cap>>>((float2*)p, (double*)(p + kRoots));
  if (cudaGetLastError() != cudaSuccess || cudaStreamSynchronize(c->cap) != cudaSuccess) {
    cudaGetLastError();
    cudaFree(p);
    return FOT_ECUDA;
  }
  c->roots = (float2*)p;
  c->cosines = (double*)(p + kRoots);
  c->fft_parts = c->cosines + kFftMax;
  return FOT_OK;
}

// I / P into c->tmp and the loss into out[0] (device); c->R, c->R2 hold the spectrum between
// the passes.  The caller checked intensity_supported.
void intensity_loss_gpu(fot_ctx* c, const float* phi, double* out) {
  const int nr = c->rows, nc = c->cols;
  const size_t N = (size_t)nr * nc;
  double* part = c->fft_parts;                            // [<= 4096] power parts, then loss parts
  auto shape = [](int len, int n_lines, int& lpc, int& ctas, int& threads, size_t& smem) {
    lpc = fft_lines_per_cta(std::max(len, 8), n_lines);
    ctas = (n_lines + lpc - 1) / lpc;
    threads = lpc * std::max(len / 8, 1);
    smem = len >= 8 ? (size_t)lpc * fft_line_stride(len, lpc) * sizeof(float) : 0;
  };
  int lpc, ctas, threads;
  size_t smem;
  shape(nc, nr, lpc, ctas, threads, smem);
  fft_line_kernel<0><<<ctas, threads, smem, c->stream>>>(c->la, phi, nullptr, nullptr, c->R, c->R2, nullptr, nullptr,
                                                         c->roots, nr, nc, log2_exact(nc), lpc, 0, 0);
  shape(nr, nc, lpc, ctas, threads, smem);
  fft_line_kernel<1><<<ctas, threads, smem, c->stream>>>(nullptr, nullptr, c->R, c->R2, nullptr, nullptr, c->tmp, part,
                                                         c->roots, nc, nr, log2_exact(nr), lpc, nr / 2, nc / 2);
  double* loss_part = c->fft_parts + kFftMax;
  intensity_loss_kernel<<<c->red_blocks, 256, 0, c->stream>>>(c->tmp, c->lb, part, ctas, N, loss_part);
  sum_parts_kernel<<<1, 256, 0, c->stream>>>(loss_part, c->red_blocks, out);
  c->launches += 4;
}

}  // namespace fot
