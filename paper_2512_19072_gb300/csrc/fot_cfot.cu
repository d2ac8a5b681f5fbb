// cFOT (Sec. 3.1): Algorithm 1 in the exponential domain with every product by the Toeplitz
// matrix Lambda replaced by a linear convolution with lambda_j = exp(-j^2 / (2 eps)),
// j = -(n-1) .. n-1, evaluated with FFTs:
//
//   u = a / (lambda * V * lambda),   V = b / (lambda * u * lambda).
//
// On its n outputs, the linear convolution of a line of length n with lambda equals the
// circular convolution of length P >= 2n - 1 (a power of two) of the zero-padded line with
// lambda wrapped around (lambda_j at index j mod P).  The forward transform (fot_fft.cuh) leaves the
// padded line in bit-reversed order, where it is multiplied by lambda's spectrum (real, lambda
// being even, and stored in that same order), and the inverse one returns natural order; one CTA
// holds one to eight lines.  Pass 0 convolves the rows and writes them transposed; pass 1
// convolves the columns and applies the update (u = e^{log a} / y, and log y for S_last).
//
// FP32 throughout, like the exponential-domain iteration the paper's cFOT is: an FFT
// convolution carries an absolute error of a few ulp of the line's largest value, so entries
// far below it lose their relative accuracy, and u, V leave the FP32 range once eps is small
// against the spread of the potentials.  A non-positive or non-finite convolution where the
// marginal has mass latches FOT_ENONFINITE: the cFOT instability Sec. 5 reports at small eps.
#include <math.h>

#include "fot_fft.cuh"

namespace fot {
namespace {

constexpr int kConvMaxP = kFftMax;

__device__ __forceinline__ int bitrev(int i, int log2p) { return (int)(__brev((unsigned)i) >> (32 - log2p)); }

// hat[bitrev(q)] = sum_{|j| <= n-1} lambda_j e^{-2 pi i j q / P} = 1 + 2 sum_{j >= 1} lambda_j cos(2 pi j q / P),
// in FP64: lambda_j once per CTA, the cosines from the table, both axes (blockIdx.y) in one launch.
// Bound by FP64 (two products per cycle and SM): 8 lanes per q, 32 q per CTA, so that the sums spread over
// the chip (one thread per q, 4 CTAs per axis, took 44 us per axis at n = 512; 14 us for both now).
struct SpectrumAxis {
  float* hat;
  int n, P, log2p;
};
struct SpectrumArgs {
  SpectrumAxis axis[2];
  const double* cosines;
  double eps;
};
__global__ void __launch_bounds__(256) lambda_spectrum_kernel(SpectrumArgs a) {
  __shared__ double s_lam[256];
  const SpectrumAxis x = a.axis[blockIdx.y];
  const int q = blockIdx.x * 32 + (threadIdx.x >> 3), part = threadIdx.x & 7;
  if ((int)blockIdx.x * 32 >= x.P) return;
  const int step = kFftMax >> x.log2p;
  double acc = 0.0;
  for (int j0 = 0; j0 < x.n; j0 += 256) {
    const int jt = j0 + threadIdx.x;
    __syncthreads();
    s_lam[threadIdx.x] = jt < x.n ? (jt == 0 ? 1.0 : 2.0) * exp(-(double)jt * (double)jt / (2.0 * a.eps)) : 0.0;
    __syncthreads();
    if (s_lam[0] == 0.0) break;                               // decreasing in j
    for (int j = part; j < 256; j += 8) acc += s_lam[j] * a.cosines[(((j0 + j) * q) & (x.P - 1)) * step];
  }
#pragma unroll
  for (int d = 1; d < 8; d <<= 1) acc += __shfl_xor_sync(0xffffffffu, acc, d);
  if (q < x.P && part == 0) x.hat[bitrev(q, x.log2p)] = (float)acc;
}

// PASS 0: y = (line of x) * lambda, written transposed: out[k][line].
// PASS 1: y likewise, then out[k][line] = e^{lmarg} / y and logsum[k][line] = log y.
template <int PASS>
__global__ void __launch_bounds__(512) conv_line_kernel(const float* __restrict__ x, const float* __restrict__ hat,
                                                        float* __restrict__ out, const float* __restrict__ lmarg,
                                                        float* __restrict__ logsum, int* err,
                                                        const float2* __restrict__ roots, int n_lines, int n,
                                                        int log2p, int lpc) {
  extern __shared__ float s_fft[];
  const int P = 1 << log2p, tpl = P >> 3;
  const int li = threadIdx.x % lpc, t = threadIdx.x / lpc;    // (lines in turn: see fot_fft.cu)
  const int line = blockIdx.x * lpc + li;
  const bool in = line < n_lines;
  const float* xl = x + (size_t)min(line, n_lines - 1) * n;
  float re[8], im[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int i = t + j * tpl;                                // n <= P / 2: the upper half is padding
    re[j] = j < 4 && in && i < n ? xl[i] : 0.f;
    im[j] = 0.f;
  }
  float* const sm = s_fft + li * fft_line_stride(P, lpc);
  fft_line<false>(re, im, log2p, t, roots, sm);
  const float scale = 1.f / (float)P;                         // (a power of two: exact)
  const float4 h0 = __ldg(reinterpret_cast<const float4*>(hat + 8 * t)), h1 = __ldg(reinterpret_cast<const float4*>(hat + 8 * t) + 1);
  const float h[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    re[j] *= h[j];
    im[j] *= h[j];
  }
  fft_line<true>(re, im, log2p, t, roots, sm);
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const int k = t + j * tpl;
    if (!in || k >= n) continue;
    const float y = re[j] * scale;
    const size_t o = (size_t)k * n_lines + line;
    if (PASS == 0) {
      out[o] = y;
    } else {
      const float lm = lmarg[o];
      float v = 0.f;
      if (lm != -INFINITY) {
        v = expf(lm) / y;
        if (!(y > 0.f) || !isfinite(v)) raise_error(err, FOT_ENONFINITE);
      }
      out[o] = v;
      if (logsum) logsum[o] = logf(y);
    }
  }
}

__global__ void fill_value_kernel(float* __restrict__ p, size_t N, float v) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x)
    p[i] = v;
}

// exponential-domain scaling -> potential: p <- eps log p (-inf where p = 0)
__global__ void to_potential_kernel(float* __restrict__ p, size_t N, float eps) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < N; i += (size_t)gridDim.x * blockDim.x) {
    const float v = p[i];
    p[i] = v > 0.f ? eps * logf(v) : -INFINITY;
  }
}

int pad_log2(int n) {                 // log2 of the smallest power of two >= max(2n - 1, 8)
  int l = 3;
  while ((1 << l) < 2 * n - 1) ++l;
  return l;
}

}  // namespace

bool cfot_supported(int rows, int cols) {
  return rows >= 2 && cols >= 2 && (1 << pad_log2(rows)) <= kConvMaxP && (1 << pad_log2(cols)) <= kConvMaxP;
}

// eps_px: the px^2 value of every iteration (host array of iters).  The context's f and psi
// hold u and V during the loop and the potentials afterwards; c->lam_hat holds the two spectra
// (rows at 0, cols at kConvMaxP).
void cfot_run(fot_ctx* c, const double* eps_px, int iters) {
  const int nr = c->rows, nc = c->cols;
  const size_t N = (size_t)nr * nc;
  const int lr = pad_log2(nr), lc = pad_log2(nc), Pr = 1 << lr, Pc = 1 << lc;
  float* hat_r = c->lam_hat;
  float* hat_c = c->lam_hat + kConvMaxP;
  const int fill_blocks = c->red_blocks;
  fill_value_kernel<<<fill_blocks, 256, 0, c->stream>>>(c->psi, N, (float)(1.0 / ((double)nr * nc)));
  int64_t k = 1;
  double e_prev = -1.0;
  const int lpc_c = fft_lines_per_cta(Pc, nr), lpc_r = fft_lines_per_cta(Pr, nc);   // lines of nc values, of nr values
  const size_t sm_c = (size_t)lpc_c * fft_line_stride(Pc, lpc_c) * sizeof(float);
  const size_t sm_r = (size_t)lpc_r * fft_line_stride(Pr, lpc_r) * sizeof(float);
  for (int t = 0; t < iters; ++t) {
    const double e = eps_px[t];
    if (e != e_prev) {
      const SpectrumArgs sa{{{hat_r, nr, Pr, lr}, {hat_c, nc, Pc, lc}}, c->cosines, e};
      lambda_spectrum_kernel<<<dim3(((Pr > Pc ? Pr : Pc) + 31) / 32, 2), 256, 0, c->stream>>>(sa);
      k += 1;
      e_prev = e;
    }
    for (int half = 0; half < 2; ++half) {
      const float* in = half == 0 ? c->psi : c->f;       // V, then u
      float* outp = half == 0 ? c->f : c->psi;           // u, then V
      const float* lm = half == 0 ? c->la : c->lb;
      float* ls = (half == 0 && t == iters - 1) ? c->S_last : nullptr;
      conv_line_kernel<0><<<(nr + lpc_c - 1) / lpc_c, lpc_c * (Pc / 8), sm_c, c->stream>>>(
          in, hat_c, c->R, nullptr, nullptr, c->err, c->roots, nr, nc, lc, lpc_c);
      conv_line_kernel<1><<<(nc + lpc_r - 1) / lpc_r, lpc_r * (Pr / 8), sm_r, c->stream>>>(
          c->R, hat_r, outp, lm, ls, c->err, c->roots, nc, nr, lr, lpc_r);
      k += 2;
    }
  }
  const float el = (float)eps_px[iters - 1];
  to_potential_kernel<<<fill_blocks, 256, 0, c->stream>>>(c->f, N, el);
  to_potential_kernel<<<fill_blocks, 256, 0, c->stream>>>(c->psi, N, el);
  c->launches += k + 2;
}

size_t cfot_spectrum_floats() { return 2 * (size_t)kConvMaxP; }

}  // namespace fot
