// Complex FFTs of power-of-two lines (8 .. 4096), shared by the far-field transform (fot_fft.cu)
// and the FFT convolutions (fot_cfot.cu).
//
// len / 8 threads hold a line, eight values each in registers.  Forward (decimation in frequency):
// radix-8 steps on values len/8, len/64, .. apart, exchanged through shared memory between steps,
// then the last one to three bits on eight neighbouring values; value s of the result is frequency
// bitrev(s).  The inverse runs the same steps backwards from that order, so a convolution
// permutes nothing.  A radix-8 step is three radix-2 ones in registers (log2(len)/3 exchanges
// instead of log2(len)); its twiddles e^{-2 pi i k / len} come from a table of the 4096-th roots
// of unity, rounded once from 64 bits.
//
// What bounds it: latency (barriers and shared-memory round trips); the radix-2 form with a sine
// and cosine per butterfly took 49 us for 512 lines of 1024 (one convolution pass) and 35 us for
// 1024 lines of 1024.
#pragma once

#include "fot_common.cuh"

namespace fot {

constexpr int kFftMax = 4096;

// shared-memory index of value i: one pad word per eight, so that the strides 8 and 64 between the
// threads of a step fall on different banks
__device__ __forceinline__ int fft_pad(int i) { return i + (i >> 3); }
__host__ __device__ constexpr int fft_line_floats(int len) { return 2 * (len + len / 8); }   // re, im
// words from one line of a CTA to the next: neighbouring lanes hold different lines, kept on
// different banks
__host__ __device__ inline int fft_line_stride(int len, int lpc) { return fft_line_floats(len) + (lpc > 1 && lpc <= 32 ? 32 / lpc : 0); }

__device__ __forceinline__ int rev3(int p) { return ((p & 1) << 2) | (p & 2) | (p >> 2); }

// y = x * (c, s), and x * conj
__device__ __forceinline__ void cmul(float& re, float& im, float c, float s) {
  const float r = re * c - im * s;
  im = fmaf(re, s, im * c);
  re = r;
}

// the last `bits` of three radix-2 steps on eight values a power of two apart; forward: sign -1
template <bool INV>
__device__ __forceinline__ void radix_steps(float (&re)[8], float (&im)[8], int bits) {
  constexpr float kR = 0.70710678118654752440f;
  auto pair = [&](int a, int b) {                         // (a, b) <- (a + b, a - b)
    const float ar = re[a], ai = im[a];
    re[a] = ar + re[b];
    im[a] = ai + im[b];
    re[b] = ar - re[b];
    im[b] = ai - im[b];
  };
  // the factor e^{-+ 2 pi i j / 8} of value b
  auto turn = [&](int b, int j) {
    const float s = INV ? 1.f : -1.f;
    const float r = re[b], i = im[b];
    if (j == 1) {
      re[b] = kR * (r - s * i);
      im[b] = kR * (i + s * r);
    } else if (j == 2) {
      re[b] = -s * i;
      im[b] = s * r;
    } else if (j == 3) {
      re[b] = kR * (-r - s * i);
      im[b] = kR * (s * r - i);
    }
  };
  if (!INV) {
    if (bits >= 3) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        pair(j, j + 4);
        turn(j + 4, j);
      }
    }
    if (bits >= 2) {
#pragma unroll
      for (int h = 0; h < 8; h += 4)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          pair(h + j, h + j + 2);
          turn(h + j + 2, 2 * j);
        }
    }
#pragma unroll
    for (int j = 0; j < 8; j += 2) pair(j, j + 1);
  } else {
#pragma unroll
    for (int j = 0; j < 8; j += 2) pair(j, j + 1);
    if (bits >= 2) {
#pragma unroll
      for (int h = 0; h < 8; h += 4)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          turn(h + j + 2, 2 * j);
          pair(h + j, h + j + 2);
        }
    }
    if (bits >= 3) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        turn(j + 4, j);
        pair(j, j + 4);
      }
    }
  }
}

// One line's transform by its len/8 threads (t: this thread's index among them).  lg = log2(len)
// >= 3; roots: the table; sm: the line's fft_line_floats(len) words.  Forward: on entry re/im[j] is
// value t + j len/8, on return value 8 t + j (frequency bitrev(8 t + j)).  Inverse: the other way
// round, unscaled.  Every thread of the CTA calls it (barriers).
template <bool INV>
__device__ __forceinline__ void fft_line(float (&re)[8], float (&im)[8], int lg, int t, const float2* __restrict__ roots,
                                         float* sm) {
  const int len = 1 << lg, steps = (lg - 1) / 3, rest = lg - 3 * steps;   // rest: 1 .. 3
  float* const sr = sm;
  float* const si = sm + len + (len >> 3);
  if (!INV) {
    for (int st = 0; st < steps; ++st) {
      // sub-transforms of L = len / 8^st, values h = L / 8 apart
      const int lh = lg - 3 * st - 3, h = 1 << lh, pos = t & (h - 1);
      const int i0 = ((t >> lh) << (lh + 3)) + pos;
      if (st > 0) {
        __syncthreads();
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          re[j] = sr[fft_pad(i0 + (j << lh))];
          im[j] = si[fft_pad(i0 + (j << lh))];
        }
        __syncthreads();
      }
      radix_steps<false>(re, im, 3);
      const int unit = pos * (kFftMax >> (lh + 3));
#pragma unroll
      for (int j = 1; j < 8; ++j) {
        const float2 w = __ldg(roots + unit * rev3(j));
        cmul(re[j], im[j], w.x, w.y);
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        sr[fft_pad(i0 + (j << lh))] = re[j];
        si[fft_pad(i0 + (j << lh))] = im[j];
      }
    }
    if (steps > 0) {
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        re[j] = sr[fft_pad(8 * t + j)];
        im[j] = si[fft_pad(8 * t + j)];
      }
    }
    radix_steps<false>(re, im, rest);
  } else {
    radix_steps<true>(re, im, rest);
    if (steps > 0) {
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        sr[fft_pad(8 * t + j)] = re[j];
        si[fft_pad(8 * t + j)] = im[j];
      }
    }
    for (int st = steps - 1; st >= 0; --st) {
      const int lh = lg - 3 * st - 3, h = 1 << lh, pos = t & (h - 1);
      const int i0 = ((t >> lh) << (lh + 3)) + pos;
      __syncthreads();
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        re[j] = sr[fft_pad(i0 + (j << lh))];
        im[j] = si[fft_pad(i0 + (j << lh))];
      }
      const int unit = pos * (kFftMax >> (lh + 3));
#pragma unroll
      for (int j = 1; j < 8; ++j) {
        const float2 w = __ldg(roots + unit * rev3(j));
        cmul(re[j], im[j], w.x, -w.y);
      }
      radix_steps<true>(re, im, 3);
      if (st > 0) {
        // (each thread writes back the places it read: no barrier before)
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          sr[fft_pad(i0 + (j << lh))] = re[j];
          si[fft_pad(i0 + (j << lh))] = im[j];
        }
      }
    }
  }
}

// lines per CTA for lines of len values: up to 512 threads, at most eight lines (32-byte segments
// of the transposed output), few enough to leave `n_lines` lines for 128 CTAs
inline int fft_lines_per_cta(int len, int n_lines) {
  int k = 1;
  while (k < 8 && 2 * k * (len / 8) <= 512 && n_lines / (2 * k) >= 128) k *= 2;
  while (k * (len / 8) < 32) k *= 2;                      // whole warps
  return k;
}

// the context's tables, made by its first transform: e^{-2 pi i k / 4096} in FP32 (c->roots), and
// cos(2 pi k / 4096) in FP64 (c->cosines)
fot_status fft_tables(fot_ctx* c);

}  // namespace fot
