// Shared-memory FFT of a block's lines, used by the component solves and by
// the regular-grid transforms.
#pragma once

#include "sg_kernels.cuh"

namespace sg {

template <typename real>
__host__ __device__ __forceinline__ cplx<real> cmul(cplx<real> a, cplx<real> w) {
  return {a.x * w.x - a.y * w.y, a.x * w.y + a.y * w.x};
}

// Radix-2 butterfly (a, b) -> (a + w b, a - w b).  Doubles: eight fused
// operations, as many as with the product first, and two roundings per output
// instead of three.  (a - w b as 2 a - (a + w b) would take two instead of
// four, but the rounding of the sum then enters the difference: the root mean
// square error of a transform of 32 to 4096 values grows by 8 to 43%.)
template <typename real>
__host__ __device__ __forceinline__ void butterfly(cplx<real> a, cplx<real> b, cplx<real> w, cplx<real>& x0, cplx<real>& x1) {
  if constexpr (sizeof(real) == 8) {
    x0 = {fma(-b.y, w.y, fma(b.x, w.x, a.x)), fma(b.y, w.x, fma(b.x, w.y, a.y))};
    x1 = {fma(b.y, w.y, fma(-b.x, w.x, a.x)), fma(-b.y, w.x, fma(-b.x, w.y, a.y))};
  } else {
    const cplx<real> m = cmul(b, w);
    x0 = {a.x + m.x, a.y + m.y};
    x1 = {a.x - m.x, a.y - m.y};
  }
}

// Shared-memory index of element x of the line buffers: one padding element
// after every 32, so that the bit-reversed stores (consecutive t land 2^(logn-5)
// apart) and the large-span butterflies spread over the banks.
__device__ __forceinline__ int fpad(int x) { return x + (x >> 5); }
__host__ __device__ constexpr size_t fpad_size(size_t n) { return n + (n >> 5); }

// Iterative decimation-in-time FFT of nl lines of length 2^logn in shared
// memory (input in bit-reversed order, output natural).  Stages are taken in
// pairs (radix 2^2): a thread loads four elements {i, i+h, i+2h, i+3h}, does
// the two butterflies of stage s (span 2h) and the two of stage s+1 (span
// 4h) in registers and stores them, halving the passes over shared memory and
// the barriers; an odd last stage is a plain radix-2 pass.
// Twiddles are stage-major (twiddle_index): the lanes of a warp read
// consecutive entries in every stage, free of bank conflicts.
template <typename real>
__device__ __forceinline__ void fft_smem(cplx<real>* buf, int nl, int logn, bool inverse,
                                         const cplx<real>* __restrict__ tw) {
  const int len = 1 << logn;
  const int halfN = len >> 1;
  int s0 = 1;
  for (; s0 + 1 <= logn; s0 += 2) {
    const int h = 1 << (s0 - 1);
    const int quarter = len >> 2;
    for (int j = threadIdx.x; j < nl * quarter; j += blockDim.x) {
      const int li = j >> (logn - 2);
      const int jj = j & (quarter - 1);
      const int pos = jj & (h - 1);
      const int grp = jj >> (s0 - 1);
      const int i0 = li * len + grp * 4 * h + pos;
      // W_{2h}^pos, W_{4h}^pos and W_{4h}^(pos + h)
      cplx<real> w1 = tw[twiddle_index(h, pos)], w2 = tw[twiddle_index(2 * h, pos)],
                 w3 = tw[twiddle_index(2 * h, pos + h)];
      if (inverse) {
        w1.y = -w1.y;
        w2.y = -w2.y;
        w3.y = -w3.y;
      }
      const cplx<real> a0 = buf[fpad(i0)], a1 = buf[fpad(i0 + h)], a2 = buf[fpad(i0 + 2 * h)],
                       a3 = buf[fpad(i0 + 3 * h)];
      cplx<real> b0, b1, b2, b3, x0, x1, x2, x3;
      butterfly(a0, a1, w1, b0, b1);
      butterfly(a2, a3, w1, b2, b3);
      butterfly(b0, b2, w2, x0, x2);
      butterfly(b1, b3, w3, x1, x3);
      buf[fpad(i0)] = x0;
      buf[fpad(i0 + 2 * h)] = x2;
      buf[fpad(i0 + h)] = x1;
      buf[fpad(i0 + 3 * h)] = x3;
    }
    __syncthreads();
  }
  for (int s = s0; s <= logn; ++s) {
    const int half = 1 << (s - 1);
    for (int j = threadIdx.x; j < nl * halfN; j += blockDim.x) {
      const int li = j >> (logn - 1);
      const int jj = j & (halfN - 1);
      const int pos = jj & (half - 1);
      const int grp = jj >> (s - 1);
      const int i0 = li * len + grp * 2 * half + pos;
      const int i1 = i0 + half;
      cplx<real> w = tw[twiddle_index(half, pos)];
      if (inverse) w.y = -w.y;
      cplx<real> x0, x1;
      butterfly(buf[fpad(i0)], buf[fpad(i1)], w, x0, x1);
      buf[fpad(i0)] = x0;
      buf[fpad(i1)] = x1;
    }
    __syncthreads();
  }
}

__device__ __forceinline__ int bitrev(int t, int logn) { return logn == 0 ? 0 : (int)(__brev((unsigned)t) >> (32 - logn)); }

}  // namespace sg
