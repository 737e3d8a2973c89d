// Regular-grid spectral work: the filter mode's Poisson solve (Algorithm 2)
// and the transforms of the tau estimator (Algorithm 1).
//
// Everything is a function of a real array, so the transforms keep half a
// spectrum, k_x = 0 .. N/2 (P = N/2 + 1 values per row, x fastest):
//   rows    two real rows make one complex transform; their spectra are
//           separated by symmetry as they are written;
//   columns transforms along the other axes, in place, P N^(d-2) lines;
//           the last forward one is fused with what is done to the spectrum
//           and with the first inverse one;
//   fields  two half spectra of real rows make one complex inverse
//           transform, whose real and imaginary parts are the rows.
// The estimator's thresholded spectra are mostly zero: column tiles without
// a non-zero mode skip their transform (its result is zero).
//
// Bound: the estimator by the double-precision pipe (GB300: two operations
// per clock and SM; k_est_rows 91% busy, k_est_columns 70%), which half spectra
// and skipped tiles spare; the filter's solve by L1 (k_solve_columns 77% busy)
// and latency.  Before, with whole complex arrays and a pass per operation:
// estimator and step 427 -> 194 us (2D n = 9, adaptive), 815 -> 264 us (3D n = 6);
// the filter's solve with profiling events 100 -> 56 us (2D n = 10).
#include <algorithm>

#include "sg_fft.cuh"

namespace sg {
namespace {

constexpr int SP_SMEM = 200 * 1024;

// Twiddles in shared memory when they fit beside the lines.
template <typename real>
__device__ __forceinline__ const cplx<real>* stage_twiddles(const cplx<real>* __restrict__ tw, int logn, cplx<real>* sm) {
  if (!sm) return tw;
  for (int e = threadIdx.x; e < twiddle_count(logn); e += blockDim.x) sm[e] = tw[e];
  return sm;
}

// Non-negative doubles order like their bits.
__device__ __forceinline__ void atomic_max_nonneg(double* addr, double v) {
  atomicMax(reinterpret_cast<unsigned long long*>(addr), (unsigned long long)__double_as_longlong(v));
}
// Largest v of the block into *out (one atomic; no barrier needed before).
__device__ __forceinline__ void block_max_store(double v, double* out) {
  __shared__ double red[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  __syncthreads();
  if (lane == 0) red[w] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) v = fmax(v, red[k]);
    atomic_max_nonneg(out, v);
  }
}

// ---------------------------------------------------------------- rows: real -> half spectra
// Block: C pairs of rows.  H[row * P + kx] = scale * F(row); largest |value|
// into *vmax when given.
template <typename Tin, typename real>
__global__ void __launch_bounds__(512) k_rows_forward(const Tin* __restrict__ in, cplx<real>* __restrict__ H, int logn,
                                                      int C, real scale, const cplx<real>* __restrict__ tw,
                                                      int tw_smem, double* vmax) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<real>* buf = reinterpret_cast<cplx<real>*>(smem_raw);
  const int N = 1 << logn, P = N / 2 + 1, total = C << logn;
  pdl_trigger();
  const cplx<real>* tws = stage_twiddles(tw, logn, tw_smem ? buf + fpad_size(total) : nullptr);
  pdl_wait(in);
  const size_t row0 = (size_t)blockIdx.x * C * 2;
  double mx = 0.0;
  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    const int p = e >> logn, t = e & (N - 1);
    const Tin* r = in + ((row0 + 2 * p) << logn) + t;
    const real a = (real)r[0], b = (real)r[N];
    if (vmax) mx = fmax(mx, fmax(fabs((double)a), fabs((double)b)));
    buf[fpad((p << logn) + bitrev(t, logn))] = {a * scale, b * scale};
  }
  __syncthreads();
  fft_smem<real>(buf, C, logn, false, tws);
  const real h = (real)0.5;
  for (int e = threadIdx.x; e < C * P; e += blockDim.x) {
    const int p = e / P, k = e - p * P;
    const cplx<real> z = buf[fpad((p << logn) + (k & (N - 1)))], m = buf[fpad((p << logn) + ((N - k) & (N - 1)))];
    cplx<real>* d = H + (row0 + 2 * p) * P + k;
    d[0] = {h * (z.x + m.x), h * (z.y - m.y)};   // (Z_k + conj Z_-k) / 2
    d[P] = {h * (z.y + m.y), h * (m.x - z.x)};   // (Z_k - conj Z_-k) / 2i
  }
  if (vmax) block_max_store(mx, vmax);
}

// ---------------------------------------------------------------- columns
struct SpectrumKF {
  double k[3];
};
constexpr int SP_MASKS = 7;
struct ColumnArgs {
  int D, logn, axis;  // axis >= 1
  int C;              // lines per block (a power of two)
  int nlines;         // P N^(D-2)
  int tw_smem;
};
// Estimator: threshold eps = frac max|z| and the products of k_m^2 of `nmask`
// masks (bit m: axis m).  m2max / vmax: max (s|z|)^2 and max|rho~|, which sets
// the power of two s that keeps the squares in range.
struct EstArgs {
  SpectrumKF kf;
  int mask[SP_MASKS];
  int nmask;
  double frac;
  const double* vmax;
  double* m2max;
  size_t wstride;
};

__device__ __forceinline__ double est_scale(const double* vmax) {
  const double m = *vmax;
  return m > 0.0 && isfinite(m) ? scalbn(1.0, -max(-1000, min(1000, ilogb(m)))) : 1.0;
}
__device__ __forceinline__ double est_square(cplx<double> z, double s) {
  const double a = z.x * s, b = z.y * s;
  return fma(a, a, b * b);
}

// A block's tile of C lines: thread -> its line and place along it.
struct Tile {
  int li, t0, dt;
  bool valid;
  size_t base, stride;
  int kx, other;  // line coordinates: k_x and the remaining axis (3D)
};
__device__ __forceinline__ Tile make_tile(const ColumnArgs& a, int block) {
  const int N = 1 << a.logn, P = N / 2 + 1, logC = __ffs(a.C) - 1;
  Tile t;
  t.li = threadIdx.x & (a.C - 1);
  t.t0 = threadIdx.x >> logC;
  t.dt = blockDim.x >> logC;
  const int line = block * a.C + t.li;
  t.valid = line < a.nlines;
  t.other = line / P;
  t.kx = line - t.other * P;
  // axis 1: lines (kx, z), step P; axis 2: lines (kx, y), step N P
  t.base = a.axis == 1 ? (size_t)t.other * N * P + t.kx : (size_t)line;
  t.stride = a.axis == 1 ? (size_t)P : (size_t)N * P;
  return t;
}

// In place along one axis.  max2: the estimator's largest (s|z|)^2 (forward,
// last axis).  Inverse passes skip tiles that are all zero.
template <typename real>
__global__ void __launch_bounds__(512) k_columns(cplx<real>* __restrict__ Z, ColumnArgs a, int inverse, size_t zstride,
                                                 const cplx<real>* __restrict__ tw, const double* vmax, double* max2) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<real>* buf = reinterpret_cast<cplx<real>*>(smem_raw);
  const int N = 1 << a.logn;
  const Tile T = make_tile(a, blockIdx.x);
  cplx<real>* z = Z + blockIdx.y * zstride + T.base;
  pdl_trigger();
  const cplx<real>* tws = stage_twiddles(tw, a.logn, a.tw_smem ? buf + fpad_size((size_t)a.C << a.logn) : nullptr);
  pdl_wait(z, vmax);
  bool any = false;
  for (int t = T.t0; t < N; t += T.dt) {
    cplx<real> v = {(real)0, (real)0};
    if (T.valid) v = z[t * T.stride];
    any |= !(v.x == (real)0 && v.y == (real)0);
    buf[fpad((T.li << a.logn) + bitrev(t, a.logn))] = v;
  }
  if (!__syncthreads_or(any) && inverse) return;
  fft_smem<real>(buf, a.C, a.logn, inverse != 0, tws);
  double m2 = 0.0;
  const double s = max2 ? est_scale(vmax) : 1.0;
  for (int t = T.t0; t < N; t += T.dt)
    if (T.valid) {
      const cplx<real> v = buf[fpad((T.li << a.logn) + t)];
      z[t * T.stride] = v;
      if (max2) m2 = fmax(m2, est_square({(double)v.x, (double)v.y}, s));
    }
  if (max2) block_max_store(m2, max2);
}

// k_m^2 products of one mode: index along each axis -> wavenumber.
__device__ __forceinline__ double est_k(const SpectrumKF& kf, int m, int i, int N) {
  return kf.k[m] * (double)(i < (N >> 1) ? i : i - N);
}

// Estimator: threshold and derivative factor of mask blockIdx.y, then the
// inverse transform along the last axis, Z -> W[mask].
__global__ void __launch_bounds__(512) k_est_columns(const cplx<double>* __restrict__ Z, cplx<double>* __restrict__ W,
                                                     ColumnArgs a, EstArgs e, const cplx<double>* __restrict__ tw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<double>* buf = reinterpret_cast<cplx<double>*>(smem_raw);
  const int N = 1 << a.logn;
  const Tile T = make_tile(a, blockIdx.x);
  const int mask = e.mask[blockIdx.y];
  pdl_trigger();
  const cplx<double>* tws = stage_twiddles(tw, a.logn, a.tw_smem ? buf + fpad_size((size_t)a.C << a.logn) : nullptr);
  pdl_wait(Z, e.vmax, e.m2max);
  const double s = est_scale(e.vmax), eps2 = e.frac * e.frac * *e.m2max;
  double fl = 1.0;  // factors of the line's own axes
  if (mask & 1) {
    const double k = est_k(e.kf, 0, T.kx, N);
    fl *= k * k;
  }
  if (a.D == 3 && (mask & 2)) {
    const double k = est_k(e.kf, 1, T.other, N);
    fl *= k * k;
  }
  const bool last = (mask >> (a.D - 1)) & 1;
  bool any = false;
  for (int t = T.t0; t < N; t += T.dt) {
    cplx<double> v = {0.0, 0.0};
    if (T.valid) {
      const cplx<double> z = Z[T.base + t * T.stride];
      if (est_square(z, s) >= eps2) {
        double f = fl;
        if (last) {
          const double k = est_k(e.kf, a.D - 1, t, N);
          f *= k * k;
        }
        v = {z.x * f, z.y * f};
        any |= !(v.x == 0.0 && v.y == 0.0);
      }
    }
    buf[fpad((T.li << a.logn) + bitrev(t, a.logn))] = v;
  }
  cplx<double>* w = W + blockIdx.y * e.wstride + T.base;
  if (!__syncthreads_or(any)) {
    for (int t = T.t0; t < N; t += T.dt)
      if (T.valid) w[t * T.stride] = {0.0, 0.0};
    return;
  }
  fft_smem<double>(buf, a.C, a.logn, true, tws);
  for (int t = T.t0; t < N; t += T.dt)
    if (T.valid) w[t * T.stride] = buf[fpad((T.li << a.logn) + t)];
}

// Estimator, empirical constants: max over the kept modes of |k^2 product z|.
__global__ void __launch_bounds__(256) k_est_modes(const cplx<double>* __restrict__ Z, int D, int logn, EstArgs e,
                                                   double* out) {
  pdl_trigger();
  pdl_wait(Z, e.vmax, e.m2max);
  const int N = 1 << logn, P = N / 2 + 1;
  const size_t n = (size_t)P << ((D - 1) * logn);
  const double s = est_scale(e.vmax), eps2 = e.frac * e.frac * *e.m2max;
  double mx[SP_MASKS] = {};
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const cplx<double> z = Z[i];
    if (!(est_square(z, s) >= eps2)) continue;
    const size_t row = i / P;
    const int idx[3] = {(int)(i - row * P), (int)(row & (N - 1)), (int)(row >> logn)};
    double k2[3] = {1.0, 1.0, 1.0};
    for (int m = 0; m < D; ++m) {
      const double k = est_k(e.kf, m, idx[m], N);
      k2[m] = k * k;
    }
#pragma unroll
    for (int q = 0; q < SP_MASKS; ++q)
      if (q < e.nmask) {
        double f = 1.0;
        for (int m = 0; m < D; ++m)
          if (e.mask[q] & (1 << m)) f *= k2[m];
        mx[q] = fmax(mx[q], hypot(z.x * f, z.y * f));
      }
  }
#pragma unroll
  for (int q = 0; q < SP_MASKS; ++q)
    if (q < e.nmask) block_max_store(mx[q], out + q);
}

// Filter mode, components blockIdx.y, blockIdx.y + gridDim.y, ...: forward
// along the last axis, E^_m = -i k_m rho^ / |k|^2 (k = 0
// and the Nyquist plane of axis m -> 0, the component-grid rules), inverse
// along the last axis, Z -> W[m] for every component.
// ktab[m * N + i] = 2 pi / L_m * (i < N/2 ? i : i - N), in the run's precision.
template <typename real>
__global__ void __launch_bounds__(512) k_solve_columns(const cplx<real>* __restrict__ Z, cplx<real>* __restrict__ W,
                                                       size_t wstride, ColumnArgs a, const real* __restrict__ ktab,
                                                       real norm, const cplx<real>* __restrict__ tw) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int N = 1 << a.logn;
  const size_t nbuf = fpad_size((size_t)a.C << a.logn);
  cplx<real>* buf0 = reinterpret_cast<cplx<real>*>(smem_raw);
  cplx<real>* buf1 = buf0 + nbuf;
  const Tile T = make_tile(a, blockIdx.x);
  pdl_trigger();
  const cplx<real>* tws = stage_twiddles(tw, a.logn, a.tw_smem ? buf1 + nbuf : nullptr);
  pdl_wait(Z);
  for (int t = T.t0; t < N; t += T.dt) {
    cplx<real> v = {(real)0, (real)0};
    if (T.valid) v = Z[T.base + t * T.stride];
    buf0[fpad((T.li << a.logn) + bitrev(t, a.logn))] = v;
  }
  __syncthreads();
  fft_smem<real>(buf0, a.C, a.logn, false, tws);
  const int last = a.D - 1;
  real kl[3] = {(real)0, (real)0, (real)0};
  bool nyq[3] = {false, false, false};
  if (T.valid) {
    kl[0] = ktab[T.kx];
    nyq[0] = T.kx == (N >> 1);
    if (a.D == 3) {
      kl[1] = ktab[N + T.other];
      nyq[1] = T.other == (N >> 1);
    }
  }
  for (int m = blockIdx.y; m < a.D; m += gridDim.y) {
    for (int t = T.t0; t < N; t += T.dt) {
      const real kt = ktab[last * N + t];
      real k2 = kl[0] * kl[0];
      if (a.D == 3) k2 += kl[1] * kl[1];
      k2 += kt * kt;
      const real km = m == last ? kt : kl[m];
      const bool zero = k2 == (real)0 || (m == last ? t == (N >> 1) : nyq[m]);
      const cplx<real> r = buf0[fpad((T.li << a.logn) + t)];
      cplx<real> out = {(real)0, (real)0};
      if (!zero) {
        const real f = km * (norm / k2);
        out = {r.y * f, -r.x * f};
      }
      buf1[fpad((T.li << a.logn) + bitrev(t, a.logn))] = out;
    }
    __syncthreads();
    fft_smem<real>(buf1, a.C, a.logn, true, tws);
    cplx<real>* w = W + m * wstride + T.base;
    for (int t = T.t0; t < N; t += T.dt)
      if (T.valid) w[t * T.stride] = buf1[fpad((T.li << a.logn) + t)];
    __syncthreads();
  }
}

// ---------------------------------------------------------------- half spectra -> real rows
// Z = A + i B over the full line from two half spectra of real rows (the
// imaginary parts of their k = 0 and Nyquist values are rounding), the
// inverse transform, then row A in the real and row B in the imaginary part.
template <typename real>
__device__ __forceinline__ void load_real_pair(cplx<real>* buf, int li, int logn, const cplx<real>* __restrict__ A,
                                               const cplx<real>* __restrict__ B, int k) {
  const int N = 1 << logn;
  cplx<real> a = A[k], b = B[k];
  if (k == 0 || k == N / 2) {
    buf[fpad((li << logn) + bitrev(k, logn))] = {a.x, b.x};
  } else {
    buf[fpad((li << logn) + bitrev(k, logn))] = {a.x - b.y, a.y + b.x};
    buf[fpad((li << logn) + bitrev(N - k, logn))] = {a.x + b.y, b.x - a.y};
  }
}

// Estimator: max |value| of mask blockIdx.y's field; a block takes C pairs of
// consecutive rows.
__global__ void __launch_bounds__(512) k_est_rows(const cplx<double>* __restrict__ W, size_t wstride, int logn, int C,
                                                  const cplx<double>* __restrict__ tw, int tw_smem, double* out) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cplx<double>* buf = reinterpret_cast<cplx<double>*>(smem_raw);
  const int N = 1 << logn, P = N / 2 + 1;
  pdl_trigger();
  const cplx<double>* tws = stage_twiddles(tw, logn, tw_smem ? buf + fpad_size((size_t)C << logn) : nullptr);
  pdl_wait(W);
  const cplx<double>* w = W + blockIdx.y * wstride + (size_t)blockIdx.x * C * 2 * P;
  for (int e = threadIdx.x; e < C * P; e += blockDim.x) {
    const int p = e / P, k = e - p * P;
    load_real_pair<double>(buf, p, logn, w + (size_t)2 * p * P, w + (size_t)(2 * p + 1) * P, k);
  }
  __syncthreads();
  fft_smem<double>(buf, C, logn, true, tws);
  double mx = 0.0;
  for (int e = threadIdx.x; e < (C << logn); e += blockDim.x) {
    const cplx<double> v = buf[fpad(e)];
    mx = fmax(mx, fmax(fabs(v.x), fabs(v.y)));
  }
  block_max_store(mx, out + blockIdx.y);
}

// Filter mode: C transforms per block.  TWO: components 0 and 1 of one row
// each (A, B their half spectra); else component m of two consecutive rows.
// E_hi is node-interleaved; per-block partials of the sum of squares from part0 on, closed by
// the last block of the last launch.
template <typename real, bool TWO>
__global__ void __launch_bounds__(512) k_field_rows(const cplx<real>* __restrict__ A, const cplx<real>* __restrict__ B,
                                                    int logn, int C, const cplx<real>* __restrict__ tw, int tw_smem,
                                                    real* __restrict__ Ehi, int stride, int m, double* __restrict__ partials, int part0, const CombineFinal fin) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ double red[32];
  cplx<real>* buf = reinterpret_cast<cplx<real>*>(smem_raw);
  const int N = 1 << logn, P = N / 2 + 1;
  pdl_trigger();
  const cplx<real>* tws = stage_twiddles(tw, logn, tw_smem ? buf + fpad_size((size_t)C << logn) : nullptr);
  pdl_wait(A, B);
  const size_t j0 = (size_t)blockIdx.x * C;  // first transform
  for (int e = threadIdx.x; e < C * P; e += blockDim.x) {
    const int p = e / P, k = e - p * P;
    if constexpr (TWO)
      load_real_pair<real>(buf, p, logn, A + (j0 + p) * P, B + (j0 + p) * P, k);
    else
      load_real_pair<real>(buf, p, logn, A + 2 * (j0 + p) * P, A + (2 * (j0 + p) + 1) * P, k);
  }
  __syncthreads();
  fft_smem<real>(buf, C, logn, true, tws);
  SquareSum<real> energy;
  for (int e = threadIdx.x; e < (C << logn); e += blockDim.x) {
    const cplx<real> v = buf[fpad(e)];
    energy.add(v.x);
    energy.add(v.y);
    if constexpr (TWO) {
      *reinterpret_cast<cplx<real>*>(Ehi + ((j0 << logn) + e) * stride) = v;
    } else {
      const int p = e >> logn, t = e & (N - 1);
      const size_t node = ((2 * (j0 + p)) << logn) + t;
      Ehi[node * stride + m] = v.x;
      Ehi[(node + N) * stride + m] = v.y;
    }
  }
  const double tot = block_sum_double(energy.value(), red);
  if (threadIdx.x == 0) partials[part0 + blockIdx.x] = tot;
  if (fin.active) combine_finalize(partials, part0 + (int)gridDim.x, fin, red);
}

// ---------------------------------------------------------------- launch shapes
// Lines per block and threads: up to 16 lines, fewer (down to cmin; two for
// columns, whose lines are read in pieces of one node each) while the grid has
// less than two blocks per SM, within shared memory.  The filter's fused
// column pass at 2D n = 10, regular solve in all: 85 us with four columns per
// block, 67 with two, 81 with one; with the components in blocks of their own
// (the forward transform done twice) 55.
struct Shape {
  int C, threads, tw_smem;
  size_t smem;
  unsigned blocks;
};
template <typename real>
int line_shape(long long lines, int logn, int cmin, int nbuf, bool divide, Shape* s) {
  const size_t cs = sizeof(cplx<real>), tws = (size_t)twiddle_count(logn) * cs;
  int C = 16;
  while (C > 1 && ((divide && lines % C) || nbuf * fpad_size((size_t)C << logn) * cs > (size_t)SP_SMEM)) C >>= 1;
  while (C > cmin && (lines + C - 1) / C < 2 * 152) C >>= 1;
  s->C = C;
  s->smem = nbuf * fpad_size((size_t)C << logn) * cs;
  if (s->smem > (size_t)SP_SMEM) {
    set_error("spectral pass: a line does not fit shared memory");
    return SG_ERR_UNSUPPORTED;
  }
  s->tw_smem = s->smem + tws <= (size_t)SP_SMEM ? 1 : 0;
  if (s->tw_smem) s->smem += tws;
  s->threads = std::max(64, std::min(512, (C << logn) / 4));
  s->blocks = (unsigned)((lines + C - 1) / C);
  return SG_OK;
}
template <typename K>
int allow_lines(K* kernel, DeviceSet& done, size_t smem) {
  return smem > 40 * 1024 ? allow_smem(kernel, done, SP_SMEM) : SG_OK;  // with the static part the total may pass 48 KB
}

template <typename Tin, typename real>
int rows_forward(const Tin* in, cplx<real>* H, int D, int n, real scale, const cplx<real>* tw, double* vmax,
                 cudaStream_t s) {
  Shape sh;
  SG_TRY(line_shape<real>(1ll << ((D - 1) * n - 1), n, 1, 1, true, &sh));
  static DeviceSet done{0};
  SG_TRY(allow_lines(k_rows_forward<Tin, real>, done, sh.smem));
  SG_CUDA(launch_pdl(k_rows_forward<Tin, real>, dim3(sh.blocks), dim3(sh.threads), sh.smem, s, in, H, n, sh.C, scale, tw, sh.tw_smem, vmax));
  SG_CHECK_LAUNCH();
  return SG_OK;
}
template <typename real>
ColumnArgs column_args(int D, int n, int axis, const Shape& sh) {
  ColumnArgs a;
  a.D = D;
  a.logn = n;
  a.axis = axis;
  a.C = sh.C;
  a.nlines = ((1 << n) / 2 + 1) << ((D - 2) * n);
  a.tw_smem = sh.tw_smem;
  return a;
}

template <typename real>
int columns(cplx<real>* Z, int D, int n, int axis, bool inverse, int count, size_t zstride, const cplx<real>* tw,
            const double* vmax, double* max2, cudaStream_t s) {
  Shape sh;
  const long long lines = (long long)((1 << n) / 2 + 1) << ((D - 2) * n);
  SG_TRY(line_shape<real>(lines, n, 2, 1, false, &sh));
  static DeviceSet done{0};
  SG_TRY(allow_lines(k_columns<real>, done, sh.smem));
  SG_CUDA(launch_pdl(k_columns<real>, dim3(sh.blocks, count), dim3(sh.threads), sh.smem, s, Z, column_args<real>(D, n, axis, sh), inverse ? 1 : 0, zstride, tw, vmax, max2));
  SG_CHECK_LAUNCH();
  return SG_OK;
}

}  // namespace

size_t half_spectrum(int dim, int n) { return (size_t)((1 << n) / 2 + 1) << ((dim - 1) * n); }

template <typename real>
int launch_regular_solve(const real* rho_f, cplx<real>* Z, cplx<real>* W, const real* ktab, const cplx<real>* tw,
                         int dim, int n, real* Ehi, int stride, double* partials, const CombineFinal& fin,
                         cudaStream_t s) {
  const size_t nd = (size_t)1 << (dim * n), hs = half_spectrum(dim, n);
  SG_TRY(rows_forward<real, real>(rho_f, Z, dim, n, (real)1, tw, nullptr, s));
  if (dim == 3) SG_TRY(columns<real>(Z, dim, n, 1, false, 1, 0, tw, nullptr, nullptr, s));
  Shape sh;
  const long long lines = (long long)((1 << n) / 2 + 1) << ((dim - 2) * n);
  SG_TRY(line_shape<real>(lines, n, 2, 2, false, &sh));
  static DeviceSet done{0};
  SG_TRY(allow_lines(k_solve_columns<real>, done, sh.smem));
  const unsigned groups = sh.blocks < 4 * 152 ? dim : 1;
  SG_CUDA(launch_pdl(k_solve_columns<real>, dim3(sh.blocks, groups), dim3(sh.threads), sh.smem, s, Z, W, hs, column_args<real>(dim, n, dim - 1, sh), ktab, (real)(1.0 / (double)nd), tw));
  SG_CHECK_LAUNCH();
  if (dim == 3) SG_TRY(columns<real>(W, dim, n, 1, true, 3, hs, tw, nullptr, nullptr, s));
  const long long rows = 1ll << ((dim - 1) * n);
  SG_TRY(line_shape<real>(rows, n, 1, 1, true, &sh));
  static DeviceSet done2{0}, done1{0};
  SG_TRY(allow_lines(k_field_rows<real, true>, done2, sh.smem));
  CombineFinal f = fin;
  if (dim == 3) f.active = 0;
  SG_CUDA(launch_pdl(k_field_rows<real, true>, dim3(sh.blocks), dim3(sh.threads), sh.smem, s, W, W + hs, n, sh.C, tw,
                     sh.tw_smem, Ehi, stride, 0, partials, 0, f));
  SG_CHECK_LAUNCH();
  if (dim == 3) {
    const int part0 = (int)sh.blocks;
    SG_TRY(line_shape<real>(rows / 2, n, 1, 1, true, &sh));
    SG_TRY(allow_lines(k_field_rows<real, false>, done1, sh.smem));
    SG_CUDA(launch_pdl(k_field_rows<real, false>, dim3(sh.blocks), dim3(sh.threads), sh.smem, s, W + 2 * hs, W, n, sh.C,
                       tw, sh.tw_smem, Ehi, stride, 2, partials, part0, fin));
    SG_CHECK_LAUNCH();
  }
  return SG_OK;
}
template int launch_regular_solve<float>(const float*, cplx<float>*, cplx<float>*, const float*, const cplx<float>*,
                                         int, int, float*, int, double*, const CombineFinal&, cudaStream_t);
template int launch_regular_solve<double>(const double*, cplx<double>*, cplx<double>*, const double*,
                                          const cplx<double>*, int, int, double*, int, double*, const CombineFinal&,
                                          cudaStream_t);

template <typename real>
int launch_estimator(const real* rho, cplx<double>* Z, cplx<double>* W, int wcount, int dim, int n,
                     const double* kfac, double frac, const int* masks, int nmask, bool paper,
                     const cplx<double>* tw, double* out, cudaStream_t s) {
  const size_t hs = half_spectrum(dim, n);
  double *vmax = out + 8, *m2max = out + 9;
  SG_CUDA(cudaMemsetAsync(out, 0, 10 * sizeof(double), s));
  SG_TRY(rows_forward<real, double>(rho, Z, dim, n, 1.0 / (double)((size_t)1 << (dim * n)), tw, vmax, s));
  for (int ax = 1; ax < dim; ++ax)
    SG_TRY(columns<double>(Z, dim, n, ax, false, 1, 0, tw, vmax, ax == dim - 1 ? m2max : nullptr, s));
  EstArgs e;
  for (int m = 0; m < 3; ++m) e.kf.k[m] = m < dim ? kfac[m] : 0.0;
  e.frac = frac;
  e.vmax = vmax;
  e.m2max = m2max;
  e.wstride = hs;
  if (!paper) {
    e.nmask = nmask;
    for (int q = 0; q < nmask; ++q) e.mask[q] = masks[q];
    SG_CUDA(launch_pdl(k_est_modes, dim3((unsigned)std::min<size_t>(304, (hs + 255) / 256)), dim3(256), 0, s, Z, dim, n, e, out));
    SG_CHECK_LAUNCH();
    return SG_OK;
  }
  Shape sh;
  static DeviceSet done{0}, done2{0};
  for (int q0 = 0; q0 < nmask; q0 += wcount) {  // as many masks at a time as W holds
    e.nmask = std::min(wcount, nmask - q0);
    for (int q = 0; q < e.nmask; ++q) e.mask[q] = masks[q0 + q];
    const long long lines = (long long)((1 << n) / 2 + 1) << ((dim - 2) * n);
    SG_TRY(line_shape<double>(lines, n, 2, 1, false, &sh));
    SG_TRY(allow_lines(k_est_columns, done, sh.smem));
    SG_CUDA(launch_pdl(k_est_columns, dim3(sh.blocks, e.nmask), dim3(sh.threads), sh.smem, s, Z, W, column_args<double>(dim, n, dim - 1, sh), e, tw));
    SG_CHECK_LAUNCH();
    if (dim == 3) SG_TRY(columns<double>(W, dim, n, 1, true, e.nmask, hs, tw, nullptr, nullptr, s));
    SG_TRY(line_shape<double>(1ll << ((dim - 1) * n - 1), n, 1, 1, true, &sh));
    SG_TRY(allow_lines(k_est_rows, done2, sh.smem));
    SG_CUDA(launch_pdl(k_est_rows, dim3(sh.blocks, e.nmask), dim3(sh.threads), sh.smem, s, W, hs, n, sh.C, tw, sh.tw_smem, out + q0));
    SG_CHECK_LAUNCH();
  }
  return SG_OK;
}
template int launch_estimator<float>(const float*, cplx<double>*, cplx<double>*, int, int, int, const double*, double,
                                     const int*, int, bool, const cplx<double>*, double*, cudaStream_t);
template int launch_estimator<double>(const double*, cplx<double>*, cplx<double>*, int, int, int, const double*,
                                      double, const int*, int, bool, const cplx<double>*, double*, cudaStream_t);

}  // namespace sg
