// Batched spectral Poisson solves over all component grids (Section 2:
// -Laplace phi = rho, E = -grad phi; spectral discretisation).
//
// Each grid's 2D/3D transform is split into passes of 1D radix-2 FFTs along
// one axis; one launch per pass covers every line of every component grid
// of the run.  A block stages a few lines in
// shared memory, transforms them with an iterative decimation-in-time FFT
// (bit-reversed load, natural-order result) and writes them back.  The last
// forward axis is fused with the spectral multiply
//   phi^ = rho^ / |k|^2 (k = 0 -> 0),  E^_m = -i k_m phi^ (Nyquist of axis m -> 0)
// and the first inverse axis of every field component.
#include "sg_fft.cuh"

namespace sg {

// element (line L, position t) -> array offset for lines along an axis whose
// stride is 2^ls in an array of power-of-two extents (line length 2^logn).
__device__ __forceinline__ long long line_addr(long long L, int t, int ls, int logn) {
  return (L & ((1ll << ls) - 1)) + (((long long)t + ((L >> ls) << logn)) << ls);
}

__device__ __forceinline__ int sfreq(int i, int N) { return i < (N >> 1) ? i : i - N; }

// Lines per block (C) are a power of two dividing the line count; for lines
// along axis > 0 consecutive threads take consecutive lines so that strided
// columns are read together.
template <typename real>
__global__ void __launch_bounds__(FFT_BLOCK_VALUES / 2) k_fft_pass(int kind, SolveArena<real> a, const FftJob* __restrict__ jobs,
                                                  int njobs) {
  extern __shared__ unsigned char smem_raw[];
  const int b = blockIdx.x;
  pdl_trigger();
  const int j = find_job(jobs, njobs);  // job and grid tables are written once, at set-up
  const FftJob& J = jobs[j];
  const GridDesc g = a.grids[J.grid];
  const int logn = J.logn;
  const int len = 1 << logn;
  const int C = J.lines_per_block;
  const int logC = __ffs(C) - 1;
  const int line0 = (b - J.block_begin) * C;
  const int nl = C;
  // twiddles staged in shared memory, then the two line buffers
  cplx<real>* tws = reinterpret_cast<cplx<real>*>(smem_raw);
  const int ntw = twiddle_count(a.log_nmax);
  for (int e = threadIdx.x; e < ntw; e += blockDim.x) tws[e] = a.tw[e];
  pdl_wait();  // the previous pass's output
  cplx<real>* buf0 = tws + ntw;
  cplx<real>* buf1 = buf0 + fpad_size((size_t)C * len);
  int ls = 0;
  for (int m = 0; m < J.axis; ++m) ls += __ffs(J.dims[m]) - 1;
  const size_t S = a.S;
  const bool contiguous = (J.axis == 0);
  const int total = nl << logn;

  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    const int li = contiguous ? (e >> logn) : (e & (nl - 1));
    const int t = contiguous ? (e & (len - 1)) : (e >> logC);
    const long long off = line_addr(line0 + li, t, ls, logn);
    cplx<real> v;
    if (kind == FFT_FWD_FIRST) {
      v.x = a.rho[g.offset + off];
      v.y = (real)0;
    } else if (kind == FFT_FWD_MID || kind == FFT_LAST) {
      v = a.A[g.offset + off];
    } else {
      v = a.B[(size_t)J.comp * S + g.offset + off];
    }
    buf0[fpad((li << logn) + bitrev(t, logn))] = v;
  }
  __syncthreads();
  const bool inverse = (kind == FFT_INV_MID || kind == FFT_INV_LAST);
  fft_smem<real>(buf0, nl, logn, inverse, tws);

  if (kind == FFT_LAST) {
    const int D = a.dim;
    const real norm = (real)1 / (real)g.size;
    const int l0 = __ffs(J.dims[0]) - 1;
    for (int p = 0; 2 * p < D; ++p) {
      const int ma = 2 * p, mb = 2 * p + 1;  // mb == D: no second component
      for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int li = e >> logn, t = e & (len - 1);
        const int L = line0 + li;  // combined index of the axes before the last
        int idx[3];
        idx[D - 1] = t;
        if (D == 2) {
          idx[0] = L;
        } else {
          idx[0] = L & (J.dims[0] - 1);
          idx[1] = L >> l0;
        }
        real k2 = 0, ka = 0, kb = 0;
        bool nyq_a = false, nyq_b = false;
        for (int q = 0; q < D; ++q) {
          const int Nq = J.dims[q];
          const real kq = (real)g.kfac[q] * (real)sfreq(idx[q], Nq);  // no FP64 on the FP32 path
          k2 += kq * kq;
          if (q == ma) {
            ka = kq;
            nyq_a = (idx[q] == (Nq >> 1));
          }
          if (q == mb) {
            kb = kq;
            nyq_b = (idx[q] == (Nq >> 1));
          }
        }
        const cplx<real> r = buf0[fpad((li << logn) + t)];
        // E^_m = -i k_m rho^ / |k|^2 : (x + iy) -> (y, -x) * k_m / |k|^2
        cplx<real> out = {(real)0, (real)0};
        if (k2 != (real)0) {
          const real inv = norm / k2;
          if (!nyq_a) {
            const real fa = ka * inv;
            out.x += r.y * fa;
            out.y -= r.x * fa;
          }
          if (mb < D && !nyq_b) {  // + i E^_b: (y, -x) * fb times i -> (x, y) * fb
            const real fb = kb * inv;
            out.x += r.x * fb;
            out.y += r.y * fb;
          }
        }
        buf1[fpad((li << logn) + bitrev(t, logn))] = out;
      }
      __syncthreads();
      fft_smem<real>(buf1, nl, logn, true, tws);
      for (int e = threadIdx.x; e < total; e += blockDim.x) {
        const int li = contiguous ? (e >> logn) : (e & (nl - 1));
        const int t = contiguous ? (e & (len - 1)) : (e >> logC);
        const long long off = line_addr(line0 + li, t, ls, logn);
        a.B[(size_t)p * S + g.offset + off] = buf1[fpad((li << logn) + t)];
      }
      __syncthreads();
    }
    return;
  }

  for (int e = threadIdx.x; e < total; e += blockDim.x) {
    const int li = contiguous ? (e >> logn) : (e & (nl - 1));
    const int t = contiguous ? (e & (len - 1)) : (e >> logC);
    const long long off = line_addr(line0 + li, t, ls, logn);
    const cplx<real> v = buf0[fpad((li << logn) + t)];
    if (kind == FFT_FWD_FIRST || kind == FFT_FWD_MID) {
      a.A[g.offset + off] = v;
    } else if (kind == FFT_INV_MID) {
      a.B[(size_t)J.comp * S + g.offset + off] = v;
    } else {  // FFT_INV_LAST: real part -> component 2p, imaginary -> 2p + 1 (none: zero)
      const bool two = 2 * J.comp + 1 < a.dim;
      const long long at = a.dim == 2 ? off - t + line_pos(t, logn, a.log_nmax) : off;  // the axis is x
      reinterpret_cast<cplx<real>*>(a.E)[(g.offset + at) * ((a.dim + 1) / 2) + J.comp] = {v.x, two ? v.y : (real)0};
    }
  }
}

template <typename real>
int launch_fft_pass(int kind, const SolveArena<real>& a, const FftJob* jobs_dev, int njobs, int nblocks,
                    int smem_bytes, cudaStream_t s) {
  if (njobs == 0 || nblocks == 0) return SG_OK;
  static DeviceSet allowed{0};
  SG_TRY(allow_smem(k_fft_pass<real>, allowed, 200 * 1024));
  SG_CUDA(launch_pdl(k_fft_pass<real>, dim3(nblocks), dim3(FFT_BLOCK_VALUES / 2),
                     smem_bytes + (size_t)twiddle_count(a.log_nmax) * sizeof(cplx<real>), s, kind, a, jobs_dev,
                     njobs));
  SG_CHECK_LAUNCH();
  return SG_OK;
}

// ---------------------------------------------------------------- one block per grid
//
// When every component grid fits in shared memory (twice in 3D: spectrum and
// one pair of field components), one launch solves all of them: a block loads
// its grid, transforms it along every axis in place, forms the E^_m and
// transforms them back.  Forward transforms decimate in frequency (natural
// order in, bit-reversed out) and inverse ones in time (bit-reversed in,
// natural out), so no pass reorders anything: the spectral step reads the
// frequency of a position by reversing its bits.  Both take their stages in
// pairs (radix 2^2), half the passes over shared memory and barriers.
// Bound: latency (one block per grid, one barrier per pass).  With
// profiling events, with single stages and bit-reversal passes -> now: 2D
// n = 10 18.4 -> 12.3 us, n = 8 10.2 -> 8.2, 3D n = 7 14.3 -> 10.3.  Half a
// grid of threads: a quarter took 12.3 us in 3D, the same in 2D.
//
// Element (o, t, i) of axis ax at ((o << logn) + t) << ls | i; consecutive
// work items take consecutive inner indices i (the axes below ax, contiguous
// in the buffer), then the butterflies of one line, then the outer lines, so
// that a warp's accesses are contiguous along every axis.
template <typename real, bool INV>
__device__ __forceinline__ void fft_axis(cplx<real>* buf, int S, int logn, int ls, const cplx<real>* __restrict__ tw) {
  const int smask = (1 << ls) - 1;
  auto radix2 = [&]() {  // span 2, no twiddle
    for (int j = threadIdx.x; j < (S >> 1); j += blockDim.x) {
      const int i0 = ((j >> ls) << (ls + 1)) + (j & smask), i1 = i0 + (1 << ls);
      const cplx<real> a = buf[i0], b = buf[i1];
      buf[i0] = {a.x + b.x, a.y + b.y};
      buf[i1] = {a.x - b.x, a.y - b.y};
    }
    __syncthreads();
  };
  if (INV && (logn & 1)) radix2();
  for (int k = INV ? (logn & 1) : logn - 2; INV ? k + 1 < logn : k >= 0; k += INV ? 2 : -2) {
    const int q = 1 << k, st = q << ls;  // elements t, t + q, t + 2q, t + 3q
    for (int j = threadIdx.x; j < (S >> 2); j += blockDim.x) {
      const int p = j >> ls;  // butterfly: (outer, group, position)
      const int pos = p & (q - 1);
      const int i0 = ((((p >> k) << (k + 2)) + pos) << ls) + (j & smask);
      cplx<real> w1 = tw[twiddle_index(q, pos)], w2 = tw[twiddle_index(2 * q, pos)];  // W_{2q}^pos, W_{4q}^pos
      const cplx<real> a0 = buf[i0], a1 = buf[i0 + st], a2 = buf[i0 + 2 * st], a3 = buf[i0 + 3 * st];
      cplx<real> x0, x1, x2, x3;
      if constexpr (INV) {
        w1.y = -w1.y;
        w2.y = -w2.y;
        const cplx<real> w3 = {-w2.y, w2.x};  // W_{4q}^(pos + q), conjugated
        cplx<real> b0, b1, b2, b3;
        butterfly(a0, a1, w1, b0, b1);
        butterfly(a2, a3, w1, b2, b3);
        butterfly(b0, b2, w2, x0, x2);
        butterfly(b1, b3, w3, x1, x3);
      } else {
        const cplx<real> w3 = {w2.y, -w2.x};  // W_{4q}^(pos + q)
        const cplx<real> b0 = {a0.x + a2.x, a0.y + a2.y}, b1 = {a1.x + a3.x, a1.y + a3.y};
        const cplx<real> b2 = cmul<real>({a0.x - a2.x, a0.y - a2.y}, w2), b3 = cmul<real>({a1.x - a3.x, a1.y - a3.y}, w3);
        x0 = {b0.x + b1.x, b0.y + b1.y};
        x1 = cmul<real>({b0.x - b1.x, b0.y - b1.y}, w1);
        x2 = {b2.x + b3.x, b2.y + b3.y};
        x3 = cmul<real>({b2.x - b3.x, b2.y - b3.y}, w1);
      }
      buf[i0] = x0;
      buf[i0 + st] = x1;
      buf[i0 + 2 * st] = x2;
      buf[i0 + 3 * st] = x3;
    }
    __syncthreads();
  }
  if (!INV && (logn & 1)) radix2();
}

// One block solves grid gi of arena a: load, forward transforms, E^_m,
// paired inverse transforms, store.
template <typename real>
__device__ __forceinline__ void solve_grid_block(const SolveArena<real>& a, int gi, int max_size) {
  extern __shared__ unsigned char smem_raw[];
  const GridDesc g = a.grids[gi];
  const int D = a.dim;
  const int l0 = g.l[0], l1 = g.l[1], l2 = D == 3 ? g.l[2] : 0;
  const int S = g.size;
  cplx<real>* A = reinterpret_cast<cplx<real>*>(smem_raw);
  cplx<real>* tws = A + (size_t)(D == 3 ? 2 : 1) * max_size;  // twiddles of the grid's longest axis
  const int ntw = twiddle_count(max(l0, max(l1, l2)));
  for (int e = threadIdx.x; e < ntw; e += blockDim.x) tws[e] = a.tw[e];
  pdl_wait();  // the component densities
  for (int e = threadIdx.x; e < S; e += blockDim.x) A[e] = {a.rho[g.offset + e], (real)0};
  __syncthreads();
  fft_axis<real, false>(A, S, l0, 0, tws);
  fft_axis<real, false>(A, S, l1, l0, tws);
  if (D == 3) fft_axis<real, false>(A, S, l2, l0 + l1, tws);
  const real norm = (real)1 / (real)S;
  const int n0 = 1 << l0, n1 = 1 << l1;
  // Field components in pairs: B = E^_a + i E^_b, one inverse transform,
  // E_a its real part and E_b its imaginary part (both fields are real).
  // The last pair takes the spectrum's place.
  const int np = (D + 1) / 2;
  for (int pr = 0; pr < np; ++pr) {
    const int ma = 2 * pr, mb = 2 * pr + 1;
    cplx<real>* B = pr == np - 1 ? A : A + max_size;
    for (int e = threadIdx.x; e < S; e += blockDim.x) {
      const int idx[3] = {bitrev(e & (n0 - 1), l0), bitrev((e >> l0) & (n1 - 1), l1),
                          D == 3 ? bitrev(e >> (l0 + l1), l2) : 0};
      const int sizes[3] = {n0, n1, 1 << l2};
      real k2 = 0, ka = 0, kb = 0;
      bool nyq_a = false, nyq_b = false;
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        if (q >= D) break;
        const int Nq = sizes[q];
        const real kq = (real)g.kfac[q] * (real)sfreq(idx[q], Nq);
        k2 += kq * kq;
        if (q == ma) {
          ka = kq;
          nyq_a = idx[q] == (Nq >> 1);
        }
        if (q == mb) {
          kb = kq;
          nyq_b = idx[q] == (Nq >> 1);
        }
      }
      const cplx<real> r = A[e];
      cplx<real> out = {(real)0, (real)0};
      if (k2 != (real)0) {
        const real inv = norm / k2;
        if (!nyq_a) {  // E^_a = -i k_a rho^ / |k|^2
          const real fa = ka * inv;
          out.x += r.y * fa;
          out.y -= r.x * fa;
        }
        if (mb < D && !nyq_b) {  // + i E^_b
          const real fb = kb * inv;
          out.x += r.x * fb;
          out.y += r.y * fb;
        }
      }
      B[e] = out;
    }
    __syncthreads();
    if (D == 3) fft_axis<real, true>(B, S, l2, l0 + l1, tws);
    fft_axis<real, true>(B, S, l1, l0, tws);
    fft_axis<real, true>(B, S, l0, 0, tws);
    for (int e = threadIdx.x; e < S; e += blockDim.x) {
      const int x = e & (n0 - 1);
      const int at = D == 2 ? e - x + line_pos(x, l0, a.log_nmax) : e;
      reinterpret_cast<cplx<real>*>(a.E)[(size_t)(g.offset + at) * np + pr] = {B[e].x, mb < D ? B[e].y : (real)0};
    }
    __syncthreads();
  }
}

// Shared memory and threads of the one-block solve.
template <typename real>
static size_t solve_block_smem(int dim, int max_size, int max_log) {
  return ((size_t)(dim == 3 ? 2 : 1) * max_size + (size_t)twiddle_count(max_log)) * sizeof(cplx<real>);
}
static int solve_block_threads(int max_size) {
  const int t = max_size / 2;
  return t < 64 ? 64 : (t > 1024 ? 1024 : t);
}

template <typename real>
__global__ void __launch_bounds__(1024) k_solve_small(SolveArena<real> a, int max_size, int grid0) {
  pdl_trigger();
  solve_grid_block<real>(a, grid0 + blockIdx.x, max_size);
}

// The cross-run solve: block b takes job b, a grid of one of the runs.
template <typename real>
__global__ void __launch_bounds__(1024) k_solve_batch(const SolveJob<real>* __restrict__ jobs, int max_size) {
  const SolveJob<real>& J = jobs[blockIdx.x];
  const SolveArena<real> a = J.a;
  solve_grid_block<real>(a, J.grid, max_size);
}

template <typename real>
int launch_solve_small(const SolveArena<real>& a, int ngrids, int max_size, cudaStream_t s, int grid0) {
  if (ngrids == 0) return SG_OK;
  const int threads = solve_block_threads(max_size);
  const size_t smem = solve_block_smem<real>(a.dim, max_size, a.log_nmax);
  static DeviceSet allowed{0};
  SG_TRY(allow_smem(k_solve_small<real>, allowed, 200 * 1024));
  SG_CUDA(launch_pdl(k_solve_small<real>, dim3(ngrids), dim3(threads), smem, s, a, max_size, grid0));
  SG_CHECK_LAUNCH();
  return SG_OK;
}

template int launch_solve_small<float>(const SolveArena<float>&, int, int, cudaStream_t, int);
template int launch_solve_small<double>(const SolveArena<double>&, int, int, cudaStream_t, int);

template <typename real>
int launch_solve_batch(const SolveJob<real>* jobs, int njobs, int max_size, int max_log, cudaStream_t s) {
  if (njobs == 0) return SG_OK;
  if (max_size > small_solve_max<real>()) {
    set_error("cross-run solve: a component grid is larger than one block's shared memory takes");
    return SG_ERR_UNSUPPORTED;
  }
  const int threads = solve_block_threads(max_size);
  const size_t smem = solve_block_smem<real>(3, max_size, max_log);  // runs of either dimension
  static DeviceSet allowed{0};
  SG_TRY(allow_smem(k_solve_batch<real>, allowed, 200 * 1024));
  k_solve_batch<real><<<njobs, threads, smem, s>>>(jobs, max_size);
  SG_CHECK_LAUNCH();
  return SG_OK;
}
template int launch_solve_batch<float>(const SolveJob<float>*, int, int, int, cudaStream_t);
template int launch_solve_batch<double>(const SolveJob<double>*, int, int, int, cudaStream_t);

template int launch_fft_pass<float>(int, const SolveArena<float>&, const FftJob*, int, int, int, cudaStream_t);
template int launch_fft_pass<double>(int, const SolveArena<double>&, const FftJob*, int, int, int, cudaStream_t);

}  // namespace sg
