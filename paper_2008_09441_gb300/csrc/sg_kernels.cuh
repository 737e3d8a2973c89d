// Launchers of the library's device kernels (host side).  Every launcher
// enqueues on the given stream and returns an SG_* status.
#pragma once

#include <cmath>
#include <vector>

#include "sg_common.cuh"

namespace sg {

// ---------------------------------------------------------------- sort
constexpr int RS_THREADS = 512;
constexpr int RS_ITEMS = 8;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;  // keys per tile

// keys[i] = Morton key of particle i's level-n cell.
template <typename real, int D>
int launch_keys(const PArrays<real, D>& p, size_t np, int n, uint32_t* keys, unsigned* status, cudaStream_t s);

// The stand-alone cell sort of positions u (dim device arrays in the given
// precision): sorted keys, stable permutation, counts per cell (may be NULL).
// scratch: cell_sort_words(n) u32 words.
size_t cell_sort_words(size_t n);
int cell_sort(int precision, int dim, int level, size_t n, const void* const* u, uint32_t* keys_sorted, uint32_t* perm,
              uint32_t* counts, uint32_t* scratch, cudaStream_t s);

// dst[pid[i]] = src[i] for every particle array (back to the original order;
// dst's pid is not used).  scratch: unpermute_scratch_bytes(np) bytes aligned
// to 32, or nullptr for the direct scatter.
template <typename real, int D>
int launch_unpermute(const PArrays<real, D>& src, const PArrays<real, D>& dst, size_t np, void* scratch,
                     cudaStream_t s);
template <typename real, int D>
size_t unpermute_scratch_bytes(size_t np);

// counts[key] += 1 for every key (counts zeroed by the caller); sorted: the
// keys are in order.
int launch_counts(const uint32_t* keys, size_t np, uint32_t* counts, cudaStream_t s, bool sorted);

// Exclusive scan of m u32 values (out may equal in).
int exclusive_scan_u32(const uint32_t* in, uint32_t* out, size_t m, uint32_t* block_sums,
                       cudaStream_t s);
size_t scan_block_sums_words(size_t m);

// ---------------------------------------------------------------- deposit
// Particles per thread: eight share the chunk's per-thread work (anchor, box,
// barriers); four on twice the threads and sixteen on half as many were slower
// (3D two-stream, 8,388,608 particles: 93.8 and 96.4 against 90.0 us, with
// the flush's divisions as multiplications in all three; with real divisions
// and four 102.7).  Small runs take 128 threads and four.
constexpr int DEP_THREADS = 256;
constexpr int DEP_ITEMS = 8;
constexpr int DEP_SMALL_THREADS = 128;
constexpr int DEP_SMALL_ITEMS = 4;
constexpr int DEP_CHUNK = DEP_THREADS * DEP_ITEMS;

// scale / inv_scale: the FP32 fixed-point scale of the window (WinAcc), 1 for FP64.
// shift: position of node 0 in cells (0 node-centred, 1/2 cell-centred).
template <typename real, int D>
int launch_deposit(const PArrays<real, D>& p, size_t np, int n, real inv_cell_vol, real* rho,
                   int win_cap_nodes, real scale, real inv_scale, real shift, cudaStream_t s);

// The upload's statistics, out[0 .. 2 nb]: per-block FP64 charge sums, per-
// block max |q|, then the status word (its bits in a double).
template <typename real>
int launch_charge_stats(const real* w, size_t n, const unsigned* status, double* out, int nblocks, cudaStream_t s);


// ---------------------------------------------------------------- line passes
// The lines of one array along one axis, processed by one kernel launch
// together with the other jobs of the same pass.
constexpr int RJ_LEVELS = 13;  // levels 0..12 (2D n <= 12, 3D n <= 8)
struct LineJob {
  const void* src;       // [outer][2^top][inner] reals
  int top;               // log2 of the line length
  int outer, inner;      // powers of two; lines = outer * inner
  int block_begin;       // first block of this job in the launch
  int tile_stride;       // reals per tile row in shared memory (inner > 1)
  int tmask;             // bit l set: level l is written
  int tmin;              // lowest level written
  int sub_mean;          // 1: the source is the regular grid; the mean is subtracted as it is read
  void* dst[RJ_LEVELS];  // level l: [outer][2^l][inner]
};

// Block -> job of a pass: the last job whose block_begin <= blockIdx.x.  The
// first warp reads 32 job headers at a time (no chain of dependent loads).
template <typename Job>
__device__ __forceinline__ int find_job(const Job* __restrict__ jobs, int njobs) {
  __shared__ int s_job;
  const int b = blockIdx.x;
  if (threadIdx.x < 32) {
    int best = 0;
    for (int base = 0; base < njobs; base += 32) {
      const int idx = base + (int)threadIdx.x;
      const bool le = idx < njobs && jobs[idx].block_begin <= b;
      const unsigned m = __ballot_sync(0xffffffffu, le);
      if (m) best = base + 31 - __clz(m);
      if (m != 0xffffffffu) break;
    }
    if (threadIdx.x == 0) s_job = best;
  }
  __syncthreads();
  return s_job;
}

// Restriction along one axis of every job's lines (full weighting 1/4,
// 1/2, 1/4 per level halving, the exact form of R along one axis for nested
// node-centred grids; cell = true: R of cell-centred grids through the
// face-averaged cascade), outputs in the natural layout.  Jobs that read
// the regular grid subtract `mean` (Q / |box|) from every value they read:
// the component densities are stored as deviations from the mean, which
// every R_i preserves (its weights sum to one), so that FP32 rounding in the
// restriction sums, in storage and in the transforms is relative to the
// density's fluctuation instead of its much larger uniform part.
template <typename real>
int launch_restrict_pass(const LineJob* jobs_dev, int njobs, int nblocks, int lines_per_block, int vpl,
                         int smem_bytes, bool cell, real mean, cudaStream_t s);

// 3D: x and y restricted plane by plane in one launch.  dst[l_1][l_2]: the
// array [z][2^l_2][2^l_1] of a level pair, or nullptr; lx_min / ly_min: the
// lowest levels needed.
constexpr int RJ_PLANE_LEVELS = 9;  // 3D levels 0..8
constexpr int RJ_PLANE_SMEM = 220 * 1024;
struct PlaneTargets {
  int lx_min, ly_min;
  void* dst[RJ_PLANE_LEVELS][RJ_PLANE_LEVELS];
};
template <typename real>
size_t restrict_planes_smem(int n, int lx_min, bool cell);
template <typename real>
int launch_restrict_planes(const real* rho, const PlaneTargets* tgt, int n, int lx_min, bool cell, real mean,
                           cudaStream_t s);

// FFT passes over the component grids.
enum FftKind { FFT_FWD_FIRST = 0, FFT_FWD_MID = 1, FFT_LAST = 2, FFT_INV_MID = 3, FFT_INV_LAST = 4 };

struct FftJob {
  int grid;          // index into the grid table
  int dims[3];
  int axis;
  int logn;
  int lines;
  int lines_per_block;
  int block_begin;
  int comp;          // inverse passes: component pair (2 comp, 2 comp + 1)
};

// FFT twiddles, stage-major: the butterflies of span 2h (h = 1, 2, 4, ...)
// use W_{2h}^p = exp(-2 pi i p / (2h)) for p < h, stored at h - 1 + p, so
// that consecutive butterflies of a stage read consecutive entries.  A table
// for transforms of up to 2^L points holds 2^L - 1 entries.
__host__ __device__ constexpr int twiddle_index(int h, int p) { return h - 1 + p; }
__host__ __device__ constexpr int twiddle_count(int L) { return L < 1 ? 1 : (1 << L) - 1; }
template <typename real>
std::vector<cplx<real>> make_twiddles(int L) {
  std::vector<cplx<real>> tw((size_t)twiddle_count(L));
  tw[0] = {(real)1, (real)0};
  for (int h = 1; h < (1 << L); h <<= 1)
    for (int p = 0; p < h; ++p) {
      const double a = M_PI * (double)p / (double)h;
      tw[(size_t)twiddle_index(h, p)] = {(real)std::cos(a), (real)(-std::sin(a))};
    }
  return tw;
}

template <typename real>
struct SolveArena {
  const GridDesc* grids;
  const real* rho;     // S
  cplx<real>* A;       // S
  cplx<real>* B;       // (D + 1) / 2 * S
  real* E;             // ec_stride * S: node-interleaved components (3D: a zero fourth)
  size_t S;
  const cplx<real>* tw;  // make_twiddles(log_nmax)
  int log_nmax;
  int dim;
};

// Complex values per block of a transform pass (whole lines, at least one
// line per block); the block has half as many threads.
constexpr int FFT_BLOCK_VALUES = 1024;

template <typename real>
int launch_fft_pass(int kind, const SolveArena<real>& a, const FftJob* jobs_dev, int njobs,
                    int nblocks, int smem_bytes, cudaStream_t s);

// All component grids in one launch, one block per grid, whole grid in shared
// memory (used when every grid has at most SMALL_SOLVE_MAX<real> points).
template <typename real>
int launch_solve_small(const SolveArena<real>& a, int ngrids, int max_size, cudaStream_t s, int grid0 = 0);
template <typename real>
constexpr int small_solve_max() { return sizeof(real) == 4 ? 4096 : 2048; }

// One component grid of one run for the cross-run solve: the run's arena
// and the grid's index in it.  A launch over a table of these solves the
// component grids of every run in it, one block per (run, grid).
template <typename real>
struct SolveJob {
  SolveArena<real> a;
  int grid;
  int pad;
};
// max_size: largest grid of the table (points); max_log: largest log_nmax.
template <typename real>
int launch_solve_batch(const SolveJob<real>* jobs, int njobs, int max_size, int max_log, cudaStream_t s);

// Device diagnostics record updated at the end of each step.
struct DevDiag {
  double field_energy;
  double field_energy_prev;
  double kinetic_energy;
  unsigned long long checksum;
  unsigned status;
  unsigned pad;
};

// Step bookkeeping closed by the last block of the kernel that writes the field:
// field energy from the per-row partials (scaled by fe_scale), the previous
// field energy, and the kinetic energy from the push partials when given.
struct CombineFinal {
  int active;
  int n_ke;
  const double* ke_partials;
  double fe_scale;
  DevDiag* dd;
  unsigned* counter;  // zero between launches; the last block resets it
};

// ---------------------------------------------------------------- regular-grid spectral work
// Complex values of a half spectrum (k_x = 0 .. N/2) of the regular grid.
size_t half_spectrum(int dim, int n);
// The filter mode's regular-grid solve: rho_f -> E on the regular nodes
// (E_hi node-interleaved with `stride`), closing the step's FP64 bookkeeping as `fin` says.  rho_f is the combination of the
// component densities, a deviation from the mean like them.  Z and W hold
// one and `dim` half spectra, partials 3/2 2^(n (dim - 1)) values.
template <typename real>
int launch_regular_solve(const real* rho_f, cplx<real>* Z, cplx<real>* W, const real* ktab, const cplx<real>* tw,
                         int dim, int n, real* Ehi, int stride, double* partials, const CombineFinal& fin,
                         cudaStream_t s);
// Algorithm 1's reductions (FP64) of the density rho: out[q] of each mask q (bit m:
// the factor k_m^2), with the spectrum thresholded at frac max|rho^|: the
// largest |value| of the inverse transform (paper) or of the modes; out[8] =
// max|rho|.  out holds 10 values; Z one half spectrum, W wcount of them.
template <typename real>
int launch_estimator(const real* rho, cplx<double>* Z, cplx<double>* W, int wcount, int dim, int n,
                     const double* kfac, double frac, const int* masks, int nmask, bool paper,
                     const cplx<double>* tw, double* out, cudaStream_t s);

// ---------------------------------------------------------------- combine
// Place of node x of a level-l line in the arrays the line kernel reads (2D:
// the component fields, 3D: the planes).  A thread of that kernel
// takes CB_RUN consecutive nodes of a level-n line and half as many one
// level below; node j of every thread's run is stored next to the other
// threads' node j, so that a warp's loads are consecutive.
constexpr int CB_RUN = 4;
__host__ __device__ __forceinline__ int line_pos(int x, int l, int n) {
  return l == n ? ((x & 3) << (l - 2)) + (x >> 2) : l == n - 1 ? ((x & 1) << (l - 1)) + (x >> 1) : x;
}
// The arrays the line kernel combines: the component grids, in 3D those of a
// plane (PlaneArray), the z axis already prolonged.  Grouped by x level: start[l] .. start[l+1] have
// l_1 = l; start[l] for l > n holds the count.
constexpr int CB_MAX_GRIDS = 128;
struct LineGrid {
  int lx, ly, off, coeff;
};
struct LevelStarts {
  int start[18];
};
// 3D: the grids that make one array of a plane, and its place there.  FP32:
// one grid; double sums: the up to three that share l_1 and l_2.
struct PlaneArray {
  int off, logs, lx, ng;  // offset in the plane, l_1 + l_2, l_1, number of grids
  int goff[3], lz[3], coeff[3];
  int pad[3];
};
struct CombineTables {
  const LineGrid* lines = nullptr;
  LevelStarts ls{};
  int lmin = 0;  // smallest x level
  // 3D only
  const PlaneArray* planes = nullptr;
  int S2 = 0;  // values of one plane and component
  void* scratch = nullptr;
  size_t scratch_bytes = 0;
};

// ---------------------------------------------------------------- push
// The combined field the push gathers from is stored node-interleaved:
// E_hi[node * ec_stride<D>() + m] (2D: (E_x, E_y); 3D: (E_x, E_y, E_z, pad)),
// so one corner of the gather is one 8- or 16-byte load.  The low parts of
// the FP32 path's float pairs are planes E_lo[m * N_c + node].
template <int D>
constexpr int ec_stride() { return D == 2 ? 2 : 4; }

template <typename real>
struct PushParams {
  real qm, dt;
  real ke_fac;    // 1 / (2 q/m): kinetic energy 0.5 m_p v.v with m_p = q_p / (q/m)
  real dt_over_L[3];
  real eext[3];   // E_ext,m = eext[m] * (u_m - 1/2)   (eext = Eext_lin * L)
  real tB[3];     // q/m * B * dt / 2 (Boris t vector)
  real sB[3];     // 2 t / (1 + t . t); 2D: only t_z turns the plane's velocities
  int boris;
  int has_eext;
  int drift;      // 0: velocity only (initial half kick), 1: kick + drift
  real shift;     // position of node 0 in cells: 0 node-centred, 1/2 cell-centred
};

// Sort work fused into the push on sort steps (keys == nullptr: none).
struct SortFuse {
  uint32_t* keys = nullptr;        // level-n Morton key per particle (storage order)
  unsigned long long* checksum = nullptr;
};

template <typename real, int D>
int launch_push(const PArrays<real, D>& p, size_t np, int n, const real* Ecomb, PushParams<real> pp,
                double* ke_partials, unsigned* status, const SortFuse& sf, cudaStream_t s, int blocks = 0);
template <typename real, int D>
int push_blocks(size_t np);  // grid of the push (size of its kinetic-energy partials)

// ---------------------------------------------------------------- step sort (tile counting sort)
// Cell keys of the current positions (the push emits them on sort steps; this
// kernel serves init and checkpoint load).  A key's tile is key >> shift.
template <typename real, int D>
int launch_tile_keys(const PArrays<real, D>& p, size_t np, int n, const SortFuse& sf, unsigned* status,
                     cudaStream_t s);
// tile_count[key >> shift] += 1 for every key (counts zeroed by the caller).
int launch_tile_hist(const uint32_t* keys, size_t np, int shift, uint32_t* tile_count, cudaStream_t s);
// Scatter every particle to its tile's slots (cursor = exclusive scan of the
// tile counts): one pass, reads key + payload, writes payload.
template <typename real, int D>
int launch_tile_scatter(const PArrays<real, D>& src, const PArrays<real, D>& dst, const uint32_t* keys, int shift,
                        uint32_t* cursor, size_t np, cudaStream_t s);

// ---------------------------------------------------------------- misc
template <typename real, int D>
int launch_wrap_check(const PArrays<real, D>& p, size_t np, unsigned* status, cudaStream_t s);


// The diagnostics record in one buffer, for one device-to-host copy: *dd at
// 0, *cks at o_cks, *st at o_cks + 8, and V_i sum_k rho_i(x_k) of every grid
// (FP64) from o_ch on (one block per grid).
template <typename real>
int launch_diag_record(const GridDesc* grids, int ngrids, const real* rho, const DevDiag* dd,
                       const unsigned long long* cks, const unsigned* st, void* out, size_t o_cks, size_t o_ch,
                       cudaStream_t s);

// Sum of squares of one thread's field values: floats, every square rounded
// once, in a float pair; doubles plainly.
template <typename real>
struct SquareSum {
  ff v{0.f, 0.f};
  __device__ __forceinline__ void add(float x) {
    const ff s = two_sum(v.hi, __fmul_rn(x, x));
    v = {s.hi, __fadd_rn(v.lo, s.lo)};
  }
  __device__ __forceinline__ double value() const { return (double)v.hi + (double)v.lo; }
};
template <>
struct SquareSum<double> {
  double v = 0.0;
  __device__ __forceinline__ void add(double x) { v = fma(x, x, v); }
  __device__ __forceinline__ double value() const { return v; }
};

// The last block of a field kernel to finish reduces the energy partials (and the push's kinetic-energy partials) in FP64, in a
// fixed order, so the step needs no separate bookkeeping launch.
__device__ __forceinline__ void combine_finalize(const double* partials, int n_part, const CombineFinal& fin,
                                                 double* red) {
  __shared__ int s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    const unsigned t = atomicAdd(fin.counter, 1u);
    s_last = (t == gridDim.x - 1);
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double a = 0.0;
  for (int i = threadIdx.x; i < n_part; i += blockDim.x) a += __ldcg(partials + i);
  const double fe = block_sum_double(a, red);
  double b = 0.0;
  if (fin.ke_partials)
    for (int i = threadIdx.x; i < fin.n_ke; i += blockDim.x) b += __ldcg(fin.ke_partials + i);
  const double ke = block_sum_double(b, red);
  if (threadIdx.x == 0) {
    DevDiag* dd = fin.dd;
    dd->field_energy_prev = dd->field_energy;
    dd->field_energy = fe * fin.fe_scale;
    if (fin.ke_partials) dd->kinetic_energy = ke;
    *fin.counter = 0u;
  }
}

// E: the component fields, node-interleaved (ncomp = D, ec_stride values per
// node), or a density (ncomp = 1); Ehi likewise.
template <typename real, int D>
int launch_combine(const CombineTables& ct, const real* E, int n, real* Ehi, float* Elo, double* energy_partials,
                   const CombineFinal& fin, cudaStream_t s, int ncomp,
                   bool cell,       // cell-centred grids
                   bool fp64_acc);  // FP32 path: accumulate in double instead of float pairs

template <typename real>
int launch_to_double(const real* src, double* dst, size_t n, cudaStream_t s);
// dst[m * nd + node] = E_hi[node * stride + m] (+ E_lo[m * nd + node] when lo != nullptr), FP64.
template <typename real>
int launch_field_to_double(const real* hi, const float* lo, double* dst, size_t nd, int dim, int stride,
                           cudaStream_t s);

}  // namespace sg
