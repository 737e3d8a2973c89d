// Cell-key sorts: the stand-alone stable sort of positions (Morton keys of the
// level-n cells, permutation, per-cell counts; integer work, bit-exact), the
// step's tile counting sort, and the particles' way back to their original
// order.
#include "sg_kernels.cuh"

namespace sg {


// ---------------------------------------------------------------- keys
template <typename real, int D>
__global__ void __launch_bounds__(256) k_keys(PArrays<real, D> p, size_t np, int n, uint32_t* keys, unsigned* status) {
  const int N = 1 << n;
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  int c[D];
  bool bad = false;
#pragma unroll
  for (int m = 0; m < D; ++m) {
    real u = p.u[m][i];
    bad |= !(u >= (real)0 && u < (real)1);
    c[m] = cell_of(u, n, N);
  }
  if (bad) atomicOr(status, ST_KEY_RANGE);
  keys[i] = morton_key<D>(c, n);
}

template <typename real, int D>
int launch_keys(const PArrays<real, D>& p, size_t np, int n, uint32_t* keys, unsigned* status, cudaStream_t s) {
  if (np == 0) return SG_OK;
  k_keys<real, D><<<(unsigned)((np + 255) / 256), 256, 0, s>>>(p, np, n, keys, status);
  SG_CHECK_LAUNCH();
  return SG_OK;
}

// ---------------------------------------------------------------- scan
constexpr int SC_THREADS = 1024;  // short serial runs per thread: the scan is latency-bound
constexpr int SC_ITEMS = 4;
constexpr int SC_TILE = SC_THREADS * SC_ITEMS;

size_t scan_block_sums_words(size_t m) { return (m + SC_TILE - 1) / SC_TILE + 1; }

// Block-wide exclusive scan of SC_TILE values staged in shared memory.
__device__ void block_exclusive_scan_tile(uint32_t* sh, uint32_t* total) {
  __shared__ uint32_t warp_tot[SC_THREADS / 32];
  int t = threadIdx.x;
  uint32_t loc[SC_ITEMS];
  uint32_t run = 0;
#pragma unroll
  for (int j = 0; j < SC_ITEMS; ++j) {
    loc[j] = run;
    run += sh[t * SC_ITEMS + j];
  }
  // inclusive warp scan of per-thread totals
  uint32_t x = run;
  int lane = t & 31, w = t >> 5;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) warp_tot[w] = x;
  __syncthreads();
  if (w == 0) {
    uint32_t v = lane < SC_THREADS / 32 ? warp_tot[lane] : 0;
    uint32_t inc = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t y = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane < SC_THREADS / 32) warp_tot[lane] = inc - v;  // exclusive
    if (lane == SC_THREADS / 32 - 1) *total = inc;
  }
  __syncthreads();
  uint32_t base = warp_tot[w] + (x - run);
#pragma unroll
  for (int j = 0; j < SC_ITEMS; ++j) sh[t * SC_ITEMS + j] = base + loc[j];
  __syncthreads();
}

__global__ void __launch_bounds__(SC_THREADS) k_scan_tiles(const uint32_t* in, uint32_t* out, size_t m,
                                                           uint32_t* block_sums) {
  __shared__ uint32_t sh[SC_TILE];
  __shared__ uint32_t tot;
  size_t base = (size_t)blockIdx.x * SC_TILE;
  for (int j = threadIdx.x; j < SC_TILE; j += SC_THREADS) sh[j] = (base + j < m) ? in[base + j] : 0u;
  __syncthreads();
  block_exclusive_scan_tile(sh, &tot);
  for (int j = threadIdx.x; j < SC_TILE; j += SC_THREADS)
    if (base + j < m) out[base + j] = sh[j];
  if (threadIdx.x == 0) block_sums[blockIdx.x] = tot;
}

// Exclusive scan of up to SC_TILE block sums in one block (repeated tiles if more).
__global__ void __launch_bounds__(SC_THREADS) k_scan_top(uint32_t* block_sums, int nb) {
  __shared__ uint32_t sh[SC_TILE];
  __shared__ uint32_t tot;
  uint32_t carry = 0;
  for (int base = 0; base < nb; base += SC_TILE) {
    for (int j = threadIdx.x; j < SC_TILE; j += SC_THREADS) sh[j] = (base + j < nb) ? block_sums[base + j] : 0u;
    __syncthreads();
    block_exclusive_scan_tile(sh, &tot);
    for (int j = threadIdx.x; j < SC_TILE; j += SC_THREADS)
      if (base + j < nb) block_sums[base + j] = sh[j] + carry;
    __syncthreads();
    carry += tot;
    __syncthreads();
  }
}

__global__ void __launch_bounds__(SC_THREADS) k_scan_add(uint32_t* out, size_t m, const uint32_t* block_sums) {
  size_t base = (size_t)blockIdx.x * SC_TILE;
  uint32_t add = block_sums[blockIdx.x];
  if (add == 0) return;
  for (int j = threadIdx.x; j < SC_TILE; j += SC_THREADS)
    if (base + j < m) out[base + j] += add;
}

int exclusive_scan_u32(const uint32_t* in, uint32_t* out, size_t m, uint32_t* block_sums, cudaStream_t s) {
  if (m == 0) return SG_OK;
  unsigned nb = (unsigned)((m + SC_TILE - 1) / SC_TILE);
  k_scan_tiles<<<nb, SC_THREADS, 0, s>>>(in, out, m, block_sums);
  SG_CHECK_LAUNCH();
  if (nb > 1) {
    k_scan_top<<<1, SC_THREADS, 0, s>>>(block_sums, (int)nb);
    SG_CHECK_LAUNCH();
    k_scan_add<<<nb, SC_THREADS, 0, s>>>(out, m, block_sums);
    SG_CHECK_LAUNCH();
  }
  return SG_OK;
}

// ---------------------------------------------------------------- cell sort
//
// Stable LSD radix sort of (key, input index), the digits of equal width: 20
// key bits take three passes of 7, 7 and 6 bits (the fewest passes of at most
// 8, then the fewest digit values, which makes the runs a tile writes longer).
// Per pass: digit counts of every tile, their scan (one block per digit), and
// the scatter, which orders its tile by digit in shared memory first, so that
// it writes runs of consecutive keys instead of one sector per key.  The first
// count makes the keys from the positions; the last scatter writes the
// caller's arrays.  Bound: L2 (the keys and indices of 4 M positions stay
// there) and the warps' chains of ranking steps.  4,194,304 positions, 2D
// level 10, with the counts: 397 us before (8-bit digits, unordered scatter
// of 89 us a pass, scans of three launches, copies into the result), 132 us
// now (65,537 positions, level 5: 93 -> 58; 3D level 7, 8 M in double: 1017 ->
// 521).
constexpr int RS_WARPS = RS_THREADS / 32;
constexpr int RS_WARP_KEYS = RS_TILE / RS_WARPS;
static_assert(RS_WARP_KEYS == 32 * RS_ITEMS, "one key per lane per chunk");

static size_t cell_sort_tiles(size_t n) { return (n + RS_TILE - 1) / RS_TILE; }
size_t cell_sort_words(size_t n) { return 3 * n + 256 * cell_sort_tiles(n) + 256; }

template <typename real, int D>
struct RawU {
  const real* u[D];
};

// Adds the tile's digits to h and writes them out: hist[digit * ntiles + tile].
__device__ __forceinline__ void store_digits(const uint32_t* h, int bins, uint32_t* hist, size_t ntiles) {
  __syncthreads();
  for (int i = threadIdx.x; i < bins; i += RS_THREADS) hist[(size_t)i * ntiles + blockIdx.x] = h[i];
}

template <typename real, int D>
__global__ void __launch_bounds__(RS_THREADS) k_cell_keys(RawU<real, D> r, size_t n, int level, uint32_t* __restrict__ keys,
                                                          int bins, uint32_t* __restrict__ hist, size_t ntiles) {
  __shared__ uint32_t h[256];
  for (int i = threadIdx.x; i < bins; i += RS_THREADS) h[i] = 0;
  __syncthreads();
  const size_t base = (size_t)blockIdx.x * RS_TILE;
  const int N = 1 << level;
#pragma unroll 4
  for (int k = 0; k < RS_ITEMS; ++k) {
    const size_t i = base + (size_t)k * RS_THREADS + threadIdx.x;
    if (i < n) {
      int c[D];
#pragma unroll
      for (int m = 0; m < D; ++m) {
        real u = __ldg(r.u[m] + i);
        // positions outside [0,1) are wrapped first (periodic box)
        if (!(u >= (real)0 && u < (real)1)) u = wrap_unit(u);
        c[m] = cell_of(u, level, N);
      }
      const uint32_t key = morton_key<D>(c, level);
      keys[i] = key;
      atomicAdd(&h[key & (uint32_t)(bins - 1)], 1u);
    }
  }
  store_digits(h, bins, hist, ntiles);
}

__global__ void __launch_bounds__(RS_THREADS) k_radix_hist(const uint32_t* __restrict__ keys, size_t n, int shift,
                                                           int bins, uint32_t* __restrict__ hist, size_t ntiles) {
  __shared__ uint32_t h[256];
  pdl_trigger();
  for (int i = threadIdx.x; i < bins; i += RS_THREADS) h[i] = 0;
  __syncthreads();
  pdl_wait(keys);
  const size_t base = (size_t)blockIdx.x * RS_TILE;
#pragma unroll
  for (int k = 0; k < RS_ITEMS; ++k) {
    const size_t i = base + (size_t)k * RS_THREADS + threadIdx.x;
    if (i < n) atomicAdd(&h[(keys[i] >> shift) & (uint32_t)(bins - 1)], 1u);
  }
  store_digits(h, bins, hist, ntiles);
}

// Block b: exclusive scan of digit b's counts over the tiles, in place, and
// their sum at total[b].
__global__ void __launch_bounds__(RS_THREADS) k_radix_scan(uint32_t* __restrict__ hist, size_t ntiles,
                                                           uint32_t* __restrict__ total) {
  __shared__ uint32_t ws[RS_WARPS];
  pdl_trigger();
  pdl_wait(hist);
  uint32_t* row = hist + (size_t)blockIdx.x * ntiles;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  uint32_t carry = 0;
  for (size_t base = 0; base < ntiles; base += 4 * RS_THREADS) {
    uint32_t v[4], sum = 0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const size_t i = base + (size_t)4 * threadIdx.x + j;
      v[j] = i < ntiles ? row[i] : 0u;
      sum += v[j];
    }
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (lane == 31) ws[w] = incl;
    __syncthreads();
    uint32_t before = carry + incl - sum, all = 0;
#pragma unroll
    for (int k = 0; k < RS_WARPS; ++k) {
      if (k < w) before += ws[k];
      all += ws[k];
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const size_t i = base + (size_t)4 * threadIdx.x + j;
      if (i < ntiles) row[i] = before;
      before += v[j];
    }
    carry += all;
    __syncthreads();
  }
  if (threadIdx.x == 0) total[blockIdx.x] = carry;
}

// Lanes of the warp with the same digit (BITS bits; invalid lanes form a
// group of their own).
template <int BITS>
__device__ __forceinline__ unsigned same_digit(uint32_t dg, bool valid) {
  unsigned m = __ballot_sync(0xffffffffu, valid);
  if (!valid) m = ~m;
#pragma unroll
  for (int b = 0; b < BITS; ++b) {
    const bool set = (dg >> b) & 1u;
    const unsigned s = __ballot_sync(0xffffffffu, set);
    m &= set ? s : ~s;
  }
  return m;
}

// Stable scatter of one tile.  Warp w owns keys [256 w, 256 (w + 1)) of the
// tile, in 8 chunks of 32 in order; a key's rank is the count of earlier
// equal digits of its warp, then of the warps before, then of the tile's
// smaller digits.
template <int BITS>
__global__ void __launch_bounds__(RS_THREADS, 2) k_radix_scatter(const uint32_t* __restrict__ keys_in,
                                                              const uint32_t* __restrict__ vals_in, size_t n,
                                                              int shift, const uint32_t* __restrict__ hist,
                                                              const uint32_t* __restrict__ total, size_t ntiles,
                                                              uint32_t* __restrict__ keys_out,
                                                              uint32_t* __restrict__ vals_out) {
  constexpr int BINS = 1 << BITS;
  extern __shared__ uint32_t stage[];     // keys, then indices, in the tile's digit order
  __shared__ uint32_t wh[RS_WARPS][BINS];  // per warp: count, then the offset within the digit's run
  __shared__ uint32_t lstart[BINS];        // digit's start in the tile
  __shared__ uint32_t gstart[BINS];        // its run's place in the output, minus lstart
  __shared__ uint32_t ws[2][RS_WARPS];
  pdl_trigger();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, tid = threadIdx.x;
  for (int i = tid; i < RS_WARPS * BINS; i += RS_THREADS) (&wh[0][0])[i] = 0;
  __syncthreads();
  pdl_wait(keys_in, vals_in, hist, total);
  const size_t tile0 = (size_t)blockIdx.x * RS_TILE;
  const size_t base = tile0 + (size_t)w * RS_WARP_KEYS + lane;
  uint32_t kk[RS_ITEMS], vv[RS_ITEMS], rank[RS_ITEMS];
#pragma unroll
  for (int c = 0; c < RS_ITEMS; ++c) {
    const size_t i = base + c * 32;
    kk[c] = i < n ? keys_in[i] : 0u;
    vv[c] = !vals_in ? (uint32_t)i : i < n ? vals_in[i] : 0u;
  }
  const unsigned lt = (1u << lane) - 1u;
#pragma unroll
  for (int c = 0; c < RS_ITEMS; ++c) {
    const bool valid = base + c * 32 < n;
    const uint32_t dg = (kk[c] >> shift) & (uint32_t)(BINS - 1);
    const unsigned peers = same_digit<BITS>(dg, valid);
    const uint32_t before = wh[w][dg];
    __syncwarp();
    if (valid && (peers & lt) == 0) wh[w][dg] = before + (uint32_t)__popc(peers);
    __syncwarp();
    rank[c] = before + (uint32_t)__popc(peers & lt);
  }
  __syncthreads();
  {  // thread d: digit d's offsets by warp, its start in the tile and in the output
    const int d = tid;
    uint32_t cnt = 0, tot = 0;
    if (d < BINS) {
#pragma unroll
      for (int ww = 0; ww < RS_WARPS; ++ww) {
        const uint32_t t = wh[ww][d];
        wh[ww][d] = cnt;
        cnt += t;
      }
      tot = total[d];
    }
    uint32_t a = cnt, b = tot;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, a, o), y = __shfl_up_sync(0xffffffffu, b, o);
      if (lane >= o) {
        a += x;
        b += y;
      }
    }
    if (lane == 31) {
      ws[0][w] = a;
      ws[1][w] = b;
    }
    __syncthreads();
    if (d < BINS) {
      uint32_t ls = a - cnt, gs = b - tot;
      for (int k = 0; k < w; ++k) {
        ls += ws[0][k];
        gs += ws[1][k];
      }
      lstart[d] = ls;
      gstart[d] = gs + hist[(size_t)d * ntiles + blockIdx.x] - ls;
    }
  }
  __syncthreads();
#pragma unroll
  for (int c = 0; c < RS_ITEMS; ++c)
    if (base + c * 32 < n) {
      const uint32_t dg = (kk[c] >> shift) & (uint32_t)(BINS - 1);
      const uint32_t at = lstart[dg] + wh[w][dg] + rank[c];
      stage[at] = kk[c];
      stage[RS_TILE + at] = vv[c];
    }
  __syncthreads();
  const int nvalid = (int)min((size_t)RS_TILE, n - tile0);
  for (int j = tid; j < nvalid; j += RS_THREADS) {
    const uint32_t key = stage[j];
    const uint32_t pos = gstart[(key >> shift) & (uint32_t)(BINS - 1)] + (uint32_t)j;
    keys_out[pos] = key;
    vals_out[pos] = stage[RS_TILE + j];
  }
}

template <typename real, int D>
static int cell_keys(const void* const* u, size_t n, int level, uint32_t* keys, int bins, uint32_t* hist,
                     size_t ntiles, cudaStream_t s) {
  RawU<real, D> r;
  for (int m = 0; m < D; ++m) r.u[m] = static_cast<const real*>(u[m]);
  k_cell_keys<real, D><<<(unsigned)ntiles, RS_THREADS, 0, s>>>(r, n, level, keys, bins, hist, ntiles);
  SG_CHECK_LAUNCH();
  return SG_OK;
}

template <int BITS>
static int radix_scatter(const uint32_t* ki, const uint32_t* vi, size_t n, int shift, const uint32_t* hist,
                         const uint32_t* total, size_t ntiles, uint32_t* ko, uint32_t* vo, cudaStream_t s) {
  static DeviceSet allowed{0};  // with the static part the total may pass 48 KB
  SG_TRY(allow_smem(k_radix_scatter<BITS>, allowed, 2 * RS_TILE * (int)sizeof(uint32_t)));
  SG_CUDA(launch_pdl(k_radix_scatter<BITS>, dim3((unsigned)ntiles), dim3(RS_THREADS), 2 * RS_TILE * sizeof(uint32_t), s,
                     ki, vi, n, shift, hist, total, ntiles, ko, vo));
  SG_CHECK_LAUNCH();
  return SG_OK;
}

int cell_sort(int precision, int dim, int level, size_t n, const void* const* u, uint32_t* keys_sorted, uint32_t* perm,
              uint32_t* counts, uint32_t* scratch, cudaStream_t s) {
  const size_t count_bytes = ((size_t)1 << (dim * level)) * 4;
  if (n == 0) {
    if (counts) SG_CUDA(cudaMemsetAsync(counts, 0, count_bytes, s));
    return SG_OK;
  }
  const size_t ntiles = cell_sort_tiles(n);
  uint32_t *tk = scratch, *tv = scratch + n, *hist = scratch + 3 * n, *total = hist + 256 * ntiles;
  const int bits = dim * level, passes = (bits + 7) / 8;
  // passes alternate between the scratch and the result, which the last one
  // writes.  The unsorted keys have a place of their own and the counts are
  // cleared after it is filled: the outputs may lie over the positions.
  uint32_t* ki = scratch + 2 * n;
  const uint32_t* vi = nullptr;  // the first pass's values are the input indices
  int shift = 0;
  for (int p = 0; p < passes; ++p) {
    const int b = (bits - shift + passes - p - 1) / (passes - p), bins = 1 << b;
    if (p == 0) {
      if (precision == SG_FP32)
        SG_TRY(dim == 2 ? cell_keys<float, 2>(u, n, level, ki, bins, hist, ntiles, s)
                        : cell_keys<float, 3>(u, n, level, ki, bins, hist, ntiles, s));
      else
        SG_TRY(dim == 2 ? cell_keys<double, 2>(u, n, level, ki, bins, hist, ntiles, s)
                        : cell_keys<double, 3>(u, n, level, ki, bins, hist, ntiles, s));
      if (counts) SG_CUDA(cudaMemsetAsync(counts, 0, count_bytes, s));
    } else {
      SG_CUDA(launch_pdl(k_radix_hist, dim3((unsigned)ntiles), dim3(RS_THREADS), 0, s, ki, n, shift, bins, hist, ntiles));
      SG_CHECK_LAUNCH();
    }
    SG_CUDA(launch_pdl(k_radix_scan, dim3((unsigned)bins), dim3(RS_THREADS), 0, s, hist, ntiles, total));
    SG_CHECK_LAUNCH();
    const bool last_parity = ((passes - 1 - p) & 1) == 0;
    uint32_t *ko = last_parity ? keys_sorted : tk, *vo = last_parity ? perm : tv;
    switch (b) {
#define SG_RS_CASE(B) \
  case B: SG_TRY(radix_scatter<B>(ki, vi, n, shift, hist, total, ntiles, ko, vo, s)); break;
      SG_RS_CASE(2)
      SG_RS_CASE(3)
      SG_RS_CASE(4)
      SG_RS_CASE(5)
      SG_RS_CASE(6)
      SG_RS_CASE(7)
      SG_RS_CASE(8)
#undef SG_RS_CASE
      default:
        set_error("cell sort: unsupported digit width");
        return SG_ERR_UNSUPPORTED;
    }
    ki = ko;
    vi = vo;
    shift += b;
  }
  if (counts) SG_TRY(launch_counts(keys_sorted, n, counts, s, true));
  return SG_OK;
}

// ---------------------------------------------------------------- original order / counts
template <typename real, int D>
__global__ void __launch_bounds__(256) k_unpermute(PArrays<real, D> src, PArrays<real, D> dst, size_t np) {
  size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  uint32_t j = src.pid[i];
#pragma unroll
  for (int m = 0; m < D; ++m) {
    dst.u[m][j] = src.u[m][i];
    dst.v[m][j] = src.v[m][i];
  }
  dst.w[j] = src.w[i];
}

// The same in two passes through an array of records, one per particle in
// the original order: (u, v, w) padded to whole 32-byte sectors.  The scatter
// writes every record with full-sector stores, so that L2 evicts complete
// sectors; the direct form above leaves seven (five in 2D) 4-byte pieces in
// as many sectors, which DRAM reads and merges once the destination no
// longer fits L2.  The second pass reads the records in order and writes
// the arrays.  Bound: HBM (the payload read, the records written in random
// 32-byte sectors and read back, the payload written).  16,777,216 particles
// in 3D: 600 us in all against 4180 us direct.  In 2D FP64 the record is one
// sector of u and v, and the charge is scattered directly: two sectors would
// not fit the place that the records have (Engine::read_back_space).
template <typename real, int D>
struct __align__(32) ParticleRecord {
  static constexpr bool charge = !(D == 2 && sizeof(real) == 8);
  static constexpr int words = ((2 * D + charge) * (int)sizeof(real) + 31) / 32 * (32 / (int)sizeof(real));
  real x[words];
};

__device__ __forceinline__ void st_sector(float* p, const float* x) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(x[0]), "f"(x[1]), "f"(x[2]),
               "f"(x[3]), "f"(x[4]), "f"(x[5]), "f"(x[6]), "f"(x[7])
               : "memory");
}
__device__ __forceinline__ void st_sector(double* p, const double* x) {
  asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(p), "d"(x[0]), "d"(x[1]), "d"(x[2]), "d"(x[3])
               : "memory");
}
__device__ __forceinline__ void ld_sector(const float* p, float* x) {
  asm volatile("ld.global.v8.f32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=f"(x[0]), "=f"(x[1]), "=f"(x[2]), "=f"(x[3]), "=f"(x[4]), "=f"(x[5]), "=f"(x[6]), "=f"(x[7])
               : "l"(p));
}
__device__ __forceinline__ void ld_sector(const double* p, double* x) {
  asm volatile("ld.global.v4.f64 {%0, %1, %2, %3}, [%4];" : "=d"(x[0]), "=d"(x[1]), "=d"(x[2]), "=d"(x[3]) : "l"(p));
}

template <typename real, int D>
__global__ void __launch_bounds__(256) k_unpermute_pack(PArrays<real, D> src, ParticleRecord<real, D>* rec,
                                                        PArrays<real, D> dst, size_t np) {
  constexpr int PER = 32 / (int)sizeof(real), W = ParticleRecord<real, D>::words;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  real x[W];
#pragma unroll
  for (int k = 0; k < W; ++k) x[k] = (real)0;
#pragma unroll
  for (int m = 0; m < D; ++m) {
    x[m] = src.u[m][i];
    x[D + m] = src.v[m][i];
  }
  const uint32_t j = src.pid[i];
  if constexpr (ParticleRecord<real, D>::charge) x[2 * D] = src.w[i];
  else dst.w[j] = src.w[i];
  real* d = rec[j].x;
#pragma unroll
  for (int k = 0; k < W; k += PER) st_sector(d + k, x + k);
}

template <typename real, int D>
__global__ void __launch_bounds__(256) k_unpermute_unpack(const ParticleRecord<real, D>* rec, PArrays<real, D> dst,
                                                          size_t np) {
  constexpr int PER = 32 / (int)sizeof(real), W = ParticleRecord<real, D>::words;
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= np) return;
  real x[W];
#pragma unroll
  for (int k = 0; k < W; k += PER) ld_sector(rec[i].x + k, x + k);
#pragma unroll
  for (int m = 0; m < D; ++m) {
    dst.u[m][i] = x[m];
    dst.v[m][i] = x[D + m];
  }
  if constexpr (ParticleRecord<real, D>::charge) dst.w[i] = x[2 * D];
}

template <typename real, int D>
size_t unpermute_scratch_bytes(size_t np) {
  return np * sizeof(ParticleRecord<real, D>);
}

template <typename real, int D>
int launch_unpermute(const PArrays<real, D>& src, const PArrays<real, D>& dst, size_t np, void* scratch,
                     cudaStream_t s) {
  if (np == 0) return SG_OK;
  const unsigned blocks = (unsigned)((np + 255) / 256);
  if (!scratch) {
    k_unpermute<real, D><<<blocks, 256, 0, s>>>(src, dst, np);
    SG_CHECK_LAUNCH();
    return SG_OK;
  }
  auto* rec = static_cast<ParticleRecord<real, D>*>(scratch);
  k_unpermute_pack<real, D><<<blocks, 256, 0, s>>>(src, rec, dst, np);
  SG_CHECK_LAUNCH();
  k_unpermute_unpack<real, D><<<blocks, 256, 0, s>>>(rec, dst, np);
  SG_CHECK_LAUNCH();
  return SG_OK;
}

// ---------------------------------------------------------------- tile counting sort
// Cell keys of the current positions (the push emits them on sort steps;
// this kernel serves init and checkpoint load) and sum (key + 1).
template <typename real, int D>
__global__ void __launch_bounds__(256) k_tile_keys(PArrays<real, D> p, size_t np, int n, SortFuse sf,
                                                   unsigned* status) {
  __shared__ unsigned long long s_part[8];
  const int N = 1 << n;
  unsigned long long part = 0;
  bool bad = false;
  for (size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x; i < np; i += (size_t)gridDim.x * blockDim.x) {
    int c[D];
#pragma unroll
    for (int m = 0; m < D; ++m) {
      real u = p.u[m][i];
      bad |= !(u >= (real)0 && u < (real)1);
      c[m] = cell_of(u, n, N);
    }
    const uint32_t k = morton_key<D>(c, n);
    sf.keys[i] = k;
    part += (unsigned long long)k + 1ull;
  }
  if (bad) atomicOr(status, ST_KEY_RANGE);
  part = warp_sum(part);
  if ((threadIdx.x & 31) == 0) s_part[threadIdx.x >> 5] = part;
  __syncthreads();
  if (threadIdx.x == 0 && sf.checksum) {  // one atomic per block: all go to one address
    for (int w = 1; w < 8; ++w) part += s_part[w];
    atomicAdd(sf.checksum, part);
  }
}

template <typename real, int D>
int launch_tile_keys(const PArrays<real, D>& p, size_t np, int n, const SortFuse& sf, unsigned* status,
                     cudaStream_t s) {
  if (np == 0) return SG_OK;
  const unsigned blocks = (unsigned)(np < (size_t)1216 * 256 ? (np + 255) / 256 : 1216);
  k_tile_keys<real, D><<<blocks, 256, 0, s>>>(p, np, n, sf, status);
  SG_CHECK_LAUNCH();
  return SG_OK;
}

// The tile of a key is its top bits (key >> shift, at most 4096 tiles).
constexpr int TB_TILES = 4096;
constexpr int TH_THREADS = 512;
constexpr int TH_ITEMS = 16 * TH_THREADS;

// Tile counts: a block counts its keys in shared memory and adds each
// non-empty tile to the global counter.  Four consecutive keys of one tile
// (the common case: input sorted a few steps earlier) count once per group of
// lanes of that tile, the others one by one.  Matching every key's lanes
// instead: the sort per step, one sort in four, 2D n = 9, 8 M particles 36 ->
// 32 us, n = 10, 4 M 22.4 -> 19.7, 3D n = 7, 16.7 M 61.6 -> 60.5.
__global__ void __launch_bounds__(TH_THREADS) k_tile_hist(const uint32_t* __restrict__ keys, size_t np, int shift,
                                                          uint32_t* tile_count) {
  __shared__ uint32_t s_cnt[TB_TILES];
  for (int i = threadIdx.x; i < TB_TILES; i += TH_THREADS) s_cnt[i] = 0;
  __syncthreads();
  const size_t base = (size_t)blockIdx.x * TH_ITEMS;
  const int lane = threadIdx.x & 31;
  constexpr int NV = TH_ITEMS / TH_THREADS / 4;
  uint4 v[NV];  // sixteen keys per thread, four vector loads in flight
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const size_t i = base + ((size_t)k * TH_THREADS + threadIdx.x) * 4;
    v[k] = make_uint4(0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu, 0xFFFFFFFFu);
    if (i + 4 <= np) {
      v[k] = __ldg(reinterpret_cast<const uint4*>(keys + i));
    } else if (i < np) {
      v[k].x = keys[i];
      if (i + 1 < np) v[k].y = keys[i + 1];
      if (i + 2 < np) v[k].z = keys[i + 2];
    }
  }
#pragma unroll
  for (int k = 0; k < NV; ++k) {
    const uint32_t t[4] = {v[k].x >> shift, v[k].y >> shift, v[k].z >> shift, v[k].w >> shift};
    const bool whole = v[k].w != 0xFFFFFFFFu && t[0] == t[1] && t[1] == t[2] && t[2] == t[3];
    const unsigned peers = __match_any_sync(0xffffffffu, whole ? t[0] : 0xFFFFFFFFu);
    if (whole) {
      if (lane == __ffs(peers) - 1) atomicAdd(&s_cnt[t[0]], 4u * (uint32_t)__popc(peers));
    } else {
      if (v[k].x != 0xFFFFFFFFu) atomicAdd(&s_cnt[t[0]], 1u);
      if (v[k].y != 0xFFFFFFFFu) atomicAdd(&s_cnt[t[1]], 1u);
      if (v[k].z != 0xFFFFFFFFu) atomicAdd(&s_cnt[t[2]], 1u);
      if (v[k].w != 0xFFFFFFFFu) atomicAdd(&s_cnt[t[3]], 1u);
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < TB_TILES; i += TH_THREADS)
    if (s_cnt[i]) atomicAdd(&tile_count[i], s_cnt[i]);
}

int launch_tile_hist(const uint32_t* keys, size_t np, int shift, uint32_t* tile_count, cudaStream_t s) {
  if (np == 0) return SG_OK;
  k_tile_hist<<<(unsigned)((np + TH_ITEMS - 1) / TH_ITEMS), TH_THREADS, 0, s>>>(keys, np, shift, tile_count);
  SG_CHECK_LAUNCH();
  return SG_OK;
}

// Scatter every particle to its tile's slots.  A block takes TB_ITEMS
// particles (tile-sorted a few steps earlier), numbers the R tiles that occur
// among them, and orders its payload in shared memory by tile, in 3D by (tile,
// part of the tile): as many parts, by the next key bits, as make R tiles fit
// TB_BUCKETS counters.  It reserves one range per tile with a single global
// atomic and writes contiguous runs per tile.
//
// The tiles are what later deposits need; the parts are for the warps of the
// 3D push, which gather from nodes of a few neighbouring cells instead of the
// whole tile of 8 x 8 x 8.  3D two-stream, 16,777,216 particles, step without /
// with parts: 582 / 557 us (push, then four particles per thread, 300 / 273), 4 M at n = 6 158 / 148, Penning
// trap n = 7 164 / 165.  2D keeps tiles only: a warp whose particles share
// cells meets itself in the deposit's shared adds (annulus, 146 particles per
// cell, step 143 / 174; Landau n = 10 117 / 122).  Within a part the order
// depends on the atomics: the step sort is a valid, not a stable, counting
// sort by tile.  Bound: HBM and shared memory about equally (2D annulus: 53%
// of DRAM's rate).  Against blocks of 1024 particles that counted over their
// range of tiles: Landau n = 9, 8 M particles 45 -> 35 us per step, n = 10
// 25.8 -> 21.9, Penning 18.6 -> 12.1, annulus 29.6 -> 32.8.
constexpr int TB_THREADS = 512;
constexpr int TB_PER_THREAD = 4;
constexpr int TB_ITEMS = TB_THREADS * TB_PER_THREAD;
constexpr int TB_BUCKETS = 4096;
static_assert(TB_ITEMS <= TB_BUCKETS, "every particle in a tile of its own still fits");

// Exclusive scan over the block of each thread's sum; *all receives the total.
__device__ __forceinline__ uint32_t block_scan(uint32_t sum, uint32_t* ws /* TB_THREADS / 32 */, uint32_t* all) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) ws[warp] = incl;
  __syncthreads();
  constexpr int NW = TB_THREADS / 32;  // every warp scans the warps' sums
  uint32_t t = lane < NW ? ws[lane] : 0u;
#pragma unroll
  for (int o = 1; o < NW; o <<= 1) {
    const uint32_t y = __shfl_up_sync(0xffffffffu, t, o);
    if (lane >= o) t += y;
  }
  const uint32_t before = __shfl_sync(0xffffffffu, t, warp > 0 ? warp - 1 : 0);
  *all = __shfl_sync(0xffffffffu, t, NW - 1);
  __syncthreads();
  return incl - sum + (warp > 0 ? before : 0u);
}

template <typename real, int D>
constexpr size_t scatter_stage_bytes() {
  return (size_t)TB_ITEMS * ((2 * D + 1) * sizeof(real) + 2 * sizeof(uint32_t));
}

template <typename real, int D>
__global__ void __launch_bounds__(TB_THREADS, sizeof(real) == 4 ? 2 : 1) k_tile_scatter(PArrays<real, D> src, PArrays<real, D> dst,
                                                             const uint32_t* __restrict__ keys, int shift,
                                                             uint32_t* cursor, size_t np) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) uint16_t s_id[TB_TILES];      // tile -> its number in the block
  __shared__ uint16_t s_tile[TB_ITEMS];                  // and back
  __shared__ __align__(16) uint32_t s_cnt[TB_BUCKETS];   // per bucket: count, then the local start
  __shared__ uint32_t s_base[TB_ITEMS];                  // per tile: the block's global base minus the local start
  __shared__ uint32_t s_ws[TB_THREADS / 32];
  const size_t chunk = (size_t)blockIdx.x * TB_ITEMS;
  const int lane = threadIdx.x & 31, tid = threadIdx.x;
  constexpr int PT = TB_TILES / TB_THREADS;
  static_assert(PT == 8, "eight 16-bit flags per thread in one vector");
  uint32_t key[TB_PER_THREAD];
#pragma unroll
  for (int k = 0; k < TB_PER_THREAD; ++k) {
    const size_t i = chunk + (size_t)k * TB_THREADS + tid;
    key[k] = i < np ? __ldg(keys + i) : 0xFFFFFFFFu;
  }
  // the payload's loads go out now, so that their latency overlaps the ranking
  real pu[TB_PER_THREAD][D], pv[TB_PER_THREAD][D], pw[TB_PER_THREAD];
  uint32_t ppid[TB_PER_THREAD];
#pragma unroll
  for (int k = 0; k < TB_PER_THREAD; ++k) {
    const size_t i = chunk + (size_t)k * TB_THREADS + tid;
    const bool valid = i < np;
#pragma unroll
    for (int m = 0; m < D; ++m) {
      pu[k][m] = valid ? __ldg(src.u[m] + i) : (real)0;
      pv[k][m] = valid ? __ldg(src.v[m] + i) : (real)0;
    }
    pw[k] = valid ? __ldg(src.w + i) : (real)0;
    ppid[k] = valid ? __ldg(src.pid + i) : 0u;
  }
  reinterpret_cast<uint4*>(s_id)[tid] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
#pragma unroll
  for (int k = 0; k < TB_PER_THREAD; ++k)
    if (key[k] != 0xFFFFFFFFu) s_id[key[k] >> shift] = 1;
  __syncthreads();
  uint32_t R;
  {  // number the tiles that occur
    const uint4 f = reinterpret_cast<const uint4*>(s_id)[tid];  // eight flags of 0 or 1
    const uint32_t f2[4] = {f.x, f.y, f.z, f.w};
    const uint32_t pairs = f.x + f.y + f.z + f.w;
    uint32_t at = block_scan((pairs & 0xFFFFu) + (pairs >> 16), s_ws, &R);
#pragma unroll
    for (int j = 0; j < PT; ++j)
      if ((f2[j >> 1] >> (16 * (j & 1))) & 1u) {
        s_tile[at] = (uint16_t)(PT * tid + j);
        s_id[PT * tid + j] = (uint16_t)at++;
      }
  }
  const int logf = min(D == 3 ? shift : 0, 12 - (R > 1 ? 32 - __clz(R - 1) : 0));  // 2^logf parts per tile
  const uint32_t fine = (1u << shift) - 1u, nb = R << logf;
  for (uint32_t i = tid; i < nb; i += TB_THREADS) s_cnt[i] = 0;
  __syncthreads();
  uint32_t bucket[TB_PER_THREAD], pos[TB_PER_THREAD];
#pragma unroll
  for (int k = 0; k < TB_PER_THREAD; ++k) {  // rank within the bucket: one shared atomic per group of a warp
    const bool valid = key[k] != 0xFFFFFFFFu;
    bucket[k] = valid ? ((uint32_t)s_id[key[k] >> shift] << logf) + ((key[k] & fine) >> (shift - logf)) : 0xFFFFFFFFu;
    const unsigned peers = __match_any_sync(0xffffffffu, bucket[k]);
    const int leader = __ffs(peers) - 1;
    uint32_t b = 0;
    if (valid && lane == leader) b = atomicAdd(&s_cnt[bucket[k]], (uint32_t)__popc(peers));
    pos[k] = __shfl_sync(0xffffffffu, b, leader) + (uint32_t)__popc(peers & ((1u << lane) - 1u));
  }
  __syncthreads();
  uint32_t nvalid;
  {  // local starts: `per` consecutive buckets per thread
    const uint32_t per = (nb + TB_THREADS - 1) / TB_THREADS, b0 = min(tid * per, nb), b1 = min(b0 + per, nb);
    uint32_t n = 0;
    for (uint32_t i = b0; i < b1; ++i) n += s_cnt[i];
    uint32_t at = block_scan(n, s_ws, &nvalid);
    for (uint32_t i = b0; i < b1; ++i) {
      const uint32_t c = s_cnt[i];
      s_cnt[i] = at;
      at += c;
    }
  }
  __syncthreads();
  for (uint32_t q = tid; q < R; q += TB_THREADS) {  // one global atomic per tile
    const uint32_t a = s_cnt[q << logf], e = q + 1 < R ? s_cnt[(q + 1) << logf] : nvalid;
    s_base[q] = atomicAdd(&cursor[s_tile[q]], e - a) - a;
  }
  real* su = reinterpret_cast<real*>(smem_raw);  // [2D+1][TB_ITEMS]: u, v, w
  uint32_t* spid = reinterpret_cast<uint32_t*>(su + (size_t)(2 * D + 1) * TB_ITEMS);
  uint32_t* stl = spid + TB_ITEMS;  // the particle's tile number
#pragma unroll
  for (int k = 0; k < TB_PER_THREAD; ++k)
    if (key[k] != 0xFFFFFFFFu) {
      const uint32_t L = s_cnt[bucket[k]] + pos[k];
#pragma unroll
      for (int m = 0; m < D; ++m) {
        su[(size_t)m * TB_ITEMS + L] = pu[k][m];
        su[(size_t)(D + m) * TB_ITEMS + L] = pv[k][m];
      }
      su[(size_t)(2 * D) * TB_ITEMS + L] = pw[k];
      spid[L] = ppid[k];
      stl[L] = bucket[k] >> logf;
    }
  __syncthreads();
  for (uint32_t j = tid; j < nvalid; j += TB_THREADS) {
    const uint32_t p = s_base[stl[j]] + j;
#pragma unroll
    for (int m = 0; m < D; ++m) {
      dst.u[m][p] = su[(size_t)m * TB_ITEMS + j];
      dst.v[m][p] = su[(size_t)(D + m) * TB_ITEMS + j];
    }
    dst.w[p] = su[(size_t)(2 * D) * TB_ITEMS + j];
    dst.pid[p] = spid[j];
  }
}

template <typename real, int D>
int launch_tile_scatter(const PArrays<real, D>& src, const PArrays<real, D>& dst, const uint32_t* keys, int shift,
                        uint32_t* cursor, size_t np, cudaStream_t s) {
  if (np == 0) return SG_OK;
  constexpr size_t smem = scatter_stage_bytes<real, D>();
  static DeviceSet allowed{0};  // with the static counters the total passes 48 KB
  SG_TRY(allow_smem(k_tile_scatter<real, D>, allowed, (int)smem));
  k_tile_scatter<real, D><<<(unsigned)((np + TB_ITEMS - 1) / TB_ITEMS), TB_THREADS, smem, s>>>(src, dst, keys, shift,
                                                                                              cursor, np);
  SG_CHECK_LAUNCH();
  return SG_OK;
}

// counts[key] of runs of equal keys (any order of the keys; runs make it
// fast).  A run inside one warp stores its length when `sorted` (it is then
// the key's only run), others add theirs.
__global__ void __launch_bounds__(256) k_counts(const uint32_t* __restrict__ keys, size_t np, uint32_t* counts,
                                                int sorted) {
  const size_t i = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int lane = threadIdx.x & 31;
  pdl_wait(keys);
  const bool valid = i < np;
  const uint32_t k = valid ? keys[i] : 0xFFFFFFFFu;
  const uint32_t up = __shfl_up_sync(0xffffffffu, k, 1), dn = __shfl_down_sync(0xffffffffu, k, 1);
  const unsigned starts = __ballot_sync(0xffffffffu, lane == 0 || up != k);
  if (!valid || (lane < 31 && dn == k)) return;  // the run's last lane writes
  const int first = 31 - __clz(starts & (0xFFFFFFFFu >> (31 - lane)));
  const uint32_t len = (uint32_t)(lane - first + 1);
  if (sorted && first > 0 && lane < 31) counts[k] = len;
  else atomicAdd(&counts[k], len);
}

int launch_counts(const uint32_t* keys, size_t np, uint32_t* counts, cudaStream_t s, bool sorted) {
  if (np == 0) return SG_OK;
  SG_CUDA(launch_pdl(k_counts, dim3((unsigned)((np + 255) / 256)), dim3(256), 0, s, keys, np, counts, sorted ? 1 : 0));
  SG_CHECK_LAUNCH();
  return SG_OK;
}

#define SG_INST_SORT(real, D)                                                                           \
  template int launch_keys<real, D>(const PArrays<real, D>&, size_t, int, uint32_t*, unsigned*, cudaStream_t); \
  template int launch_unpermute<real, D>(const PArrays<real, D>&, const PArrays<real, D>&, size_t, void*,        \
                                         cudaStream_t);                                                          \
  template size_t unpermute_scratch_bytes<real, D>(size_t);                                              \
  template int launch_tile_keys<real, D>(const PArrays<real, D>&, size_t, int, const SortFuse&, unsigned*,         \
                                         cudaStream_t);                                                            \
  template int launch_tile_scatter<real, D>(const PArrays<real, D>&, const PArrays<real, D>&, const uint32_t*, int, \
                                            uint32_t*, size_t, cudaStream_t);

SG_INST_SORT(float, 2)
SG_INST_SORT(float, 3)
SG_INST_SORT(double, 2)
SG_INST_SORT(double, 3)

}  // namespace sg
