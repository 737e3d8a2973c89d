// Cell-key sort without device allocation.
//
// sg_cell_sort obtains its scratch (key/index ping-pong buffers, digit
// histograms and totals) from the stream-ordered allocator
// on every call.  Some callers cannot do that: code that runs under a device
// memory budget owned by another allocator (a framework's caching allocator
// that holds all device memory), or latency-critical loops in which an
// allocation or a free may synchronise the device or fail under
// fragmentation.  For them, sg_cell_sort_static runs the same kernels on a
// fixed scratch area that is part of the library image: a file-scope device
// array of SG_CELL_SORT_STATIC_WORDS words, present on every GPU that loads
// the library for the life of the process.
//
// Host code cannot use the array's name as a device address (it denotes a
// host-side stand-in), so the first call on each device looks the address up
// with cudaGetSymbolAddress while that device is current and caches it.
// Every call shares the array and it keeps the previous call's contents:
// everything is fully rewritten before it is read.  Two
// calls whose work overlaps on the GPU (different streams, no ordering) race
// on the array.
#include <mutex>

#include "sg_kernels.cuh"

namespace sg {

// Keys and indices of the radix sort's alternate passes and the unsorted keys
// (3 x max), digit histograms and totals.
constexpr size_t kStaticMax = SG_CELL_SORT_STATIC_MAX;
constexpr size_t kStaticWords = 3 * kStaticMax + 256 * ((kStaticMax + RS_TILE - 1) / RS_TILE) + 256;  // cell_sort_words
static_assert(kStaticWords <= SG_CELL_SORT_STATIC_WORDS, "scratch layout exceeds the declared size");

static __device__ __align__(256) uint32_t g_cell_sort_scratch[SG_CELL_SORT_STATIC_WORDS];

namespace {
std::mutex g_static_mu;
uint32_t* g_static_addr[256] = {};  // per device ordinal

int static_scratch(uint32_t** out) {
  int dev = 0;
  SG_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 256) {
    set_error("sg_cell_sort_static: device ordinal out of range");
    return SG_ERR_UNSUPPORTED;
  }
  std::lock_guard<std::mutex> lk(g_static_mu);
  if (!g_static_addr[dev]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_cell_sort_scratch);
    if (e != cudaSuccess) {
      set_error(std::string("sg_cell_sort_static: cudaGetSymbolAddress: ") + cudaGetErrorString(e));
      return SG_ERR_CUDA;
    }
    g_static_addr[dev] = static_cast<uint32_t*>(p);
  }
  *out = g_static_addr[dev];
  return SG_OK;
}
}  // namespace

}  // namespace sg

using namespace sg;

extern "C" int sg_cell_sort_static(int precision, int dim, int level, size_t n, const void* const* u,
                                   uint32_t* keys_sorted, uint32_t* perm, uint32_t* counts, void* stream) {
  if (dim != 2 && dim != 3) {
    set_error("sg_cell_sort_static: dim must be 2 or 3");
    return SG_ERR_INVALID;
  }
  if (level < 1 || dim * level > 24) {
    set_error("sg_cell_sort_static: need 1 <= level and dim*level <= 24");
    return SG_ERR_INVALID;
  }
  if (precision != SG_FP32 && precision != SG_FP64) {
    set_error("sg_cell_sort_static: bad precision");
    return SG_ERR_INVALID;
  }
  if (n > kStaticMax) {
    set_error("sg_cell_sort_static: " + std::to_string(n) + " positions exceed the fixed scratch capacity of " +
              std::to_string(kStaticMax) + " (use sg_cell_sort)");
    return SG_ERR_SIZE;
  }
  if (n > 0 && (!u || !keys_sorted || !perm)) {
    set_error("sg_cell_sort_static: NULL pointer");
    return SG_ERR_INVALID;
  }
  for (int m = 0; n > 0 && m < dim; ++m)
    if (!u[m]) {
      set_error("sg_cell_sort_static: NULL position array");
      return SG_ERR_INVALID;
    }
  cudaStream_t s = (cudaStream_t)stream;
  if (n == 0) return cell_sort(precision, dim, level, 0, u, keys_sorted, perm, counts, nullptr, s);
  uint32_t* buf = nullptr;
  SG_TRY(static_scratch(&buf));
  return cell_sort(precision, dim, level, n, u, keys_sorted, perm, counts, buf, s);
}
