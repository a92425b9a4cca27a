// Divergence diagnostics of a Cartesian field without any device allocation.
//
// Some callers cannot call cudaMalloc: code that runs between the steps of
// a host framework which owns all device memory and forbids allocations in
// its time loop, or code whose allocations would synchronise the device
// and break the overlap of its streams.  They cannot create a hierarchy
// (mg_create_hierarchy allocates), yet still want the divergence monitor.
// This file gives them mg_divb_norms_noalloc: the central divergence and its
// norms as mg_clean_divB reports them, with the scratch (block partial
// results, a counter of finished blocks and the result) in a file-scope
// __device__ array instead of the hierarchy's arena.
//
// The call is bound by its launches and round trips: one launch whose last
// block to finish combines the blocks' results, and one 16-byte read-back.
// (With a cleared max word, a divergence and a norms kernel and two
// read-backs a 56x40x48 block took 55 us; so, 43 us.)
//
// Every GPU that loads the library keeps the array until the process exits.
// All calls share it: calls whose work overlaps on the GPU race with each
// other.
#include <cmath>
#include <cstring>
#include <mutex>

#include "mg.h"
#include "mg_internal.h"
#include "mg_kernels.cuh"

namespace {

constexpr int NOALLOC_BLOCKS = 1024;
constexpr int NOALLOC_MAX_DEVICES = 64;
// Per block the sum of div^2 and max |div| (bit pattern), then the result in
// the same form, then the counter of finished blocks (the last block resets
// it; behind calls that overlapped, Call clears it).
struct NoallocScratch {
  double sum[NOALLOC_BLOCKS];
  unsigned long long max[NOALLOC_BLOCKS];
  double total;
  unsigned long long top;
  unsigned int done;
};

}  // namespace

static __device__ __align__(256) NoallocScratch g_divb_scratch;

namespace {

std::mutex g_setup_mutex;
NoallocScratch* g_scratch_addr[NOALLOC_MAX_DEVICES] = {};
int g_inside = 0;                                // calls in progress
unsigned long long g_spoilt = 0;                 // times a counter may have been left off zero
unsigned long long g_cleared[NOALLOC_MAX_DEVICES] = {};  // g_spoilt when the device's was last cleared

// A call in progress.  Calls end synchronised, so only calls that are inside
// at the same time can overlap on the GPU.  The first one alone behind such
// calls (or behind one that failed) clears the counter they may have left off
// zero; without it every later call would end its reduction at the wrong
// block.  Calls that nothing overlapped pay no launch for it (40 to 44 us with
// and without, 56x40x48).
struct Call {
  bool done = false;
  // *clear: the counter of device dev is to be cleared first.
  Call(int dev, bool* clear) {
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    if (g_inside++ > 0) ++g_spoilt;
    *clear = g_inside == 1 && g_cleared[dev] != g_spoilt;
    if (*clear) g_cleared[dev] = g_spoilt;
  }
  ~Call() {
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    --g_inside;
    if (!done) ++g_spoilt;
  }
};

// Sum and max over the block's threads, to thread 0 (fixed order).
__device__ __forceinline__ void block_norms(double& s, unsigned long long& m) {
  __shared__ double ss[8];
  __shared__ unsigned long long sm[8];
  s = gmg::warp_sum(s);
  m = gmg::warp_max_bits(m);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) {
    ss[w] = s;
    sm[w] = m;
  }
  __syncthreads();
  if (w == 0) {
    s = lane < 8 ? ss[lane] : 0.0;
    m = lane < 8 ? sm[lane] : 0ULL;
    for (int o = 4; o > 0; o >>= 1) {
      s += __shfl_xor_sync(0xffffffffu, s, o);
      m = gmg::umax64(m, __shfl_xor_sync(0xffffffffu, m, o));
    }
  }
}

// Central divergence with zero-gradient (copied) ghosts, its sum of squares
// and largest magnitude (NaN counts as infinite).
__global__ void __launch_bounds__(256)
    k_noalloc_norms(int n0, int n1, int n2, int three, double c0, double c1, double c2,
                    const double* __restrict__ B0, const double* __restrict__ B1, const double* __restrict__ B2,
                    NoallocScratch* __restrict__ S) {
  gmg::pdl_entry();
  __shared__ bool last;
  const unsigned n = (unsigned)n0 * n1 * n2, s1 = n0, s2 = (unsigned)n0 * n1;
  double s = 0.0;
  unsigned long long m = 0ULL;
  for (unsigned q = blockIdx.x * blockDim.x + threadIdx.x; q < n; q += gridDim.x * blockDim.x) {
    const unsigned jk = q / s1, k = jk / (unsigned)n1, j = jk - k * n1, i = q - jk * s1;
    double d = (B0[i < s1 - 1 ? q + 1 : q] - B0[i > 0 ? q - 1 : q]) * c0 +
               (B1[(int)j < n1 - 1 ? q + s1 : q] - B1[j > 0 ? q - s1 : q]) * c1;
    if (three) d += (B2[(int)k < n2 - 1 ? q + s2 : q] - B2[k > 0 ? q - s2 : q]) * c2;
    s += d * d;
    m = gmg::umax64(m, gmg::abs_bits(d));
  }
  block_norms(s, m);
  if (threadIdx.x == 0) {
    S->sum[blockIdx.x] = s;
    S->max[blockIdx.x] = m;
    __threadfence();
    last = atomicAdd(&S->done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  s = 0.0;
  m = 0ULL;
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) {
    s += __ldcg(&S->sum[b]);
    m = gmg::umax64(m, __ldcg(&S->max[b]));
  }
  block_norms(s, m);
  if (threadIdx.x == 0) {
    S->total = s;
    S->top = m;
    S->done = 0u;
  }
}

// Device address of the scratch array on the current device, looked up
// once per device (cudaGetSymbolAddress with that device current).
int scratch_address(NoallocScratch** out, int* device) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return MG_ERR_CUDA;
  if (dev < 0 || dev >= NOALLOC_MAX_DEVICES) return MG_ERR_INVALID;
  std::lock_guard<std::mutex> lock(g_setup_mutex);
  if (!g_scratch_addr[dev]) {
    NoallocScratch* p = nullptr;
    e = cudaGetSymbolAddress((void**)&p, g_divb_scratch);
    if (e != cudaSuccess || !p) return MG_ERR_CUDA;
    g_scratch_addr[dev] = p;
  }
  *out = g_scratch_addr[dev];
  *device = dev;
  return MG_OK;
}

}  // namespace

extern "C" int mg_divb_norms_noalloc(int ndim, const int n[3], const double lo[3], const double hi[3],
                                     const double* B[3], void* cuda_stream, double* max_div, double* l2_div) {
  using gmg::set_last_error;
  if (ndim != 2 && ndim != 3) return set_last_error(MG_ERR_INVALID, "ndim must be 2 or 3");
  if (!n || !lo || !hi || !B || !max_div || !l2_div) return set_last_error(MG_ERR_INVALID, "null argument");
  long cells = 1;
  for (int d = 0; d < ndim; ++d) {
    if (n[d] < 1 || !(hi[d] > lo[d])) return set_last_error(MG_ERR_INVALID, "need n >= 1 and lo < hi");
    if (!B[d]) return set_last_error(MG_ERR_INVALID, "null B component");
    cells *= n[d];
    if (cells > (long)MG_NOALLOC_MAX_CELLS)
      return set_last_error(MG_ERR_INVALID,
                            "grid larger than MG_NOALLOC_MAX_CELLS (2097152 cells), the size of the static "
                            "scratch of the allocation-free entry point");
  }
  // an error left by earlier, unrelated work of the caller must not be
  // reported as this call's: drop it (launch errors are checked below)
  (void)cudaGetLastError();
  NoallocScratch* scratch = nullptr;
  int dev = 0;
  int st = scratch_address(&scratch, &dev);
  if (st) return set_last_error(st, "looking up the device address of the static scratch failed");
  cudaStream_t s = (cudaStream_t)cuda_stream;
  const int n0 = n[0], n1 = n[1], n2 = ndim == 3 ? n[2] : 1;
  const double c0 = 0.5 / ((hi[0] - lo[0]) / n0), c1 = 0.5 / ((hi[1] - lo[1]) / n1);
  const double c2 = ndim == 3 ? 0.5 / ((hi[2] - lo[2]) / n2) : 0.0;
  long g = (cells + 255) / 256;
  if (g > NOALLOC_BLOCKS) g = NOALLOC_BLOCKS;
  bool clear = false;
  Call call(dev, &clear);
  if (clear && cudaMemsetAsync(&scratch->done, 0, sizeof(scratch->done), s) != cudaSuccess)
    return set_last_error(MG_ERR_CUDA, "clearing the counter failed");
  gmg::count_launch();
  gmg::launch_k(k_noalloc_norms, (unsigned)g, 256, 0, s, n0, n1, n2, ndim == 3, c0, c1, c2, B[0], B[1],
                ndim == 3 ? B[2] : B[0], scratch);
  if (cudaGetLastError() != cudaSuccess) return set_last_error(MG_ERR_CUDA, "launching the divergence kernel failed");
  struct {
    double sum;
    unsigned long long max;
  } res;
  if (cudaMemcpyAsync(&res, &scratch->total, sizeof(res), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return set_last_error(MG_ERR_CUDA, "divergence kernel or read-back failed");
  call.done = true;
  double mx;
  static_assert(sizeof(mx) == sizeof(res.max), "word size");
  memcpy(&mx, &res.max, sizeof(mx));
  *max_div = mx;
  *l2_div = sqrt(res.sum / (double)cells);
  return MG_OK;
}
