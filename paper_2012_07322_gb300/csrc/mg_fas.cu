// The FP64 FAS V-cycle of a scalar equation (Sec. 2.7) from a level of a few thousand cells down,
// in one launch of a thread-block cluster.
//
// On such levels a launched pass is a dependent chain of its launch (~1.2
// us), one L2 round trip and an FP64 chain of ~1500 cycles (a dependent FP64
// operation takes ~64 cycles, a division ~430): 3.3 us in the captured cycle,
// whatever the level's size, 12 of them per level and cycle.  Here the same
// passes are separated by cluster barriers instead of kernel boundaries.  A
// cluster rather than one block because the FP64 pipe takes ~16 cycles per
// warp instruction: 1024 cells of one colour are 23 k cycles on one SM and
// 1.4 k on sixteen.  Levels of at most FAS_SOLO_CELLS cells run on block 0
// alone with block barriers.  Every pass applies the per-cell functions of
// the launched kernels in their order, so the results are the same.  Eq. psi
// on 64 x 32 cells: 207 us per cycle with launches, 170 us so.  (A vector
// cycle, with a ghost fill after every pass, was slower so than launched:
// 106 against 103 ms per 64x32x32 solve.)
#include <cooperative_groups.h>

#include "mg_coarse.cuh"
#include "mg_internal.h"
#include "mg_kernels.cuh"

namespace cg = cooperative_groups;

namespace gmg {

constexpr int FAS_THREADS = 256;

// The blocks that take part in a pass: the cluster, or block 0 alone.  Warps
// are dealt round the blocks, so that a pass of few cells spreads its warps
// over the SMs.
struct FasTeam {
  int rank, size;
  __device__ __forceinline__ int start() const {
    return ((int)(threadIdx.x >> 5) * size + rank) * 32 + (int)(threadIdx.x & 31);
  }
  __device__ __forceinline__ int stride() const { return size * FAS_THREADS; }
  __device__ __forceinline__ void sync() const {
    if (size > 1)
      asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
    else
      __syncthreads();
  }
};

template <int G, int KIND>
__device__ __forceinline__ void fas_smooth(const FasTeam& T, const FasLevel& F, int nsweeps) {
  const LevelView<double>& L = F.v;
  const int nh = L.n0 * L.n1 * L.n2 / 2;
  for (int h = 0; h < 2 * nsweeps; ++h) {
    for (int q = T.start(); q < nh; q += T.stride()) {
      int i, j, k;
      L.colour_cell(q, h & 1, i, j, k);
      scalar_update<double, G, KIND>(L, F.u, F.f, F.s0, F.s1, i, j, k);
    }
    T.sync();
  }
}

// FAS restriction (fas_down64): r = f - L(u); u_H = R u, kept in uh_H; f_H =
// L_H(u_H) + R r.  T: the team of the fine level, TC of the coarse one.
template <int G, int KIND>
__device__ __forceinline__ void fas_down(const FasTeam& T, const FasTeam& TC, const FasLevel& F, const FasLevel& C) {
  const LevelView<double>&L = F.v, &Lc = C.v;
  const int n = L.n0 * L.n1 * L.n2, nc = Lc.n0 * Lc.n1 * Lc.n2;
  for (int q = T.start(); q < n; q += T.stride()) {
    int i, j, k;
    L.cell(q, i, j, k);
    const long p = L.idx(i, j, k);
    double Sv;
    F.r[p] = scalar_residual_cell<double, G, KIND>(L, F.u, F.f, F.s0, F.s1, i, j, k, p, Sv);
  }
  T.sync();
  for (int q = T.start(); q < nc; q += T.stride()) {
    int I, J, K;
    Lc.cell(q, I, J, K);
    const double* const as[2] = {F.u, F.r};
    double *const bs[2] = {C.u, C.f}, *const cs[3] = {C.uh, nullptr, nullptr};
    restrict_cell<double, 2>(L, Lc, 2, as, bs, cs, I, J, K);
  }
  T.sync();
  // from here on only the coarse level's team works
  if (TC.rank >= TC.size) return;
  for (int q = TC.start(); q < nc; q += TC.stride()) {
    int i, j, k;
    Lc.cell(q, i, j, k);
    const long p = Lc.idx(i, j, k);
    double D;
    C.f[p] += scalar_op<double, G, KIND>(Lc, C.u, C.s0, C.s1, i, j, k, p, D);
  }
  TC.sync();
}

// FAS correction (fas_up64): u += P(u_H - uh_H).
__device__ __forceinline__ void fas_up(const FasTeam& T, const FasLevel& F, const FasLevel& C) {
  const LevelView<double>& L = F.v;
  const int n = L.n0 * L.n1 * L.n2;
  for (int q = T.start(); q < n; q += T.stride()) {
    int i, j, k;
    L.cell(q, i, j, k);
    prolong_cell(L, C.v, F.u, (const double*)C.u, (const double*)C.uh, -1, i, j, k);
  }
  T.sync();
}

template <int G, int KIND>
__global__ void __launch_bounds__(FAS_THREADS) k_fas_cycle(const __grid_constant__ FasCycle P) {
  pdl_entry();
  __shared__ CoarseShared cs;
  // the levels in shared memory: handed by reference to the out-of-line edge
  // rules, a kernel parameter would be read through the generic address of
  // the constant bank, a dependent load per field
  __shared__ __align__(16) unsigned char lv_raw[sizeof(FasLevel) * FAS_MAX];
  FasLevel* const lv = reinterpret_cast<FasLevel*>(lv_raw);
  for (int q = threadIdx.x; q < (int)(sizeof(FasLevel) / 4) * P.nl; q += FAS_THREADS)
    reinterpret_cast<unsigned*>(lv_raw)[q] = reinterpret_cast<const unsigned*>(P.lv)[q];
  __syncthreads();
  const int rank = (int)cg::this_cluster().block_rank(), size = (int)cg::this_cluster().num_blocks();
  const FasTeam all{rank, size}, solo{rank, 1};
  // levels solo_from .. nl - 1 run on block 0
  for (int l = 0; l + 1 < P.nl; ++l) {
    const FasTeam T = l < P.solo_from ? all : solo, TC = l + 1 < P.solo_from ? all : solo;
    if (rank >= T.size) break;
    fas_smooth<G, KIND>(T, lv[l], P.nu1);
    fas_down<G, KIND>(T, TC, lv[l], lv[l + 1]);
  }
  if (rank == 0) {
    const FasLevel& C = lv[P.nl - 1];
    coarse_scalar_small<G, KIND>(cs, C.v, C.u, C.f, C.s0, C.s1, P.coarse_sweeps);
    __syncthreads();
  }
  for (int l = P.nl - 2; l >= 0; --l) {
    const FasTeam T = l < P.solo_from ? all : solo;
    if (rank >= T.size) continue;
    // block 0 hands the coarse level over to the cluster
    if (T.size > 1 && l + 1 >= P.solo_from) T.sync();
    fas_up(T, lv[l], lv[l + 1]);
    fas_smooth<G, KIND>(T, lv[l], P.nu2);
  }
}

using FasKernel = void (*)(FasCycle);

template <int G>
static FasKernel fas_kernel_g(int kind) {
  return kind == EQ_PSI ? k_fas_cycle<G, EQ_PSI> : k_fas_cycle<G, EQ_LIN>;
}
static FasKernel fas_kernel(int geom, int kind) {
  return geom == CART ? fas_kernel_g<CART>(kind) : (geom == CYL ? fas_kernel_g<CYL>(kind) : fas_kernel_g<SPH>(kind));
}

// The largest cluster (16 blocks, else 8) every instantiation can launch
// with, 0 when none can.
static int g_fas_cluster = -1;

static cudaLaunchConfig_t fas_config(int cluster, cudaStream_t st, cudaLaunchAttribute* at) {
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cluster);
  cfg.blockDim = dim3(FAS_THREADS);
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cfg;
}

void init_fas_attributes() {
  if (g_fas_cluster >= 0) return;
  int best = 16;
  for (int g = 0; g < 3; ++g)
    for (int kind = EQ_PSI; kind <= EQ_LIN; ++kind) {
      FasKernel k = fas_kernel(g, kind);
      cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      for (; best >= 8; best /= 2) {
        cudaLaunchAttribute at[2];
        cudaLaunchConfig_t cfg = fas_config(best, nullptr, at);
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, k, &cfg) == cudaSuccess && nc > 0) break;
        cudaGetLastError();
      }
    }
  g_fas_cluster = best >= 8 ? best : 0;
}

bool fas_cycle_available() { return g_fas_cluster > 0; }

void launch_fas_cycle(const FasCycle& P, int geom, int kind, cudaStream_t st) {
  count_launch();
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t cfg = fas_config(g_fas_cluster, st, at);
  cudaLaunchKernelEx(&cfg, fas_kernel(geom, kind), P);
}

}  // namespace gmg
