// The FP64 FAS V-cycle of the vector equation (Sec. 2.7) from a level of a few thousand cells down,
// in one launch of a thread-block cluster.
//
// Launched, a (colour, component) pass of such a level takes 4 - 5 us in the
// captured cycle and 7.6 us cold whatever the level's size: its launch, an L2
// round trip, the coefficients' loads and a dependent FP64 chain (~64 cycles
// an operation); a cycle has 24 of them per level.  Here a thread owns one
// cell, with its coefficients in registers over the sweeps of a visit, u of
// every level lies in every block's shared memory, and a new value is stored
// into the blocks that read it: a pass is a cluster barrier, the neighbours'
// shared loads, ~30 FP64 operations in short chains and the refill of the
// ghosts the block reads (tables as in mg_clus.cu).  Levels of at most
// FAS_SOLO_CELLS cells run on block 0.  FP64 xCFC on 64 x 32 x 32 cells, whose
// cycles run levels 16 x 8 x 8 and below so: 79.9 to 71.4 ms per solve.
#include <cooperative_groups.h>

#include "mg_cell.cuh"
#include "mg_coarse.cuh"
#include "mg_internal.h"
#include "mg_kernels.cuh"

namespace cg = cooperative_groups;

namespace gmg {

constexpr int FV_THREADS = 256;
static_assert(FV_THREADS == CV_THREADS, "block 0 runs the coarsest solve");

template <int G>
struct FasVec {
  const ClCell& t;
  const LevelView<double>& L;
  double *u[3], *x[3];  // ghosted; x: restricted residual, later u - uh
  double* slot;         // right-hand side and restricted u of the own cell
  unsigned mask;        // blocks that read the cell
  const uint2* list;    // ghosts this block reads
  int nlist;
  uint2 g[2];
  long hp;              // the cell in HBM (first level)
  double a[12], b[10], c[10], iD[3], f[3], wt;

  __device__ __forceinline__ FasVec(const ClCell& t_, const FasVecCycle& Q, int l, double* sm)
      : t(t_), L(Q.lv[l].v), mask(0) {
    const FasVecLevel& T = Q.lv[l];
    const int ng = T.ng;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      u[m] = sm + T.u_at + m * ng;
      x[m] = sm + T.x_at + m * ng;
    }
    slot = sm + T.slot_at + t.tid;
    nlist = 0;
    if (T.list) {
      list = T.list + T.start[t.rank];
      nlist = T.start[t.rank + 1] - T.start[t.rank];
    }
#pragma unroll
    for (int r = 0; r < 2; ++r)
      g[r] = t.tid + r * FV_THREADS < nlist ? list[t.tid + r * FV_THREADS] : make_uint2(0, 0);
    if (!t.on) return;
    hp = Q.off + t.i + t.j * Q.sx + t.k * Q.sy;
    if (T.mask) mask = T.mask[t.i + L.n0 * (t.j + L.n1 * t.k)];
    wt = t.weight(L);
#pragma unroll
    for (int m = 0; m < 3; ++m) f[m] = l == 0 && Q.f[m] ? Q.f[m][hp] : 0.0;
    // the coefficients of vec_op_dc
    const double* __restrict__ V = L.vc;
    if (G == SPH) {
      const long qs = (long)L.n0 * L.n1, at = (long)t.j * L.n0 + t.i;
      auto cf = [&](int m) { return V[m * qs + at]; };
#pragma unroll
      for (int m = 0; m < 5; ++m) {
        a[m] = cf(m);
        b[m] = cf(12 + m);
        c[m] = cf(22 + m);
        a[6 + m] = cf(6 + m);
      }
      a[5] = cf(33), b[5] = cf(34), c[5] = cf(35), a[11] = cf(11);
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        b[6 + m] = cf(18 + m);
        c[6 + m] = cf(28 + m);
      }
#pragma unroll
      for (int m = 0; m < 3; ++m) iD[m] = cf(36 + m);
    } else if (G == CYL) {
      auto cf = [&](int m) { return V[m * L.n0 + t.i]; };
      const double ih1 = L.ih1s;
      a[0] = cf(0), a[1] = cf(1), a[2] = a[3] = ih1, a[4] = cf(2), a[5] = cf(3);
      a[6] = a[7] = a[8] = 0.0, a[9] = cf(4), a[10] = cf(5), a[11] = cf(6);
      b[0] = cf(8), b[1] = cf(9), b[2] = b[3] = cf(10), b[4] = cf(11), b[5] = 0.0;
      b[6] = cf(12), b[7] = cf(4), b[8] = 0.0, b[9] = cf(13);
      c[0] = cf(8), c[1] = cf(9), c[2] = c[3] = cf(15), c[4] = cf(16), c[5] = cf(17);
      c[6] = cf(18), c[7] = cf(6), c[8] = 0.0, c[9] = cf(13);
      iD[0] = cf(7), iD[1] = cf(14), iD[2] = cf(19);
    } else {
      auto cf = [&](int m) { return V[m]; };
      a[0] = a[1] = cf(3), a[2] = a[3] = cf(1), a[4] = cf(2), a[5] = a[6] = a[7] = a[8] = a[10] = 0.0;
      a[9] = cf(6), a[11] = cf(7);
      b[0] = b[1] = cf(0), b[2] = b[3] = cf(4), b[4] = cf(2), b[5] = b[6] = b[8] = 0.0, b[7] = cf(6), b[9] = cf(8);
      c[0] = c[1] = cf(0), c[2] = c[3] = cf(1), c[4] = cf(5), c[5] = c[6] = c[8] = 0.0, c[7] = cf(7), c[9] = cf(8);
#pragma unroll
      for (int m = 0; m < 3; ++m) iD[m] = cf(9 + m);
    }
  }
  __device__ __forceinline__ double mix(const double* F, int p, int q) const {
    return ((F[p + q] - F[p - q]) - F[q - p]) + F[-p - q];
  }
  // (lap V + 1/3 grad div V)_m - f_m at the own cell
  template <int M>
  __device__ __forceinline__ double defect() const {
    const double *A = u[0] + t.p, *B = u[1] + t.p, *C = u[2] + t.p;
    const int sx = (int)L.sx, sy = (int)L.sy;
    const double* w = M == 0 ? a : (M == 1 ? b : c);
    const double* F = M == 0 ? A : (M == 1 ? B : C);
    const double v = F[0];
    double s = fma(w[0], F[1] - v, w[1] * (F[-1] - v)), r = fma(w[2], F[sx] - v, w[3] * (F[-sx] - v));
    if (L.three) s = fma(w[4], (F[sy] - v) + (F[-sy] - v), s);
    double y = M == 1 || (M == 0 && G == CART) ? 0.0 : w[5] * v;
    if (M == 1 && G == SPH) y = w[5] * v;
    if (M == 0) {
      if (G == SPH) y = fma(w[6], B[sx] - B[-sx], fma(w[7], B[0], fma(w[8], B[1] - B[-1], y)));
      r = fma(w[9], mix(B, 1, sx), r);
      if (L.three) y = fma(w[10], C[sy] - C[-sy], fma(w[11], mix(C, 1, sy), y));
    } else if (M == 1) {
      if (G != CART) y = fma(w[6], A[sx] - A[-sx], y);
      r = fma(w[7], mix(A, 1, sx), r);
      if (L.three) {
        if (G == SPH) y = fma(w[8], C[sy] - C[-sy], y);
        y = fma(w[9], mix(C, sx, sy), y);
      }
    } else if (L.three) {
      if (G != CART) y = fma(w[6], A[sy] - A[-sy], y);
      y = fma(w[7], mix(A, 1, sy), y);
      if (G == SPH) r = fma(w[8], B[sy] - B[-sy], r);
      r = fma(w[9], mix(B, sx, sy), r);
    }
    return ((s + r) + y) - f[M];
  }
  __device__ __forceinline__ void put(double* const* F, int m, double v) {
    double* p = F[m] + t.p;
    *p = v;
    for (unsigned k = mask; k; k &= k - 1u) cl_store(cl_addr(p), __ffs(k) - 1, v);
  }
  __device__ __forceinline__ void fill(double* const* F, int m) {
    auto one = [&](uint2 q) {
      const double v = F[m][q.x >> 16];
      F[m][q.x & 0xffffu] = (q.y >> m) & 1u ? -v : v;
    };
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (t.tid + r * FV_THREADS < nlist) one(g[r]);
    for (int q = t.tid + 2 * FV_THREADS; q < nlist; q += FV_THREADS) one(list[q]);
  }
  __device__ __forceinline__ void fill(double* const* F) {
#pragma unroll
    for (int m = 0; m < 3; ++m) fill(F, m);
  }
  template <int M>
  __device__ __forceinline__ void pass(int colour) {
    if (t.on && t.colour == colour) put(u, M, u[M][t.p] - defect<M>() * iD[M]);
    t.sync();
    fill(u, M);
    __syncthreads();
  }
  __device__ __forceinline__ void sweeps(int n) {
#pragma unroll 1
    for (int h = 0; h < 2 * n; ++h) {
      pass<0>(h & 1);
      pass<1>(h & 1);
      pass<2>(h & 1);
    }
  }
  // Right-hand side L_H(u_H) + R r of a level below the first (u_H current
  // but for its ghosts).  It reads what the first sweep replaces.
  __device__ __forceinline__ void rhs() {
    fill(u);
    __syncthreads();
    if (!t.on) return;
    f[0] = defect<0>() + x[0][t.p];
    f[1] = defect<1>() + x[1][t.p];
    f[2] = defect<2>() + x[2][t.p];
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      slot[m * FV_THREADS] = f[m];
      slot[(3 + m) * FV_THREADS] = u[m][t.p];
    }
  }
  __device__ __forceinline__ void recall() {
    if (!t.on) return;
#pragma unroll
    for (int m = 0; m < 3; ++m) f[m] = slot[m * FV_THREADS];
  }
  __device__ __forceinline__ void restrict_to(const FasVecCycle& Q, int l, const ClCell& tc, double* sm, double* w) {
    if (t.on) {
      w[t.tid] = -wt * defect<0>();
      w[FV_THREADS + t.tid] = -wt * defect<1>();
      w[2 * FV_THREADS + t.tid] = -wt * defect<2>();
#pragma unroll
      for (int m = 0; m < 3; ++m) w[(3 + m) * FV_THREADS + t.tid] = wt * u[m][t.p];
    }
    __syncthreads();
    const FasVecLevel& C = Q.lv[l + 1];
    for (int q = t.tid; q < 6 * t.groups; q += FV_THREADS) {
      const int m = q / t.groups, gr = q - m * t.groups, cell = (t.rank << t.lgroups) + gr;
      int I, J, K;
      C.v.cell(cell, I, J, K);
      const int p = (int)C.v.idx(I, J, K), to = tc.size > 1 ? tc.owner(C.v, I, J, K) : 0;
      const double s = t.group_sum(w + m * FV_THREADS, gr);
      if (m < 3) {
        cl_store(cl_addr(sm + C.x_at + m * C.ng + p), to, s);
      } else {
        const unsigned d = cl_addr(sm + C.u_at + (m - 3) * C.ng + p);
        for (unsigned k = (C.mask ? (unsigned)C.mask[cell] : 0u) | 1u << to; k; k &= k - 1u) cl_store(d, __ffs(k) - 1, s);
      }
    }
  }
  __device__ __forceinline__ void prolong(const FasVecCycle& Q, int l, bool remote, double* sm) {
    if (!t.on) return;
    const FasVecLevel& T = Q.lv[l + 1];
    const LevelView<double>& C = T.v;
    const int pc = (int)C.idx(t.i >> 1, t.j >> 1, L.three ? (t.k >> 1) : 0);
    const int si = (t.i & 1) ? 1 : -1, sj = ((t.j & 1) ? 1 : -1) * (int)C.sx, sk = ((t.k & 1) ? 1 : -1) * (int)C.sy;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const double* e = sm + T.x_at + m * T.ng;
      if (remote) e = cg::this_cluster().map_shared_rank(e, 0);
      e += pc;
      const double add = L.three ? 0.25 * (e[0] + e[si] + e[sj] + e[sk]) : 0.25 * (2.0 * e[0] + e[si] + e[sj]);
      put(u, m, u[m][t.p] + add);
    }
  }
  // u - uh for the finer level, with its ghosts.
  __device__ __forceinline__ void correction() {
    if (t.on)
#pragma unroll
      for (int m = 0; m < 3; ++m) put(x, m, u[m][t.p] - slot[(3 + m) * FV_THREADS]);
    t.sync();
    fill(x);
    __syncthreads();
  }
  __device__ __forceinline__ void out(const FasVecCycle& Q) const {
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      if (t.on) Q.u[m][hp] = u[m][t.p];
      for (int q = t.tid; q < nlist; q += FV_THREADS) Q.u[m][list[q].y >> 3] = u[m][list[q].x & 0xffffu];
    }
  }
};

template <int G>
__global__ void __launch_bounds__(FV_THREADS, 1) k_fas_vec_cycle(const __grid_constant__ FasVecCycle Q) {
  extern __shared__ __align__(16) double fv_smem[];
  __shared__ CoarseShared cs;
  double* const sm = fv_smem;
  double* const w = sm + Q.w_at;
  const int rank = (int)cg::this_cluster().block_rank(), size = (int)cg::this_cluster().num_blocks(), nl = Q.nl;
  pdl_entry();
  {
    // u of the first level, ghosts included
    const FasVecLevel& T = Q.lv[0];
    const LevelView<double>& L = T.v;
    const int nx = L.n0 + 2, ny = L.n1 + 2;
    for (int q = threadIdx.x; q < T.ng; q += FV_THREADS) {
      const int r = q / nx, i = q - r * nx - 1, kz = r / ny, j = r - kz * ny - 1, k = L.three ? kz - 1 : 0;
      const long p = Q.off + i + j * Q.sx + k * Q.sy;
#pragma unroll
      for (int m = 0; m < 3; ++m) sm[T.u_at + m * T.ng + q] = Q.u[m][p];
    }
  }
  auto team = [&](int l) { return l < Q.solo_from ? size : 1; };
  cl_sync();  // every block has started
  for (int l = 0; l + 1 < nl && rank < team(l); ++l) {
    const ClCell t(Q.lv[l].v, rank, team(l)), tc(Q.lv[l + 1].v, rank, team(l + 1));
    FasVec<G> T(t, Q, l, sm);
    if (l > 0) {
      T.rhs();
      t.sync();  // every right-hand side before the first new value
    }
    T.sweeps(Q.nu1);
    T.restrict_to(Q, l, tc, sm, w);
    t.sync();
  }
  if (rank == 0) {
    const LevelView<double>& L = Q.lv[nl - 1].v;
    const ClCell t(L, 0, 1);
    FasVec<G> T(t, Q, nl - 1, sm);
    // the coarsest level has no table: its ghosts by the rules
    const long ngh = ghost_count(L);
    auto ghosts = [&](double* const* F) {
#pragma unroll
      for (int m = 0; m < 3; ++m)
        for (long q = threadIdx.x; q < ngh; q += FV_THREADS) fill_one_ghost(L, F[m], m, q);
      __syncthreads();
    };
    ghosts(T.u);
    T.rhs();
    if (t.on)
#pragma unroll
      for (int m = 0; m < 3; ++m) T.x[m][t.p] = T.f[m];
    __syncthreads();
    coarse_vec_rows<G>(cs, L, T.u[0], T.u[1], T.u[2], T.x[0], T.x[1], T.x[2], Q.rows);
    __syncthreads();
    T.correction();
    ghosts(T.x);
  }
  for (int l = nl - 2; l >= 0; --l) {
    if (rank >= team(l)) continue;
    const ClCell t(Q.lv[l].v, rank, team(l));
    FasVec<G> T(t, Q, l, sm);
    if (l > 0) T.recall();
    t.sync();  // the coarse level's correction
    T.prolong(Q, l, team(l) > team(l + 1), sm);
    t.sync();
    T.fill(T.u);
    t.sync();  // the first pass replaces sources of ghosts other blocks refill
    T.sweeps(Q.nu2);
    if (l > 0)
      T.correction();
    else
      T.out(Q);
  }
}

using FasVecKernel = void (*)(FasVecCycle);
static FasVecKernel fas_vec_kernel(int geom) {
  return geom == CART ? k_fas_vec_cycle<CART> : (geom == CYL ? k_fas_vec_cycle<CYL> : k_fas_vec_cycle<SPH>);
}

static cudaLaunchConfig_t fas_vec_config(int cluster, size_t smem, cudaStream_t st, cudaLaunchAttribute* at) {
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cluster);
  cfg.blockDim = dim3(FV_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cfg;
}

// Blocks of a cluster every instantiation can launch with (16, else 8), 0
// when none can.
static int g_fas_vec_cluster = -1;

void init_fas_vec_attributes() {
  int best = 16;
  for (int g = 0; g < 3; ++g) {
    FasVecKernel k = fas_vec_kernel(g);
    cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)FV_SMEM_MAX) != cudaSuccess) {
      cudaGetLastError();
      best = 0;
    }
    for (; g_fas_vec_cluster < 0 && best >= 8; best /= 2) {
      cudaLaunchAttribute at[2];
      cudaLaunchConfig_t cfg = fas_vec_config(best, FV_SMEM_MAX, nullptr, at);
      cfg.numAttrs = 1;
      int nc = 0;
      if (cudaOccupancyMaxActiveClusters(&nc, k, &cfg) == cudaSuccess && nc > 0) break;
      cudaGetLastError();
    }
  }
  if (g_fas_vec_cluster < 0) g_fas_vec_cluster = best >= 8 ? best : 0;
}

bool fas_vec_attributes_set() {
  cudaFuncAttributes a;
  if (cudaFuncGetAttributes(&a, fas_vec_kernel(SPH)) == cudaSuccess) return a.maxDynamicSharedSizeBytes >= (int)FV_SMEM_MAX;
  cudaGetLastError();
  return false;
}

int fas_vec_blocks() { return g_fas_vec_cluster > 0 ? g_fas_vec_cluster : 0; }

void launch_fas_vec_cycle(const FasVecCycle& Q, int geom, cudaStream_t st) {
  count_launch();
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t cfg = fas_vec_config(g_fas_vec_cluster, Q.smem, st, at);
  cudaLaunchKernelEx(&cfg, fas_vec_kernel(geom), Q);
}

}  // namespace gmg
