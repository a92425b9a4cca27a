// The FP32 correction V-cycle from a level of 2048 to 8192 cells down in one
// launch of a thread-block cluster: levels of more than CL_SOLO_CELLS cells
// on all its blocks, smaller ones on the first, the coarsest solve as in
// mg_block.cuh.
//
// Launched, a colour pass of such a level is its launch and one L2 round
// trip, 2.5 us and more whatever its size (24 of them per vector cycle); in
// one block it is the instructions of its cells, ~0.45 us (800 cycles) even
// for a few dozen of them: index arithmetic, metric factors, a division.
// Here a thread owns one cell: its stencil coefficients and right-hand side
// stay in registers over the sweeps of a visit, every block holds the level's
// correction in shared memory, and a new value is stored into the blocks that
// read it (distributed shared memory).  A pass is a barrier (the cluster's
// ~400 cycles), the neighbours' shared loads and one cell's multiply-adds;
// for the vector equation also the refill of the ghosts the block reads, each
// plus or minus an interior cell (their sources and the blocks that read a
// cell come from a table the host builds once per hierarchy).  Mixed xCFC on
// 64 x 128 cylindrical cells 4.92 to 3.90 ms per solve, on 128 x 64 x 64
// spherical ones (32 x 16 x 16 and below here) 228 to 212 ms.
#include <cooperative_groups.h>

#include "mg_block.cuh"
#include "mg_cell.cuh"
#include "mg_internal.h"
#include "mg_kernels.cuh"

namespace cg = cooperative_groups;

namespace gmg {

// ------------------------------------------------------ scalar equations

template <int G>
struct ClScalar {
  const ClCell& t;
  const LevelView<float>& L;
  float* e;          // the level's cells, without ghosts
  unsigned mask;     // blocks that own a neighbour
  int q, nb[6];
  float c[5], cC, iD, f, K, wt, u;
  // down: resolve the stencil and keep it in shared memory for the visit up
  __device__ __forceinline__ ClScalar(const ClCell& t_, const ClusterCycle32& Q, int l, float* sm, bool down)
      : t(t_), L(Q.P.lv[l].v), e(sm + Q.P.lv[l].e[0]), mask(0) {
    if (!t.on) return;
    const BlockLevel32& B = Q.P.lv[l];
    float* const slot = sm + Q.slot_at[l] + t.tid;
    const int stride = 2 * t.half;
    if (!down) {
      q = t.i + L.n0 * (t.j + L.n1 * t.k);
#pragma unroll
      for (int m = 0; m < 5; ++m) c[m] = slot[m * stride];
      cC = slot[5 * stride];
      iD = slot[6 * stride];
      f = slot[7 * stride];
#pragma unroll
      for (int m = 0; m < 3; ++m) {
        const unsigned x = __float_as_uint(slot[(8 + m) * stride]);
        nb[2 * m] = (int)(x & 0xffffu);
        nb[2 * m + 1] = (int)(x >> 16);
      }
      mask = __float_as_uint(slot[11 * stride]);
      u = e[q];
      return;
    }
    wt = t.weight(L);
    const int n0 = L.n0, n1 = L.n1, n2 = L.n2, i = t.i, j = t.j, k = t.k;
    q = i + n0 * (j + n1 * k);
    c[0] = L.TI(TI_CE, i);
    c[1] = L.TI(TI_CW, i);
    if (G == SPH) {
      const float ir2 = L.TI(TI_IX2, i);
      c[2] = ir2 * L.TJ(TJ_TN, j);
      c[3] = ir2 * L.TJ(TJ_TS, j);
    } else {
      c[2] = c[3] = L.ih1s;
    }
    c[4] = 0.0f;
    if (L.three) c[4] = G == CART ? L.ih2s : (G == CYL ? L.TI(TI_PHI, i) : L.TI(TI_IX2, i) * L.TJ(TJ_PF, j));
    K = l > 0 && Q.P.fold_k ? sm[B.k_at + t.p] : (Q.lv[l].k ? Q.lv[l].k[t.p] : 0.0f);
    f = l > 0 ? sm[B.f32[0] + t.p] : Q.P.f_in[0][t.p];
    u = e[q];
    iD = 1.0f / (-(c[0] + c[1]) - (c[2] + c[3]) - 2.0f * c[4] - K);
    // an outer ghost is a factor times the cell's own value; across the
    // origin and the poles the coupling is zero; phi wraps
    cC = -K;
    auto side = [&](int m, int d, int s) {
      int a = i + (d == 0) * s, b = j + (d == 1) * s, h = k + (d == 2) * s;
      const bool out = d == 0 ? (a < 0 || a >= n0) : (d == 1 ? (b < 0 || b >= n1) : (h < 0 || h >= n2));
      nb[m] = q;
      if (d == 2 && !L.three) return;
      if (out && d == 2 && G != CART) {
        h &= n2 - 1;
      } else if (out) {
        const bool zero = (G != CART && d == 0 && s < 0) || (G == SPH && d == 1);
        const float cf = d == 0 ? c[m] : (d == 1 ? c[m] : c[4]);
        if (!zero) cC += cf * (outer_factor(L, a, b, h, i, j, k) - 1.0f);
        return;
      }
      nb[m] = a + n0 * (b + n1 * h);
      mask |= 1u << t.owner(L, a, b, h);
    };
    side(0, 0, 1);
    side(1, 0, -1);
    side(2, 1, 1);
    side(3, 1, -1);
    side(4, 2, 1);
    side(5, 2, -1);
    mask &= ~(1u << t.rank);
#pragma unroll
    for (int m = 0; m < 5; ++m) slot[m * stride] = c[m];
    slot[5 * stride] = cC;
    slot[6 * stride] = iD;
    slot[7 * stride] = f;
#pragma unroll
    for (int m = 0; m < 3; ++m) slot[(8 + m) * stride] = __uint_as_float((unsigned)nb[2 * m] | (unsigned)nb[2 * m + 1] << 16);
    slot[11 * stride] = __uint_as_float(mask);
  }
  // L e - K e - f
  __device__ __forceinline__ float defect() const {
    float a = fmaf(c[0], e[nb[0]] - u, fmaf(cC, u, -f)), b = c[2] * (e[nb[2]] - u);
    a = fmaf(c[1], e[nb[1]] - u, a);
    b = fmaf(c[3], e[nb[3]] - u, b);
    if (L.three) a = fmaf(c[4], (e[nb[4]] - u) + (e[nb[5]] - u), a);
    return a + b;
  }
  __device__ __forceinline__ void put(bool others) {
    e[q] = u;
    if (others)
      for (unsigned m = mask; m; m &= m - 1u) cl_store(cl_addr(e + q), __ffs(m) - 1, u);
  }
  __device__ __forceinline__ void sweeps(int n, bool last) {
    for (int h = 0; h < 2 * n; ++h) {
      const bool end = last && h == 2 * n - 1;
      if (t.on && t.colour == (h & 1)) {
        u -= defect() * iD;
        put(!end);
      }
      if (!end) t.sync();
    }
  }
  __device__ __forceinline__ void restrict_to(const BlockCycle32& P, int l, const ClCell& tc, float* sm, float* w) {
    if (t.on) {
      w[t.tid] = -wt * defect();
      if (P.fold_k) w[BC_THREADS + t.tid] = wt * K;
    }
    __syncthreads();
    const int m = t.tid >= t.groups;
    if (t.tid < (P.fold_k ? 2 : 1) * t.groups) {
      const int g = t.tid - m * t.groups;
      const BlockLevel32& C = P.lv[l + 1];
      int I, J, K3;
      C.v.cell(t.rank * t.groups + g, I, J, K3);
      cl_store(cl_addr(sm + (m ? C.k_at : C.f32[0]) + C.v.idx(I, J, K3)), tc.size > 1 ? tc.owner(C.v, I, J, K3) : 0,
               t.group_sum(w + m * BC_THREADS, g));
    }
  }
  __device__ __forceinline__ void prolong(const BlockCycle32& P, int l, bool remote, float* sm) {
    if (!t.on) return;
    const LevelView<float>& C = P.lv[l + 1].v;
    const float* ec = sm + P.lv[l + 1].e[0];
    if (remote) ec = cg::this_cluster().map_shared_rank(ec, 0);
    // the coarsest level's array has ghosts
    auto value = [&](int a, int b, int d) {
      return l + 2 == P.nl ? ec[C.idx(a, b, d)] : ec[a + C.n0 * (b + C.n1 * d)];
    };
    const int I = t.i >> 1, J = t.j >> 1, K3 = L.three ? (t.k >> 1) : 0;
    auto side = [&](int d) {
      int x = I, y = J, z = K3;
      bool out;
      if (d == 0) {
        x += (t.i & 1) ? 1 : -1;
        out = x < 0 || x >= C.n0;
      } else if (d == 1) {
        y += (t.j & 1) ? 1 : -1;
        out = y < 0 || y >= C.n1;
      } else {
        z += (t.k & 1) ? 1 : -1;
        out = z < 0 || z >= C.n2;
      }
      const float g = out ? ghost_rule(C, -1, d, x, y, z) : 1.0f;
      return g * value(x, y, z);
    };
    const float e0 = value(I, J, K3), x = side(0), y = side(1);
    if (L.three)
      u += 0.25f * (e0 + x + y + side(2));
    else
      u += 0.25f * (2.0f * e0 + x + y);
    put(true);
  }
  // The final values, for the finer level: to every block, or out.
  __device__ __forceinline__ void finish(const ClusterCycle32& Q, int l) {
    if (!t.on) return;
    if (l == 0)
      Q.P.e_out[0][t.p] = u;
    else
      for (int b = 0; b < t.size; ++b) cl_store(cl_addr(e + q), b, u);
  }
  __device__ __forceinline__ void fill() {}
};

// ------------------------------------------------------ vector equations

template <int G>
struct ClVector {
  const ClCell& t;
  const LevelView<float>& L;
  float* e[3];         // ghosted components
  unsigned mask;       // blocks that read the cell
  const uint2* list;   // ghosts this block reads: ghost | source << 16, sign per component
  int nlist;
  uint2 g[2];
  long hp;             // the cell in HBM
  float wt;
  float a[12], b[10], c[10], iD[3], f[3];
  __device__ __forceinline__ ClVector(const ClCell& t_, const ClusterCycle32& Q, int l, float* sm, bool down)
      : t(t_), L(Q.P.lv[l].v), mask(0) {
    const BlockLevel32& W = Q.P.lv[l];
    const ClusterLevel32& T = Q.lv[l];
#pragma unroll
    for (int m = 0; m < 3; ++m) e[m] = sm + W.e[m];
    list = T.list + T.start[t.rank];
    nlist = T.start[t.rank + 1] - T.start[t.rank];
#pragma unroll
    for (int r = 0; r < 2; ++r)
      g[r] = t.tid + r * BC_THREADS < nlist ? list[t.tid + r * BC_THREADS] : make_uint2(0, 0);
    if (!t.on) return;
    if (down) wt = t.weight(L);
    hp = Q.off + t.i + t.j * Q.sx + t.k * Q.sy;
    mask = T.mask[t.i + L.n0 * (t.j + L.n1 * t.k)];
#pragma unroll
    for (int m = 0; m < 3; ++m) f[m] = l > 0 ? sm[W.f32[m] + t.p] : Q.P.f_in[m][hp];
    // the coefficients of vec_op_dc
    const float* __restrict__ V = T.vc;
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
      const float ih1 = L.ih1s;
      a[0] = cf(0), a[1] = cf(1), a[2] = a[3] = ih1, a[4] = cf(2), a[5] = cf(3);
      a[6] = a[7] = a[8] = 0.0f, a[9] = cf(4), a[10] = cf(5), a[11] = cf(6);
      b[0] = cf(8), b[1] = cf(9), b[2] = b[3] = cf(10), b[4] = cf(11), b[5] = 0.0f;
      b[6] = cf(12), b[7] = cf(4), b[8] = 0.0f, b[9] = cf(13);
      c[0] = cf(8), c[1] = cf(9), c[2] = c[3] = cf(15), c[4] = cf(16), c[5] = cf(17);
      c[6] = cf(18), c[7] = cf(6), c[8] = 0.0f, c[9] = cf(13);
      iD[0] = cf(7), iD[1] = cf(14), iD[2] = cf(19);
    } else {
      auto cf = [&](int m) { return V[m]; };
      a[0] = a[1] = cf(3), a[2] = a[3] = cf(1), a[4] = cf(2), a[5] = a[6] = a[7] = a[8] = a[10] = 0.0f;
      a[9] = cf(6), a[11] = cf(7);
      b[0] = b[1] = cf(0), b[2] = b[3] = cf(4), b[4] = cf(2), b[5] = b[6] = b[8] = 0.0f, b[7] = cf(6), b[9] = cf(8);
      c[0] = c[1] = cf(0), c[2] = c[3] = cf(1), c[4] = cf(5), c[5] = c[6] = c[8] = 0.0f, c[7] = cf(7), c[9] = cf(8);
#pragma unroll
      for (int m = 0; m < 3; ++m) iD[m] = cf(9 + m);
    }
  }
  __device__ __forceinline__ float mix(const float* F, int x, int y) const {
    return ((F[x + y] - F[x - y]) - F[y - x]) + F[-x - y];
  }
  // (lap V + 1/3 grad div V)_m - f_m at the own cell
  template <int M>
  __device__ __forceinline__ float defect() const {
    const float *A = e[0] + t.p, *B = e[1] + t.p, *C = e[2] + t.p;
    const int sx = (int)L.sx, sy = (int)L.sy;
    const float* w = M == 0 ? a : (M == 1 ? b : c);
    const float* F = M == 0 ? A : (M == 1 ? B : C);
    const float v = F[0];
    float s = fmaf(w[0], F[1] - v, w[1] * (F[-1] - v)), r = fmaf(w[2], F[sx] - v, w[3] * (F[-sx] - v));
    float x = fmaf(w[5], v, -f[M]);
    if (L.three) s = fmaf(w[4], (F[sy] - v) + (F[-sy] - v), s);
    if (M == 0) {
      if (G == SPH) x = fmaf(w[6], B[sx] - B[-sx], fmaf(w[7], B[0], fmaf(w[8], B[1] - B[-1], x)));
      r = fmaf(w[9], mix(B, 1, sx), r);
      if (L.three) x = fmaf(w[10], C[sy] - C[-sy], fmaf(w[11], mix(C, 1, sy), x));
    } else if (M == 1) {
      x = fmaf(w[6], A[sx] - A[-sx], x);
      r = fmaf(w[7], mix(A, 1, sx), r);
      if (L.three) x = fmaf(w[8], C[sy] - C[-sy], fmaf(w[9], mix(C, sx, sy), x));
    } else if (L.three) {
      x = fmaf(w[6], A[sy] - A[-sy], fmaf(w[7], mix(A, 1, sy), x));
      r = fmaf(w[8], B[sy] - B[-sy], fmaf(w[9], mix(B, sx, sy), r));
    }
    return (s + r) + x;
  }
  __device__ __forceinline__ void put(int m, float v) {
    float* p = e[m] + t.p;
    *p = v;
    for (unsigned k = mask; k; k &= k - 1u) cl_store(cl_addr(p), __ffs(k) - 1, v);
  }
  __device__ __forceinline__ void fill(int m) {
    auto one = [&](uint2 a) {
      const float x = e[m][a.x >> 16];
      e[m][a.x & 0xffffu] = (a.y >> m) & 1u ? -x : x;
    };
#pragma unroll
    for (int r = 0; r < 2; ++r)
      if (t.tid + r * BC_THREADS < nlist) one(g[r]);
    for (int q = t.tid + 2 * BC_THREADS; q < nlist; q += BC_THREADS) one(list[q]);
  }
  __device__ __forceinline__ void fill() {
#pragma unroll
    for (int m = 0; m < 3; ++m) fill(m);
    t.sync();  // the first pass replaces sources of ghosts other blocks refill
  }
  template <int M>
  __device__ __forceinline__ void pass(int colour) {
    if (t.on && t.colour == colour) put(M, e[M][t.p] - defect<M>() * iD[M]);
    t.sync();
    fill(M);
    __syncthreads();
  }
  __device__ __forceinline__ void sweeps(int n, bool) {
#pragma unroll 1
    for (int h = 0; h < 2 * n; ++h) {
      pass<0>(h & 1);
      pass<1>(h & 1);
      pass<2>(h & 1);
    }
  }
  __device__ __forceinline__ void restrict_to(const BlockCycle32& P, int l, const ClCell& tc, float* sm, float* w) {
    if (t.on) {
      w[t.tid] = -wt * defect<0>();
      w[BC_THREADS + t.tid] = -wt * defect<1>();
      w[2 * BC_THREADS + t.tid] = -wt * defect<2>();
    }
    __syncthreads();
    if (t.tid < 3 * t.groups) {
      const int m = t.tid / t.groups, g = t.tid - m * t.groups;
      const BlockLevel32& C = P.lv[l + 1];
      int I, J, K3;
      C.v.cell(t.rank * t.groups + g, I, J, K3);
      cl_store(cl_addr(sm + C.f32[m] + C.v.idx(I, J, K3)), tc.size > 1 ? tc.owner(C.v, I, J, K3) : 0,
               t.group_sum(w + m * BC_THREADS, g));
    }
  }
  __device__ __forceinline__ void prolong(const BlockCycle32& P, int l, bool remote, float* sm) {
    if (!t.on) return;
    const LevelView<float>& C = P.lv[l + 1].v;
    const int pc = (int)C.idx(t.i >> 1, t.j >> 1, L.three ? (t.k >> 1) : 0);
    const int si = (t.i & 1) ? 1 : -1, sj = ((t.j & 1) ? 1 : -1) * (int)C.sx, sk = ((t.k & 1) ? 1 : -1) * (int)C.sy;
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const float* ec = sm + P.lv[l + 1].e[m];
      if (remote) ec = cg::this_cluster().map_shared_rank(ec, 0);
      ec += pc;
      const float add = L.three ? 0.25f * (ec[0] + ec[si] + ec[sj] + ec[sk]) : 0.25f * (2.0f * ec[0] + ec[si] + ec[sj]);
      put(m, e[m][t.p] + add);
    }
  }
  __device__ __forceinline__ void finish(const ClusterCycle32& Q, int l) const {
    if (l > 0) return;  // the blocks that prolong from a value read it
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      if (t.on) Q.P.e_out[m][hp] = e[m][t.p];
      for (int q = t.tid; q < nlist; q += BC_THREADS) Q.P.e_out[m][list[q].y >> 3] = e[m][list[q].x & 0xffffu];
    }
  }
};

template <int G, bool VEC>
__global__ void __launch_bounds__(BC_THREADS, 1) k_cluster_vcycle32(const __grid_constant__ ClusterCycle32 Q) {
  const BlockCycle32& P = Q.P;
  float* const sm = bc_smem();
  float* const w = sm + Q.w_at;
  const int rank = (int)cg::this_cluster().block_rank(), size = (int)cg::this_cluster().num_blocks(), nl = P.nl;
  using Top = typename std::conditional<VEC, ClVector<G>, ClScalar<G>>::type;
  for (int l = 0; l < nl; ++l) {
    const LevelView<float>& L = P.lv[l].v;
    const int ng = (int)L.sy * (L.n2 + 2 * L.three);
#pragma unroll
    for (int c = 0; c < (VEC ? 3 : 1); ++c)
      for (int q = threadIdx.x; q < (ng + 3) / 4; q += BC_THREADS)
        reinterpret_cast<float4*>(sm + P.lv[l].e[c])[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
  if (rank == 0) bc_stage_tables(P, nl - 1);
  pdl_entry();
  if (rank == 0) {
    if (!VEC && !P.fold_k) bc_stage_k(P, nl - 1);
    bc_rules<G, VEC>(P, nl - 1);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  }
  auto team = [&](int l) { return l < Q.solo_from ? size : 1; };
  cl_sync();  // every block has started, with a zero correction
  for (int l = 0; l + 1 < nl && rank < team(l); ++l) {
    const ClCell t(P.lv[l].v, rank, team(l)), tc(P.lv[l + 1].v, rank, team(l + 1));
    Top T(t, Q, l, sm, true);
    T.sweeps(P.nu1, false);
    T.restrict_to(P, l, tc, sm, w);
    t.sync();
  }
  if (rank == 0) bc_coarse<G, VEC>(P, bc_level<VEC>(P, nl - 1));
  for (int l = nl - 2; l >= 0; --l) {
    if (rank >= team(l)) continue;
    const ClCell t(P.lv[l].v, rank, team(l));
    Top T(t, Q, l, sm, false);
    t.sync();  // the coarse level's values
    T.prolong(P, l, team(l) > team(l + 1), sm);
    t.sync();
    T.fill();
    T.sweeps(P.nu2, true);
    T.finish(Q, l);
  }
}

using ClusterKernel = void (*)(ClusterCycle32);
template <int G>
static ClusterKernel cluster_kernel_g(int vec) {
  return vec ? k_cluster_vcycle32<G, true> : k_cluster_vcycle32<G, false>;
}
static ClusterKernel cluster_kernel(int geom, int vec) {
  return geom == CART ? cluster_kernel_g<CART>(vec) : (geom == CYL ? cluster_kernel_g<CYL>(vec) : cluster_kernel_g<SPH>(vec));
}

static cudaLaunchConfig_t cluster_config(int cluster, size_t smem, cudaStream_t st, cudaLaunchAttribute* at) {
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cluster);
  cfg.blockDim = dim3(BC_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cfg;
}

// Blocks of a cluster every instantiation can launch with (16, else 8), 0
// when none can.
static int g_cluster32 = -1;

void init_cluster_cycle_attributes() {
  int best = 16;
  for (int g = 0; g < 3; ++g)
    for (int vec = 0; vec < 2; ++vec) {
      ClusterKernel k = cluster_kernel(g, vec);
      cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)CL_SMEM_MAX) != cudaSuccess) {
        cudaGetLastError();
        best = 0;
      }
      for (; g_cluster32 < 0 && best >= 8; best /= 2) {
        cudaLaunchAttribute at[2];
        cudaLaunchConfig_t cfg = cluster_config(best, CL_SMEM_MAX, nullptr, at);
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, k, &cfg) == cudaSuccess && nc > 0) break;
        cudaGetLastError();
      }
    }
  if (g_cluster32 < 0) g_cluster32 = best >= 8 ? best : 0;
}

int cluster_cycle_blocks() { return g_cluster32 > 0 ? g_cluster32 : 0; }

void launch_cluster_vcycle32(const ClusterCycle32& Q, int geom, cudaStream_t st) {
  count_launch();
  cudaLaunchAttribute at[2];
  const cudaLaunchConfig_t cfg = cluster_config(g_cluster32, Q.P.smem, st, at);
  cudaLaunchKernelEx(&cfg, cluster_kernel(geom, Q.P.vec), Q);
}

}  // namespace gmg
