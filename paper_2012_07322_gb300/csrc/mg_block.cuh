// The one-block FP32 correction V-cycle as device code: the phases of
// k_block_vcycle32 (mg_block.cu), callable from any kernel whose block has
// BC_THREADS threads and P.smem bytes of dynamic shared memory.
//
// One SM runs a chain of ~100 (scalar) to ~200 (vector) barrier-separated
// phases of at most a few cells per thread, so a phase's time is the
// instructions of one cell.  Hence:
//  - shared-memory addresses, strides and ranks in 32 bits (BcView);
//  - the boundary rules out of the stencil: scalar levels keep their outer
//    ghosts in the array (a ghost is read only by its own boundary cell, so
//    the thread that updates the cell rewrites its ghosts, factors tabulated
//    once per cycle), vector levels copy theirs from a table of sources
//    built once per cycle;
//  - the residual restricted by the thread that owns the coarse cell, and K
//    of eq. psi restricted on the way down (no launches of its own).
// Before, every phase evaluated the rules (square roots for Cartesian and
// cylindrical Robin) for every cell or ghost it touched; per call, cold:
// scalar 36 us (spherical 16x8x8), 67 us (Cartesian 16^3), 71 us
// (cylindrical 32x64); vector 126 us (spherical 16x8x8), 170 us (cylindrical
// 32x64).
#pragma once
#include "mg_internal.h"
#include "mg_kernels.cuh"

namespace gmg {

constexpr int BC_THREADS = 512;

// The dynamic shared memory by its declaration, so that every access
// compiles to a shared-memory instruction (a pointer handed through an
// out-of-line call would be generic).
__device__ __forceinline__ float* bc_smem() {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  return reinterpret_cast<float*>(smem_raw);
}

// LevelView of a level in shared memory: 32-bit strides, tables in shared
// memory.
struct BcView {
  int n0, n1, n2, three, ln0, ln1, mixed, sx, sy, off;
  float ih0s, ih1s, ih2s, hc0, hc1, hc2, m01, m02, m12;
  const float *ti, *tj;
  __device__ __forceinline__ int idx(int i, int j, int k) const { return off + i + j * sx + k * sy; }
  __device__ __forceinline__ float TI(int s, int i) const { return ti[s * (n0 + 2) + i + 1]; }
  __device__ __forceinline__ float TJ(int s, int j) const { return tj[s * (n1 + 2) + j + 1]; }
  __device__ __forceinline__ int cells() const { return n0 * n1 * n2; }
  __device__ __forceinline__ int ghosted() const { return sy * (n2 + 2 * three); }
  __device__ __forceinline__ void cell(int r, int& i, int& j, int& k) const {
    i = r & (n0 - 1);
    const int jk = r >> ln0;
    j = jk & (n1 - 1);
    k = jk >> ln1;
  }
  __device__ __forceinline__ void colour_cell(int r, int colour, int& i, int& j, int& k) const {
    const int jk = r >> (ln0 - 1);
    j = jk & (n1 - 1);
    k = jk >> ln1;
    i = 2 * (r & ((n0 >> 1) - 1)) + ((j + k + colour) & 1);
  }
};

struct BcLevel {
  BcView v;
  float* e[3];
  float* f[3];
  float* k;            // c of (L - c) e = f, or null
  const float* gf;     // scalar levels: factors of the outer ghosts per face, or null: gc on every face;
                       // vector levels: |factor| of every ghost, or null: 1
  int g_at[6];         // offsets of the faces (low, high per dimension) in gf
  float gc;
  const uint2* gt;     // vector levels: ghost | source << 16 offsets, sign bit per component
  int ng;
};

template <bool VEC>
__device__ __forceinline__ BcLevel bc_level(const BlockCycle32& P, int l) {
  float* sm = bc_smem();
  const BlockLevel32& B = P.lv[l];
  BcLevel o;
  BcView& v = o.v;
  v.n0 = B.v.n0, v.n1 = B.v.n1, v.n2 = B.v.n2, v.three = B.v.three;
  v.ln0 = B.v.ln0, v.ln1 = B.v.ln1, v.mixed = B.v.mixed;
  v.sx = (int)B.v.sx, v.sy = (int)B.v.sy, v.off = (int)B.v.off;
  v.ih0s = B.v.ih0s, v.ih1s = B.v.ih1s, v.ih2s = B.v.ih2s;
  v.hc0 = B.v.hc0, v.hc1 = B.v.hc1, v.hc2 = B.v.hc2;
  v.m01 = B.v.m01, v.m02 = B.v.m02, v.m12 = B.v.m12;
  v.ti = sm + B.ti_at;
  v.tj = sm + B.tj_at;
  for (int c = 0; c < (VEC ? 3 : 1); ++c) {
    o.e[c] = sm + B.e[c];
    o.f[c] = sm + B.f32[c];
  }
  o.k = B.k32 ? sm + B.k_at : nullptr;
  o.gf = B.gf_at >= 0 ? sm + B.gf_at : nullptr;
  for (int m = 0; m < 6; ++m) o.g_at[m] = B.g_face[m];
  o.gc = B.gc;
  o.gt = reinterpret_cast<const uint2*>(sm + B.gt_at);
  o.ng = B.ng;
  return o;
}

// A 4-byte asynchronous copy into shared memory.
__device__ __forceinline__ void bc_cp4(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}
__device__ __forceinline__ void bc_cp16(float* dst, const float* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
               : "memory");
}

// Copies of every level's coefficient tables into shared memory
// (asynchronous: bc_run waits); they do not change during a solve.
__device__ __forceinline__ void bc_stage_tables(const BlockCycle32& P, int from = 0) {
  float* sm = bc_smem();
  for (int l = from; l < P.nl; ++l) {
    const BlockLevel32& B = P.lv[l];
    const int nti = NTI * (B.v.n0 + 2), ntj = NTJ * (B.v.n1 + 2);
    for (int q = threadIdx.x; q < nti; q += BC_THREADS) bc_cp4(sm + B.ti_at + q, B.v.ti + q);
    for (int q = threadIdx.x; q < ntj; q += BC_THREADS) bc_cp4(sm + B.tj_at + q, B.v.tj + q);
  }
}

// c of levels from .. to - 1 from HBM (asynchronous).
__device__ __forceinline__ void bc_stage_k(const BlockCycle32& P, int from, int to = BC_MAX) {
  for (int l = from; l < P.nl && l < to; ++l)
    if (P.lv[l].k32) {
      const int ng = (int)(P.lv[l].v.sy * (P.lv[l].v.n2 + 2 * P.lv[l].v.three));
      float* k = bc_smem() + P.lv[l].k_at;
      for (int q = threadIdx.x; q < ng / 4; q += BC_THREADS) bc_cp16(k + 4 * q, P.lv[l].k32 + 4 * q);
    }
}

// Ghost rules of every level, evaluated once per cycle: scalar levels with a
// position-dependent outer factor (Cartesian and cylindrical Robin), the
// factors per face; vector levels, the source and the signs of every ghost
// (+-1 times an interior cell; with the Robin rule a factor as well).
template <int G, bool VEC>
__device__ __forceinline__ void bc_rules(const BlockCycle32& P, int from = 0) {
  float* sm = bc_smem();
  for (int l = from; l < P.nl; ++l) {
    const BlockLevel32& B = P.lv[l];
    const LevelView<float>& L = B.v;
    if (VEC) {
      uint2* gt = reinterpret_cast<uint2*>(sm + B.gt_at);
      for (int g = threadIdx.x; g < B.ng; g += BC_THREADS) {
        int i, j, k;
        ghost_coords(L, g, i, j, k);
        const unsigned dst = (unsigned)L.idx(i, j, k);
        unsigned sign = 0, src = 0;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          int si = i, sj = j, sk = k;
          float f0, f1, f2;
          ghost_source(L, c, si, sj, sk, f0, f1, f2);
          src = (unsigned)L.idx(si, sj, sk);
          sign |= ((f0 * f1) * f2 < 0.0f ? 1u : 0u) << c;
        }
        gt[g] = make_uint2(dst | src << 16, sign);
        if (B.gf_at >= 0) {  // Robin vectors: outer factors other than one
          float f0, f1, f2;
          ghost_source(L, 0, i, j, k, f0, f1, f2);
          sm[B.gf_at + g] = fabsf((f0 * f1) * f2);
        }
      }
    } else if (G != SPH && B.gf_at >= 0) {
      float* gf = sm + B.gf_at;
      const int n0 = L.n0, n1 = L.n1, n2 = L.n2;
      for (int q = threadIdx.x; q < n1 * n2; q += BC_THREADS) {
        const int j = q & (n1 - 1), k = q >> L.ln1;
        gf[B.g_face[1] + q] = outer_factor(L, n0, j, k, n0 - 1, j, k);
        if (G == CART) gf[B.g_face[0] + q] = outer_factor(L, -1, j, k, 0, j, k);
      }
      for (int q = threadIdx.x; q < n0 * n2; q += BC_THREADS) {
        const int i = q & (n0 - 1), k = q >> L.ln0;
        gf[B.g_face[2] + q] = outer_factor(L, i, -1, k, i, 0, k);
        gf[B.g_face[3] + q] = outer_factor(L, i, n1, k, i, n1 - 1, k);
      }
      if (G == CART && L.three)
        for (int q = threadIdx.x; q < n0 * n1; q += BC_THREADS) {
          const int i = q & (n0 - 1), j = q >> L.ln0;
          gf[B.g_face[4] + q] = outer_factor(L, i, j, -1, i, j, 0);
          gf[B.g_face[5] + q] = outer_factor(L, i, j, n2, i, j, n2 - 1);
        }
    }
  }
}

// ---------------------------------------------------------- scalar levels

// Value v of cell (i, j, k) with the outer ghosts it sources.  (Across the
// origin, the axis and the poles the flux coefficient is zero: those ghosts
// stay zero.)
template <int G>
__device__ __forceinline__ void bc_put(const BcLevel& B, int p, int i, int j, int k, float v) {
  const BcView& L = B.v;
  float* e = B.e[0];
  e[p] = v;
  auto fac = [&](int face, int q) { return B.gf ? B.gf[B.g_at[face] + q] : B.gc; };
  if (i == L.n0 - 1) e[p + 1] = fac(1, j + L.n1 * k) * v;
  if (G == CART && i == 0) e[p - 1] = fac(0, j + L.n1 * k) * v;
  if (G != SPH) {
    if (j == L.n1 - 1) e[p + L.sx] = fac(3, i + L.n0 * k) * v;
    if (j == 0) e[p - L.sx] = fac(2, i + L.n0 * k) * v;
  }
  if (G == CART && L.three) {
    if (k == L.n2 - 1) e[p + L.sy] = fac(5, i + L.n0 * j) * v;
    if (k == 0) e[p - L.sy] = fac(4, i + L.n0 * j) * v;
  }
}

// Flux-form Laplacian (lap_scalar) with the ghosts in the array; phi wraps.
template <int G>
__device__ __forceinline__ float bc_lap(const BcView& L, const float* e, int p, int i, int j, int k, float uc,
                                        float& D) {
  const float cE = L.TI(TI_CE, i), cW = L.TI(TI_CW, i);
  float Lu = cE * (e[p + 1] - uc) - cW * (uc - e[p - 1]);
  D = -(cE + cW);
  if (G == SPH) {
    const float ir2 = L.TI(TI_IX2, i);
    const float tN = L.TJ(TJ_TN, j), tS = L.TJ(TJ_TS, j);
    Lu += ir2 * (tN * (e[p + L.sx] - uc) - tS * (uc - e[p - L.sx]));
    D -= ir2 * (tN + tS);
  } else {
    Lu += L.ih1s * (e[p + L.sx] - 2.0f * uc + e[p - L.sx]);
    D -= 2.0f * L.ih1s;
  }
  if (L.three) {
    float c;
    if (G == CART)
      c = L.ih2s;
    else if (G == CYL)
      c = L.TI(TI_PHI, i);
    else
      c = L.TI(TI_IX2, i) * L.TJ(TJ_PF, j);
    int pu = p + L.sy, pd = p - L.sy;
    if (G != CART) {
      if (k == L.n2 - 1) pu = p - (L.n2 - 1) * L.sy;
      if (k == 0) pd = p + (L.n2 - 1) * L.sy;
    }
    Lu += c * (e[pu] - 2.0f * uc + e[pd]);
    D -= 2.0f * c;
  }
  return Lu;
}

template <int G>
__device__ __forceinline__ void bc_smooth_scalar(const BcLevel& B, int nsweeps) {
  const BcView& L = B.v;
  const int nh = L.cells() / 2;
  const float *e = B.e[0], *f = B.f[0], *kk = B.k;
  for (int h = 0; h < 2 * nsweeps; ++h) {
    for (int q = threadIdx.x; q < nh; q += BC_THREADS) {
      int i, j, k;
      L.colour_cell(q, h & 1, i, j, k);
      const int p = L.idx(i, j, k);
      const float uc = e[p];
      float D;
      float Lu = bc_lap<G>(L, e, p, i, j, k, uc, D);
      if (kk) {
        const float c = kk[p];
        Lu -= c * uc;
        D -= c;
      }
      bc_put<G>(B, p, i, j, k, uc - (Lu - f[p]) / D);
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------- vector levels

// The ghosts of component c from their sources.
__device__ __forceinline__ void bc_fill(const BcLevel& B, float* V, int c) {
  for (int g = threadIdx.x; g < B.ng; g += BC_THREADS) {
    const uint2 t = B.gt[g];
    float x = V[t.x >> 16];
    if (B.gf) x *= B.gf[g];
    V[t.x & 0xffffu] = (t.y >> c) & 1u ? -x : x;
  }
  __syncthreads();
}

template <int G>
__device__ __forceinline__ void bc_smooth_vec(const BcLevel& B, int nsweeps) {
  const BcView& L = B.v;
  const int nh = L.cells() / 2;
  for (int h = 0; h < 2 * nsweeps; ++h) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      for (int q = threadIdx.x; q < nh; q += BC_THREADS) {
        int i, j, k;
        L.colour_cell(q, h & 1, i, j, k);
        const int p = L.idx(i, j, k);
        B.e[c][p] = vec_new_value<float, G, false>(L, B.e[0], B.e[1], B.e[2], B.f[c], c, i, j, p);
      }
      __syncthreads();
      bc_fill(B, B.e[c], c);
    }
  }
}

template <int G, bool VEC>
__device__ __forceinline__ void bc_smooth(const BcLevel& B, int nsweeps) {
  if (VEC)
    bc_smooth_vec<G>(B, nsweeps);
  else
    bc_smooth_scalar<G>(B, nsweeps);
}

// ---------------------------------------------------------- grid transfer

// Residual of level F restricted into C's right-hand side (weights and
// summation order of restrict_cell), C's correction zeroed, and with fold K
// restricted: one thread per coarse cell (and component).
template <int G, bool VEC>
__device__ __forceinline__ void bc_down(const BcLevel& F, const BcLevel& C, bool fold) {
  const BcView &L = F.v, &Lc = C.v;
  const int nC = Lc.cells(), nk = L.three ? 2 : 1;
  for (int q = threadIdx.x; q < (VEC ? 3 : 1) * nC; q += BC_THREADS) {
    const int c = VEC ? (q >= nC) + (q >= 2 * nC) : 0;
    int I, J, K;
    Lc.cell(VEC ? q - c * nC : q, I, J, K);
    float wi[2], wj[2];
    wi[0] = L.TI(TI_VW, 2 * I);
    wi[1] = L.TI(TI_VW, 2 * I + 1);
    wj[0] = L.TJ(TJ_VW, 2 * J);
    wj[1] = L.TJ(TJ_VW, 2 * J + 1);
    float wsum = 0.0f;
    for (int dk = 0; dk < nk; ++dk)
      for (int dj = 0; dj < 2; ++dj)
        for (int di = 0; di < 2; ++di) wsum += wi[di] * wj[dj];
    const float inv = 1.0f / wsum;
    float s = 0.0f, sk = 0.0f;
    for (int dk = 0; dk < nk; ++dk)
#pragma unroll(VEC ? 1 : 2)
      for (int dj = 0; dj < 2; ++dj)
#pragma unroll
        for (int di = 0; di < 2; ++di) {
          const int i = 2 * I + di, j = 2 * J + dj, k = L.three ? 2 * K + dk : 0, p = L.idx(i, j, k);
          float r;
          if (VEC) {
            r = c == 0 ? vec_residual_cell<float, G, false>(L, F.e[0], F.e[1], F.e[2], F.f[0], 0, i, j, p)
                       : (c == 1 ? vec_residual_cell<float, G, false>(L, F.e[0], F.e[1], F.e[2], F.f[1], 1, i, j, p)
                                 : vec_residual_cell<float, G, false>(L, F.e[0], F.e[1], F.e[2], F.f[2], 2, i, j, p));
          } else {
            float D;
            const float uc = F.e[0][p];
            float Lu = bc_lap<G>(L, F.e[0], p, i, j, k, uc, D);
            if (F.k) Lu -= F.k[p] * uc;
            r = F.f[0][p] - Lu;
            if (fold) sk += wi[di] * wj[dj] * F.k[p];
          }
          s += wi[di] * wj[dj] * r;
        }
    const int pc = Lc.idx(I, J, K);
    (VEC ? (c == 0 ? C.f[0] : (c == 1 ? C.f[1] : C.f[2])) : C.f[0])[pc] = s * inv;
    if (!VEC && fold) C.k[pc] = sk * inv;
  }
#pragma unroll
  for (int c = 0; c < (VEC ? 3 : 1); ++c)
    for (int q = threadIdx.x; q < Lc.ghosted(); q += BC_THREADS) C.e[c][q] = 0.0f;
  __syncthreads();
}

// Coarse scalar value at (I, J, K), outside the level in at most one
// dimension: outer ghosts are in the array, those across the origin or the
// axis are reflections (parity +1), phi wraps.
template <int G>
__device__ __forceinline__ float bc_coarse_value(const BcView& C, const float* e, int I, int J, int K) {
  if (G != CART) {
    const int ks = C.three ? (K + (C.n2 >> 1)) & (C.n2 - 1) : K;
    if (I < 0) {
      I = 0;
      if (G == SPH) J = C.n1 - 1 - J;
      K = ks;
    } else if (G == SPH && (J < 0 || J >= C.n1)) {
      J = J < 0 ? 0 : C.n1 - 1;
      K = ks;
    } else if (C.three) {
      K &= C.n2 - 1;
    }
  }
  return e[C.idx(I, J, K)];
}

// Kwak prolongation (prolong_cell) of C's correction added into F's.
template <int G, bool VEC>
__device__ __forceinline__ void bc_up(const BcLevel& F, const BcLevel& C) {
  const BcView &L = F.v, &Lc = C.v;
  const int n = L.cells();
#pragma unroll
  for (int c = 0; c < (VEC ? 3 : 1); ++c) {
    const float* ec = C.e[c];
    for (int q = threadIdx.x; q < n; q += BC_THREADS) {
      int i, j, k;
      L.cell(q, i, j, k);
      const int I = i >> 1, J = j >> 1, K = L.three ? (k >> 1) : 0;
      const int si = (i & 1) ? 1 : -1, sj = (j & 1) ? 1 : -1, sk = (k & 1) ? 1 : -1;
      const int pc = Lc.idx(I, J, K);
      float x, y, z = 0.0f;
      if (VEC) {  // every face ghost is in the array
        x = ec[pc + si];
        y = ec[pc + sj * Lc.sx];
        if (L.three) z = ec[pc + sk * Lc.sy];
      } else {
        x = bc_coarse_value<G>(Lc, ec, I + si, J, K);
        y = bc_coarse_value<G>(Lc, ec, I, J + sj, K);
        if (L.three) z = bc_coarse_value<G>(Lc, ec, I, J, K + sk);
      }
      const float e0 = ec[pc];
      const float add = L.three ? 0.25f * (e0 + x + y + z) : 0.25f * (2.0f * e0 + x + y);
      const int p = L.idx(i, j, k);
      if (VEC)
        F.e[c][p] += add;
      else
        bc_put<G>(F, p, i, j, k, F.e[0][p] + add);
    }
  }
  __syncthreads();
  if (VEC)
#pragma unroll
    for (int c = 0; c < 3; ++c) bc_fill(F, F.e[c], c);
}

// ---------------------------------------------------------- coarsest level

// Shared-memory scratch of the coarsest solves with a dense operator: one
// per translation unit, so that the instantiations of bc_coarse in one
// kernel share it.
union BcCoarseShared {
  double uq[BC_CMAT_MAX];
  double fp[BC_CINV_MAX];
};
static __shared__ BcCoarseShared bc_coarse_sh;

// coarse32: the coarsest correction equation in FP64 (right-hand side and
// c converted up, zero start), the solution rounded back into e.
// DENSE_ONLY: the hierarchy is known to carry the dense coarsest operator
// (scalar) or its inverse (vector); the sweeping fallbacks are not compiled.
template <int G, bool VEC, bool DENSE_ONLY = false>
__device__ void bc_coarse(const BlockCycle32& P, const BcLevel& B) {
  const BcView& Lv = B.v;
  constexpr int nc = VEC ? 3 : 1;
  if (!VEC && P.cA) {
    // red-black NGS sweeps with rows of the coarsest operator (its boundary
    // rules folded in): a thread per cell, the red ones in the first warp, the
    // black ones in the second, the row's face neighbours in registers.  A
    // pass is six shared loads and ~5 dependent FP64 operations (~64 cycles
    // each); summed densely by eight lanes a row it took ~1000 cycles, and the
    // solve 11.6 k.
    double* const uq = bc_coarse_sh.uq;
    const int n = P.cn, tid = threadIdx.x, g = tid & 31;
    if (tid < 64) {
      const bool on = g < n / 2;
      double a[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0}, d = 0.0, iD = 0.0, f = 0.0, u = 0.0;
      int nb[6] = {0, 0, 0, 0, 0, 0}, p = 0, r = 0, i = 0, j = 0, k = 0;
      if (on) {
        Lv.colour_cell(g, tid >> 5, i, j, k);
        r = i + Lv.n0 * (j + Lv.n1 * k);
        p = Lv.idx(i, j, k);
        const int sj = Lv.n0, sk = Lv.n0 * Lv.n1;
        auto side = [&](int m, int q) {
          nb[m] = q;
          a[m] = P.cA[(long)q * n + r];
        };
        if (i < Lv.n0 - 1) side(0, r + 1);
        if (i > 0) side(1, r - 1);
        if (j < Lv.n1 - 1) side(2, r + sj);
        if (j > 0) side(3, r - sj);
        // phi wraps; two planes are each other's neighbour once
        const bool wrap = G != CART && Lv.three && Lv.n2 > 2;
        if (k < Lv.n2 - 1)
          side(4, r + sk);
        else if (wrap)
          side(4, r - (Lv.n2 - 1) * sk);
        if (k > 0)
          side(5, r - sk);
        else if (wrap)
          side(5, r + (Lv.n2 - 1) * sk);
        f = (double)B.f[0][p];
        d = P.cA[(long)r * n + r] - (B.k ? (double)B.k[p] : 0.0);
        iD = 1.0 / d;
        uq[r] = 0.0;
      }
      auto warps = [] { asm volatile("bar.sync 1, 64;" ::: "memory"); };
      warps();
      for (int h = 0; h < 2 * P.coarse_sweeps; ++h) {
        if (on && (tid >> 5) == (h & 1)) {
          double x = fma(a[0], uq[nb[0]], fma(d, u, -f)), y = a[2] * uq[nb[2]];
          x = fma(a[1], uq[nb[1]], x);
          y = fma(a[3], uq[nb[3]], y);
          if (Lv.three) {
            x = fma(a[4], uq[nb[4]], x);
            y = fma(a[5], uq[nb[5]], y);
          }
          u = fma(-(x + y), iD, u);
          uq[r] = u;
        }
        warps();
      }
      if (on) bc_put<G>(B, p, i, j, k, (float)u);
    }
    __syncthreads();
    return;
  }
  if (VEC && P.cinv) {
    // exact solve with the precomputed inverse of the coarsest operator:
    // unknown r = c * cells + q (q the interior flat index); row r is summed
    // by the BC_SPLIT lanes of one group, each over every BC_SPLIT-th column,
    // and the partial sums folded by shuffles: the dependent FP64 chain of a
    // row is n / BC_SPLIT long instead of n
    double* const fp = bc_coarse_sh.fp;
    const int n = P.cn, cells = n / 3;
    for (int r = threadIdx.x; r < n; r += BC_THREADS) {
      const int c = (r >= cells) + (r >= 2 * cells);
      int i, j, k;
      Lv.cell(r - c * cells, i, j, k);
      fp[r] = (double)(c == 0 ? B.f[0] : (c == 1 ? B.f[1] : B.f[2]))[Lv.idx(i, j, k)];
    }
    __syncthreads();
    constexpr int BC_SPLIT = 8;
    const int sub = threadIdx.x % BC_SPLIT, rows = BC_THREADS / BC_SPLIT;
    for (int base = 0; base < n; base += rows) {  // the same trip count in every thread
      const int r = base + (int)threadIdx.x / BC_SPLIT;
      double x = 0.0;
      if (r < n)
        for (int col = sub; col < n; col += BC_SPLIT) x += P.cinv[(long)col * n + r] * fp[col];
#pragma unroll
      for (int o = BC_SPLIT / 2; o >= 1; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o, BC_SPLIT);
      if (r < n && sub == 0) {
        const int c = (r >= cells) + (r >= 2 * cells);
        int i, j, k;
        Lv.cell(r - c * cells, i, j, k);
        (c == 0 ? B.e[0] : (c == 1 ? B.e[1] : B.e[2]))[Lv.idx(i, j, k)] = (float)x;
      }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < 3; ++c) bc_fill(B, B.e[c], c);
    return;
  }
  if constexpr (!DENSE_ONLY) {
    // larger coarsest levels: stencil sweeps in FP64
    const LevelView<double>& L = P.c64;
    double* smd = reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(bc_smem()) + P.fp64_at);
    const int n = Lv.cells(), ng = Lv.ghosted();
    double* cu[3] = {smd + P.cu[0], smd + P.cu[1], smd + P.cu[2]};
    double* cf[3] = {smd + P.cf[0], smd + P.cf[1], smd + P.cf[2]};
    double* ck = P.ck >= 0 ? smd + P.ck : nullptr;
#pragma unroll
    for (int c = 0; c < nc; ++c) {
      for (int q = threadIdx.x; q < n; q += BC_THREADS) {
        int i, j, k;
        Lv.cell(q, i, j, k);
        const int p = Lv.idx(i, j, k);
        cf[c][p] = (double)B.f[c][p];
        if (!VEC && ck) ck[p] = (double)B.k[p];
      }
      for (int q = threadIdx.x; q < ng; q += BC_THREADS) cu[c][q] = 0.0;
    }
    __syncthreads();
    if (VEC)
      coarse_vec_body<double, G>(L, cu[0], cu[1], cu[2], cf[0], cf[1], cf[2], P.coarse_sweeps);
    else
      coarse_scalar_body<double, G, EQ_LIN, false>(L, cu[0], cf[0], nullptr, ck, P.coarse_sweeps);
    __syncthreads();
#pragma unroll
    for (int c = 0; c < nc; ++c)
      for (int q = threadIdx.x; q < n; q += BC_THREADS) {
        int i, j, k;
        Lv.cell(q, i, j, k);
        const int p = Lv.idx(i, j, k);
        if (VEC)
          B.e[c][p] = (float)cu[c][p];
        else
          bc_put<G>(B, p, i, j, k, (float)cu[0][p]);
      }
    __syncthreads();
    if (VEC)
#pragma unroll
      for (int c = 0; c < 3; ++c) bc_fill(B, B.e[c], c);
  }
}

// The cycle from level from of P down and back, its right-hand side and zero
// correction in shared memory.
template <int G, bool VEC, bool DENSE_ONLY = false>
__device__ __forceinline__ void bc_levels(const BlockCycle32& P, int from) {
  // down: pre-smooth, residual restricted into the next level's right-hand
  // side, zero correction there
  for (int l = from; l + 1 < P.nl; ++l) {
    const BcLevel F = bc_level<VEC>(P, l);
    bc_smooth<G, VEC>(F, P.nu1);
    bc_down<G, VEC>(F, bc_level<VEC>(P, l + 1), P.fold_k);
  }
  bc_coarse<G, VEC, DENSE_ONLY>(P, bc_level<VEC>(P, P.nl - 1));
  // up: Kwak prolongation of the correction, post-smooth
  for (int l = P.nl - 2; l >= from; --l) {
    const BcLevel F = bc_level<VEC>(P, l);
    bc_up<G, VEC>(F, bc_level<VEC>(P, l + 1));
    bc_smooth<G, VEC>(F, P.nu2);
  }
}

// The whole cycle from level l0 of P: its right-hand side in from P.f_in,
// the correction out to P.e_out (ghosts included).  No barrier after the
// final stores.  DENSE_ONLY: P carries the dense coarsest operator (cA) or
// its inverse (cinv).  problem_at: offset of the block's problem in them.
// TABLES: the coefficient tables are on their way to
// shared memory already (bc_stage_tables).
template <int G, bool VEC, bool DENSE_ONLY = false, bool TABLES = false>
__device__ void bc_run(const BlockCycle32& P, long problem_at = 0) {
  constexpr int nc = VEC ? 3 : 1;
  if (!TABLES) bc_stage_tables(P);
  {
    // level l0: right-hand side and K in (K of the deeper levels too, unless
    // it is restricted on the way down), zero correction
    const BcLevel B = bc_level<VEC>(P, 0);
#pragma unroll
    for (int c = 0; c < nc; ++c) {
      for (int q = threadIdx.x; q < (int)P.ng0 / 4; q += BC_THREADS) bc_cp16(B.f[c] + 4 * q, P.f_in[c] + problem_at + 4 * q);
      for (int q = threadIdx.x; q < (int)P.ng0; q += BC_THREADS) B.e[c][q] = 0.0f;
    }
    if (!VEC) bc_stage_k(P, 0, P.fold_k ? 1 : BC_MAX);
    bc_rules<G, VEC>(P);
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    __syncthreads();
  }
  bc_levels<G, VEC, DENSE_ONLY>(P, 0);
  // level l0 correction out (ghosts included)
  const BcLevel B = bc_level<VEC>(P, 0);
#pragma unroll
  for (int c = 0; c < nc; ++c)
    for (int q = threadIdx.x; q < (int)P.ng0 / 4; q += BC_THREADS)
      reinterpret_cast<float4*>(P.e_out[c] + problem_at)[q] = reinterpret_cast<const float4*>(B.e[c])[q];
}

}  // namespace gmg
