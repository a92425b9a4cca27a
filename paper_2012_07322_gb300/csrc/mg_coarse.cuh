// The FP64 coarsest-grid solves of the FAS cycle (Newton-Gauss-Seidel sweeps
// until the residual has dropped 1e-12 x, at most max_sweeps; Sec. 2.7.2) on
// coarsest levels of a few dozen cells.
//
// What bounds them is the length of dependent FP64 chains on one SM: a
// dependent FP64 operation takes ~64 cycles here, a division ~430, and a
// sweep with its residual maximum is a chain of colour passes.  The general
// bodies (coarse_scalar_body, coarse_vec_body) re-evaluate the boundary
// rules and metric factors in every pass and end every sweep with a block
// reduction: 93 us per call for eq. psi on 4 x 2 cells, 104 us on 4 x 2 x 2,
// 455 us for the vector equation on 4 x 2 x 2 (64 x 32 x 32 hierarchy).
#pragma once
#include "mg_internal.h"
#include "mg_kernels.cuh"

namespace gmg {

constexpr int CS_MAX = CS_CELLS;  // cells of a scalar coarsest level: at most one warp of each colour
constexpr int CV_THREADS = 256;

union CoarseShared {
  struct {
    double u[2][CS_MAX];
    unsigned long long r[2];
  } scalar;
  struct {
    double x[CV_N + 1], r[CV_N];
  } vec;
};

// ------------------------------------------------------ scalar equations

// A cell of the coarsest level with its boundary rules resolved: the stencil
// neighbours as compact cell numbers (b < 0: a ghost, g times the cell's own
// value) and the coefficients of lap_scalar.
template <int G>
struct CoarseCell {
  int q;          // compact cell number, < 0: none
  int b[6];       // east, west, north, south, up, down
  double g[6];
  double cE, cW, cN, cS, cC, cZ, D;
  double f, s0, s1;
};

template <int G>
__device__ __forceinline__ void coarse_cell_load(CoarseCell<G>& c, const LevelView<double>& L,
                                                 const double* __restrict__ f, const double* __restrict__ s0,
                                                 const double* __restrict__ s1, int i, int j, int k) {
  const int n0 = L.n0, n1 = L.n1, n2 = L.n2;
  c.q = i + n0 * (j + n1 * k);
  auto at = [&](int a, int b, int d) { return a + n0 * (b + n1 * d); };
#pragma unroll
  for (int m = 0; m < 6; ++m) {
    c.b[m] = -1;
    c.g[m] = 1.0;
  }
  if (i < n0 - 1)
    c.b[0] = at(i + 1, j, k);
  else
    c.g[0] = outer_factor(L, n0, j, k, n0 - 1, j, k);
  if (i > 0)
    c.b[1] = at(i - 1, j, k);
  else if (G == CART)
    c.g[1] = outer_factor(L, -1, j, k, 0, j, k);
  if (j < n1 - 1)
    c.b[2] = at(i, j + 1, k);
  else if (G != SPH)
    c.g[2] = outer_factor(L, i, n1, k, i, n1 - 1, k);
  if (j > 0)
    c.b[3] = at(i, j - 1, k);
  else if (G != SPH)
    c.g[3] = outer_factor(L, i, -1, k, i, 0, k);
  if (L.three) {
    if (G == CART) {
      if (k < n2 - 1)
        c.b[4] = at(i, j, k + 1);
      else
        c.g[4] = outer_factor(L, i, j, n2, i, j, n2 - 1);
      if (k > 0)
        c.b[5] = at(i, j, k - 1);
      else
        c.g[5] = outer_factor(L, i, j, -1, i, j, 0);
    } else {
      c.b[4] = at(i, j, k < n2 - 1 ? k + 1 : 0);
      c.b[5] = at(i, j, k > 0 ? k - 1 : n2 - 1);
    }
  }
  c.cE = L.TI(TI_CE, i);
  c.cW = L.TI(TI_CW, i);
  c.D = -(c.cE + c.cW);
  c.cC = 0.0;
  if (G == SPH) {
    c.cC = L.TI(TI_IX2, i);
    c.cN = L.TJ(TJ_TN, j);
    c.cS = L.TJ(TJ_TS, j);
    c.D -= c.cC * (c.cN + c.cS);
  } else {
    c.cN = c.cS = L.ih1s;
    c.D -= 2.0 * L.ih1s;
  }
  c.cZ = 0.0;
  if (L.three) {
    c.cZ = G == CART ? L.ih2s : (G == CYL ? L.TI(TI_PHI, i) : L.TI(TI_IX2, i) * L.TJ(TJ_PF, j));
    c.D -= 2.0 * c.cZ;
  }
  const long p = L.idx(i, j, k);
  c.f = f ? f[p] : 0.0;
  c.s0 = s0 ? s0[p] : 0.0;
  c.s1 = s1 ? s1[p] : 0.0;
}

// lap_scalar at a cell: own value uc, neighbours from u.
template <int G>
__device__ __forceinline__ double coarse_lap(const CoarseCell<G>& c, const double* u, double uc, bool three) {
  double nb[6];
#pragma unroll
  for (int m = 0; m < 6; ++m) nb[m] = c.b[m] >= 0 ? u[c.b[m]] : c.g[m] * uc;
  double Lu = c.cE * (nb[0] - uc) - c.cW * (uc - nb[1]);
  if (G == SPH)
    Lu += c.cC * (c.cN * (nb[2] - uc) - c.cS * (uc - nb[3]));
  else
    Lu += c.cN * (nb[2] - 2.0 * uc + nb[3]);
  if (three) Lu += c.cZ * (nb[4] - 2.0 * uc + nb[5]);
  return Lu;
}

// One Newton-Gauss-Seidel value (scalar_update; linear equations with the
// inverted diagonal, scalar_update_lin_inv).
template <int G, int KIND>
__device__ __forceinline__ double coarse_new(const CoarseCell<G>& c, const double* u, double uc, double invD,
                                             bool three) {
  const double lap = coarse_lap<G>(c, u, uc, three);
  if (KIND == EQ_PSI) {
    const double q = 1.0 + uc, q2 = q * q, q4 = q2 * q2, q6 = q4 * q2, q8 = q4 * q4;
    const double a = (2 * PI_D) * c.s0, b = c.s1;
    const double num = (lap - c.f) * q8 + a * q6 * q + 0.125 * b * q;
    const double den = c.D * q8 - a * q6 - 0.875 * b;
    return uc - num / den;
  }
  return uc - (lap - c.s1 * uc - c.f) * invD;
}

// |f - L(u)| of a cell as ordered bits (scalar_op).
template <int G, int KIND>
__device__ __forceinline__ unsigned long long coarse_res(const CoarseCell<G>& c, const double* u, bool three) {
  if (c.q < 0) return 0ULL;
  const double uc = u[c.q];
  double Lu = coarse_lap<G>(c, u, uc, three);
  if (KIND == EQ_PSI) {
    const double ip = 1.0 / (1.0 + uc), ip2 = ip * ip, ip4 = ip2 * ip2, ip7 = ip4 * ip2 * ip;
    Lu += (2 * PI_D) * c.s0 * ip + 0.125 * c.s1 * ip7;
  } else {
    Lu -= c.s1 * uc;
  }
  return abs_bits(c.f - Lu);
}

// Two warps: warp 0 sweeps, a lane holding one red and one black cell with
// everything but u in registers; warp 1 evaluates the residual maximum of
// the state before that sweep, so the stopping rule costs no time of its own
// (a sweep started before the rule is known is dropped: the state before it
// is in the other buffer).  Same sweeps and same stopping rule as
// coarse_scalar_body.  Eq. psi on 4 x 2 cells: 93 -> 26 us.
// Called by the first two warps of a block; no barrier after the stores.
template <int G, int KIND>
__device__ __forceinline__ void coarse_scalar_small(CoarseShared& sh, const LevelView<double>& L, double* u,
                                                    const double* f, const double* s0, const double* s1,
                                                    int max_sweeps) {
  if (threadIdx.x >= 64) return;
  auto& su = sh.scalar.u;
  auto& rs = sh.scalar.r;
  auto sync = [] { asm volatile("bar.sync 1, 64;" ::: "memory"); };  // the two warps
  const int n = L.n0 * L.n1 * L.n2, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool three = L.three;
  for (int q = threadIdx.x; q < n; q += 64) su[0][q] = u[interior_p(L, q)];
  // warp 0: the lane-th cell of each colour; warp 1: cells lane and lane + 32
  CoarseCell<G> c[2];
  double invD[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int r = warp ? lane + 32 * h : lane;
    c[h].q = -1;
    if (r >= (warp ? n : n / 2)) continue;
    int i, j, k;
    if (warp)
      L.cell(r, i, j, k);
    else
      L.colour_cell(r, h, i, j, k);
    coarse_cell_load<G>(c[h], L, f, s0, s1, i, j, k);
    invD[h] = KIND == EQ_LIN ? 1.0 / (c[h].D - c[h].s1) : 0.0;
  }
  sync();
  double r0 = 0.0;
  int it = 0;
  for (; it < max_sweeps; ++it) {
    const double* a = su[it & 1];
    double* b = su[(it & 1) ^ 1];
    if (warp == 0) {
      if (c[0].q >= 0) b[c[0].q] = coarse_new<G, KIND>(c[0], a, a[c[0].q], invD[0], three);
      __syncwarp();
      if (c[1].q >= 0) b[c[1].q] = coarse_new<G, KIND>(c[1], b, a[c[1].q], invD[1], three);
    } else {
      const unsigned long long m =
          warp_max_bits(umax64(coarse_res<G, KIND>(c[0], a, three), coarse_res<G, KIND>(c[1], a, three)));
      if (lane == 0) rs[it & 1] = m;
    }
    sync();
    // the residual before sweep it (after it sweeps)
    const double r = __longlong_as_double((long long)rs[it & 1]);
    if (it == 0) {
      r0 = r;
      if (!(r0 > 0.0)) return;  // u is the solution already
    } else if (!(r > 1e-12 * r0)) {
      break;
    }
  }
  for (int q = threadIdx.x; q < n; q += 64) u[interior_p(L, q)] = su[it & 1][q];
}

// ------------------------------------------------------ vector equations

// Row r of the operator applied to x, by the CV_LANES lanes of a group: entry
// m adds cf (x[a] - x[b]), b the row's own cell in a's component (or the zero
// behind x, for the operator's action on constants), so that, as in the flux
// form, smooth fields are subtracted before they are multiplied.
constexpr int CV_LANES = 4, CV_PER_LANE = 8;

__device__ __forceinline__ double sparse_row(const CoarseRows& R, const double* x, int r, int sub, bool on) {
  double s0 = 0.0, s1 = 0.0;
  if (on) {
#pragma unroll
    for (int m = 0; m < CV_PER_LANE; ++m) {
      const int e = sub + CV_LANES * m;
      if (e < R.width) {
        const unsigned ab = R.ab[e * R.n + r];
        const double t = x[ab & 0xffffu] - x[ab >> 16], cf = R.cf[e * R.n + r];
        if (m & 1)
          s1 += cf * t;
        else
          s0 += cf * t;
      }
    }
  }
  double s = s0 + s1;
#pragma unroll
  for (int o = CV_LANES >> 1; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, 32);
  return s;
}

// The coarsest vector solve.  The sweeps of a linear equation are one affine
// map of the state: u + S (f - A u), S the sum of the sweeps' response to a
// residual, which the host tabulates by sweeping the rows on unit residuals
// (CoarseRows).  What is left is one residual and one product with S, two
// short FP64 chains in place of max_sweeps x 6 dependent passes: 158 us per
// solve of 4 x 2 x 2 cells from dense rows, 106 us swept from the nonzeros.
// The sweeps' early stop (residual down 1e-12 x) has no counterpart: past it
// a sweep moves u by less than that.  Called by a block of CV_THREADS threads.
template <int G>
__device__ __forceinline__ void coarse_vec_rows(CoarseShared& sh, const LevelView<double>& L, double* U, double* V,
                                                double* W, const double* f0, const double* f1, const double* f2,
                                                const CoarseRows& R) {
  auto& x = sh.vec.x;
  auto& res = sh.vec.r;
  const int n = R.n, cells = n / 3, tid = threadIdx.x, t = tid / CV_LANES, sub = tid % CV_LANES;
  constexpr int rows = CV_THREADS / CV_LANES;
  for (int r = tid; r < n; r += CV_THREADS) {
    const int c = (r >= cells) + (r >= 2 * cells);
    const long p = interior_p(L, r - c * cells);
    const double* f = c == 0 ? f0 : (c == 1 ? f1 : f2);
    x[r] = (c == 0 ? U : (c == 1 ? V : W))[p];
    res[r] = f ? f[p] : 0.0;
  }
  if (tid == 0) x[n] = 0.0;
  __syncthreads();
  for (int base = 0; base < n; base += rows) {
    const int r = base + t;
    const double Lu = sparse_row(R, x, r, sub, r < n);
    if (r < n && sub == 0) res[r] -= Lu;
  }
  __syncthreads();
  for (int base = 0; base < n; base += rows) {
    const int r = base + t;
    double s0 = 0.0, s1 = 0.0;
    if (r < n) {
      const double* __restrict__ S = R.S + r;
      for (int q = sub; q < n; q += 2 * CV_LANES) {
        s0 += S[(long)q * n] * res[q];
        if (q + CV_LANES < n) s1 += S[(long)(q + CV_LANES) * n] * res[q + CV_LANES];
      }
    }
    double s = s0 + s1;
#pragma unroll
    for (int o = CV_LANES >> 1; o >= 1; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o, 32);
    if (r < n && sub == 0) {
      const int c = (r >= cells) + (r >= 2 * cells);
      (c == 0 ? U : (c == 1 ? V : W))[interior_p(L, r - c * cells)] = x[r] + s;
    }
  }
  __syncthreads();
  const long ngh = ghost_count(L);
  for (long gq = tid; gq < 3 * ngh; gq += CV_THREADS) {
    const int c = (gq >= ngh) + (gq >= 2 * ngh);
    fill_one_ghost(L, c == 0 ? U : (c == 1 ? V : W), c, gq - c * ngh);
  }
}

}  // namespace gmg
