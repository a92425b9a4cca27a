// Streaming kernels of 3D Cartesian levels with a linear scalar equation
// without c (the Poisson problem of divergence cleaning): the FP64 residual
// on the integer units, and the FP32 residual-restriction and prolongation
// with one thread per coarse cell.
#include "mg_cart.cuh"
#include "mg_internal.h"
#include "mg_kernels.cuh"

namespace gmg {

// ------------------------------------------------------- FP64 residual

// r = f - lap u of every cell of a level with equal spacings (r, r32
// nullable), and the norms of the stopping rule into red (nullable; weighted
// != 0 also the source norm).  A thread marches KZ planes of its column, its
// decoded values of three planes in registers.  The FP64 pipe (2 operations
// per SM and clock) bounds the flux form (557 us at 256^3, 12 operations per
// cell); here a cell costs it three (conversion of the sum, one FMA, the
// rounding to FP32) and the integer units ~110 instructions.
template <int KZ>
__global__ void __launch_bounds__(256, 4)
    k_resid_cart(LevelView<double> L, const double* __restrict__ u, const double* __restrict__ f,
                 double* __restrict__ r, float* __restrict__ r32, unsigned long long* red, int weighted) {
  pdl_entry();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const int j = blockIdx.y * blockDim.y + threadIdx.y;
  int b;
  const int k0 = (L.z_block(b) * blockDim.z + threadIdx.z) * KZ;
  u += b * L.bst;
  if (f) f += b * L.bst;
  if (r) r += b * L.bst;
  if (r32) r32 += b * L.bst;
  if (red) red += 3 * b;
  const long sx = L.sx, sy = L.sy;
  const bool neumann = L.bc == BC_NEUMANN;
  const bool edge_ij = i == 0 || i == L.n0 - 1 || j == 0 || j == L.n1 - 1;
  unsigned long long m0 = 0ULL, m2 = 0ULL;
  long p = L.idx(i, j, k0);
  double uc = u[p];
  Fixed c = fix_decode(uc), dn = k0 > 0 ? fix_decode(u[p - sy]) : c;
#pragma unroll 1
  for (int t = 0; t < KZ; ++t, p += sy) {
    const int k = k0 + t;
    const double un = k < L.n2 - 1 ? u[p + sy] : uc;
    const Fixed up = fix_decode(un);
    double res;
    const double fv = f ? f[p] : 0.0;
    bool done = false;
    if (neumann || !(edge_ij || k == 0 || k == L.n2 - 1)) {
      // a Neumann ghost is the cell's own value: it drops out of the sum
      const Fixed e = fix_decode(u[i < L.n0 - 1 ? p + 1 : p]), w = fix_decode(u[i > 0 ? p - 1 : p]);
      const Fixed n = fix_decode(u[j < L.n1 - 1 ? p + sx : p]), s = fix_decode(u[j > 0 ? p - sx : p]);
      done = fix_residual(c, e, w, n, s, up, dn, L.ih0s, fv, res);
    }
    if (!done) {
      double D;
      res = fv - lap_scalar<double, CART>(L, u, i, j, k, p, D);
    }
    if (r) r[p] = res;
    if (r32) r32[p] = (float)res;
    m0 = umax64(m0, abs_bits(res));
    if (weighted) m2 = umax64(m2, abs_bits(fv));
    dn = c;
    c = up;
    uc = un;
  }
  if (red) {
    unsigned long long m[3] = {m0, weighted ? m0 : 0ULL, m2};
    block_max_bits<3>(m, red);
  }
}

bool resid_cart_applies(const LevelView<double>& L) {
  return L.geom == CART && L.three && L.ih0s == L.ih1s && L.ih1s == L.ih2s && L.n0 >= 32 && L.n1 >= 8 && L.n2 >= 8;
}

void launch_resid_cart(const LevelView<double>& L, const double* u, const double* f, double* r,
                       unsigned long long* red, int weighted, cudaStream_t st, float* r32) {
  count_launch();
  // long marches reuse the column's decoded planes; levels too small to fill
  // the device that way take two planes per thread
  const bool big = (long)L.n0 * L.n1 * L.n2 >= (1L << 21);
  const dim3 b(32, 8, 1);
  const dim3 g(L.n0 / 32, L.n1 / 8, L.nb * (L.n2 / (big ? 8 : 2)));
  if (big)
    launch_k(k_resid_cart<8>, g, b, 0, st, L, u, f, r, r32, red, weighted);
  else
    launch_k(k_resid_cart<2>, g, b, 0, st, L, u, f, r, r32, red, weighted);
}

// ----------------------------------------------- FP32 residual-restriction

// f - lap e of the eight fine cells of a coarse cell, averaged into fc (the
// arithmetic and the summation order of k_resid_restrict32, whose weights are
// one here); the coarse correction ec zeroed, ghosts included.  A thread owns
// a coarse column and marches KC coarse planes: a fine plane costs it eight
// loads for four cells (k_resid_restrict32: eight per cell), and the planes
// above and below stay in registers.  256^3: 125 us before (cold).
template <int KC>
__global__ void __launch_bounds__(256)
    k_resid_restrict_cart(LevelView<float> F, LevelView<float> C, const float* __restrict__ e,
                          const float* __restrict__ f, float* __restrict__ fc, float* __restrict__ ec) {
  pdl_entry();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  int bq;
  const int K0 = (F.z_block(bq) * blockDim.z + threadIdx.z) * KC;
  e += bq * F.bst;
  f += bq * F.bst;
  fc += bq * C.bst;
  const int i = 2 * I, j = 2 * J;
  const long sx = F.sx, sy = F.sy;
  const bool ie = i + 2 == F.n0, iw = i == 0, jn = j + 2 == F.n1, js = j == 0;
  const float cE = F.TI(TI_CE, i), cY = F.ih1s, cZ = F.ih2s;
  struct Plane {
    float2 a, b;  // rows j and j + 1
  };
  auto load = [&](long p) {
    Plane P;
    P.a = *reinterpret_cast<const float2*>(e + p);
    P.b = *reinterpret_cast<const float2*>(e + p + sx);
    return P;
  };
  // outer ghost of a boundary cell: factor times its value
  auto scale = [](Plane P, float fa, float fb, float fc2, float fd) {
    P.a.x *= fa, P.a.y *= fb, P.b.x *= fc2, P.b.y *= fd;
    return P;
  };
  auto ghost_plane = [&](const Plane& P, int kg, int ks) {
    return scale(P, outer_factor(F, i, j, kg, i, j, ks), outer_factor(F, i + 1, j, kg, i + 1, j, ks),
                 outer_factor(F, i, j + 1, kg, i, j + 1, ks), outer_factor(F, i + 1, j + 1, kg, i + 1, j + 1, ks));
  };
  long p = F.idx(i, j, 2 * K0);
  Plane c = load(p);
  Plane d = K0 > 0 ? load(p - sy) : ghost_plane(c, -1, 0);
#pragma unroll
  for (int t = 0; t < KC; ++t) {
    const int K = K0 + t;
    float s = 0.0f;
#pragma unroll
    for (int h = 0; h < 2; ++h, p += sy) {
      const int k = 2 * K + h;
      const Plane u = k < F.n2 - 1 ? load(p + sy) : ghost_plane(c, F.n2, F.n2 - 1);
      // neighbours in i of the pairs, in j of the rows
      const float wa = iw ? outer_factor(F, -1, j, k, 0, j, k) * c.a.x : e[p - 1];
      const float wb = iw ? outer_factor(F, -1, j + 1, k, 0, j + 1, k) * c.b.x : e[p + sx - 1];
      const float ea = ie ? outer_factor(F, F.n0, j, k, F.n0 - 1, j, k) * c.a.y : e[p + 2];
      const float eb = ie ? outer_factor(F, F.n0, j + 1, k, F.n0 - 1, j + 1, k) * c.b.y : e[p + sx + 2];
      float2 sa, nb;
      if (js)
        sa = make_float2(outer_factor(F, i, -1, k, i, 0, k) * c.a.x, outer_factor(F, i + 1, -1, k, i + 1, 0, k) * c.a.y);
      else
        sa = *reinterpret_cast<const float2*>(e + p - sx);
      if (jn)
        nb = make_float2(outer_factor(F, i, F.n1, k, i, F.n1 - 1, k) * c.b.x,
                         outer_factor(F, i + 1, F.n1, k, i + 1, F.n1 - 1, k) * c.b.y);
      else
        nb = *reinterpret_cast<const float2*>(e + p + 2 * sx);
      const float2 fa = *reinterpret_cast<const float2*>(f + p), fb = *reinterpret_cast<const float2*>(f + p + sx);
      auto res = [&](float uc, float ue, float uw, float un, float us, float uu, float ud, float fv) {
        float Lu = cE * (ue - uc) - cE * (uc - uw);
        Lu += cY * (un - 2.0f * uc + us);
        Lu += cZ * (uu - 2.0f * uc + ud);
        return fv - Lu;
      };
      s += res(c.a.x, c.a.y, wa, c.b.x, sa.x, u.a.x, d.a.x, fa.x);
      s += res(c.a.y, ea, c.a.x, c.b.y, sa.y, u.a.y, d.a.y, fa.y);
      s += res(c.b.x, c.b.y, wb, nb.x, c.a.x, u.b.x, d.b.x, fb.x);
      s += res(c.b.y, eb, c.b.x, nb.y, c.a.y, u.b.y, d.b.y, fb.y);
      d = c;
      c = u;
    }
    fc[C.idx(I, J, K)] = s * 0.125f;
  }
  const long nz = C.nb * (C.sy * (C.n2 + 2) / 4);
  const long nb = (long)blockDim.x * blockDim.y * blockDim.z;
  const long gt = threadIdx.x + (long)blockDim.x * (threadIdx.y + blockDim.y * threadIdx.z) +
                  nb * (blockIdx.x + gridDim.x * (blockIdx.y + (long)gridDim.y * blockIdx.z));
  const long gs = nb * gridDim.x * gridDim.y * gridDim.z;
  for (long q = gt; q < nz; q += gs) reinterpret_cast<float4*>(ec)[q] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
}

// ------------------------------------------------------------- prolongation

// Kwak prolongation (prolong_cell) of e = uH - uhH (uhH nullable) into the eight fine cells of a coarse
// cell: seven coarse loads and four 8-byte updates per thread, instead of
// four coarse loads and a 4-byte update per fine cell.  256^3: 105 us before (cold).
template <typename T, typename T2>
__global__ void __launch_bounds__(256)
    k_prolong_cart(LevelView<T> F, LevelView<T> C, T* __restrict__ u, const T* __restrict__ uH,
                   const T* __restrict__ uhH) {
  pdl_entry();
  const int I = blockIdx.x * blockDim.x + threadIdx.x, J = blockIdx.y * blockDim.y + threadIdx.y;
  int b;
  const int K = F.z_block(b) * blockDim.z + threadIdx.z;
  u += b * F.bst;
  uH += b * C.bst;
  if (uhH) uhH += b * C.bst;
  const long q = C.idx(I, J, K);
  auto e = [&](long p) { return uhH ? uH[p] - uhH[p] : uH[p]; };
  const T ec = e(q);
  T x[2], y[2], z[2];
  x[0] = I > 0 ? e(q - 1) : outer_factor(C, -1, J, K, 0, J, K) * ec;
  x[1] = I < C.n0 - 1 ? e(q + 1) : outer_factor(C, C.n0, J, K, C.n0 - 1, J, K) * ec;
  y[0] = J > 0 ? e(q - C.sx) : outer_factor(C, I, -1, K, I, 0, K) * ec;
  y[1] = J < C.n1 - 1 ? e(q + C.sx) : outer_factor(C, I, C.n1, K, I, C.n1 - 1, K) * ec;
  z[0] = K > 0 ? e(q - C.sy) : outer_factor(C, I, J, -1, I, J, 0) * ec;
  z[1] = K < C.n2 - 1 ? e(q + C.sy) : outer_factor(C, I, J, C.n2, I, J, C.n2 - 1) * ec;
  T* o = u + F.idx(2 * I, 2 * J, 2 * K);
  T2 v[4];
#pragma unroll
  for (int m = 0; m < 4; ++m) v[m] = *reinterpret_cast<const T2*>(o + (m & 1) * F.sx + (m >> 1) * F.sy);
#pragma unroll
  for (int m = 0; m < 4; ++m) {
    v[m].x += T(0.25) * (ec + x[0] + y[m & 1] + z[m >> 1]);
    v[m].y += T(0.25) * (ec + x[1] + y[m & 1] + z[m >> 1]);
    *reinterpret_cast<T2*>(o + (m & 1) * F.sx + (m >> 1) * F.sy) = v[m];
  }
}

// Levels from which a thread per coarse cell fills the device (below, the
// kernels with a thread per fine cell have eight times the parallelism).
template <typename T>
bool transfer_cart_applies(const LevelView<T>& F) {
  return F.geom == CART && F.three && F.n0 >= 64 && F.n1 >= 16 && F.n2 >= 16 &&
         (long)F.n0 * F.n1 * F.n2 >= (1L << 18);
}

void launch_resid_restrict_cart(const LevelView<float>& F, const LevelView<float>& C, const float* e, const float* f,
                                float* fc, float* ec, cudaStream_t st) {
  count_launch();
  const dim3 b(32, 8, 1);
  if ((long)F.n0 * F.n1 * F.n2 >= (1L << 23))
    launch_k(k_resid_restrict_cart<4>, dim3(C.n0 / 32, C.n1 / 8, C.nb * (C.n2 / 4)), b, 0, st, F, C, e, f, fc, ec);
  else
    launch_k(k_resid_restrict_cart<1>, dim3(C.n0 / 32, C.n1 / 8, C.nb * C.n2), b, 0, st, F, C, e, f, fc, ec);
}

void launch_prolong_cart(const LevelView<float>& F, const LevelView<float>& C, float* u, const float* uH,
                         const float* uhH, cudaStream_t st) {
  count_launch();
  launch_k(k_prolong_cart<float, float2>, dim3(C.n0 / 32, C.n1 / 8, C.nb * C.n2), dim3(32, 8, 1), 0, st, F, C, u, uH, uhH);
}
void launch_prolong_cart(const LevelView<double>& F, const LevelView<double>& C, double* u, const double* uH,
                         const double* uhH, cudaStream_t st) {
  count_launch();
  launch_k(k_prolong_cart<double, double2>, dim3(C.n0 / 32, C.n1 / 8, C.nb * C.n2), dim3(32, 8, 1), 0, st, F, C, u, uH, uhH);
}
template bool transfer_cart_applies<float>(const LevelView<float>&);
template bool transfer_cart_applies<double>(const LevelView<double>&);

}  // namespace gmg
