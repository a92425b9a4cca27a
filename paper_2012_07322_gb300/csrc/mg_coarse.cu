// The FP64 coarsest-grid solves of mg_coarse.cuh as kernels, and the matrix
// the rows of the vector solve come from.
#include "mg_coarse.cuh"

namespace gmg {

template <int G, int KIND>
__global__ void __launch_bounds__(64)
    k_coarse_scalar_small(LevelView<double> L, double* u, const double* f, const double* s0, const double* s1,
                          int max_sweeps) {
  pdl_entry();
  __shared__ CoarseShared sh;
  coarse_scalar_small<G, KIND>(sh, L, u, f, s0, s1, max_sweeps);
}

template <int G>
static void launch_small(const LevelView<double>& L, int kind, double* u, const double* f, const double* s0,
                         const double* s1, int max_sweeps, cudaStream_t st) {
  if (kind == EQ_PSI)
    launch_k(k_coarse_scalar_small<G, EQ_PSI>, 1, 64, 0, st, L, u, f, s0, s1, max_sweeps);
  else
    launch_k(k_coarse_scalar_small<G, EQ_LIN>, 1, 64, 0, st, L, u, f, s0, s1, max_sweeps);
}

bool launch_coarse_scalar_small(const LevelView<double>& L, int kind, double* u, const double* f, const double* s0,
                                const double* s1, int max_sweeps, cudaStream_t st) {
  if ((long)L.n0 * L.n1 * L.n2 > CS_MAX) return false;
  count_launch();
  if (L.geom == CART)
    launch_small<CART>(L, kind, u, f, s0, s1, max_sweeps, st);
  else if (L.geom == CYL)
    launch_small<CYL>(L, kind, u, f, s0, s1, max_sweeps, st);
  else
    launch_small<SPH>(L, kind, u, f, s0, s1, max_sweeps, st);
  return true;
}

// The coarsest vector operator as a matrix, from which the host takes the rows
// of coarse_vec_rows: column col <
// n of A (A[col * n + r]) is the operator (its ghost rules folded in) applied
// to the unit field of unknown col = comp * cells + q; columns n .. n + 2
// are the operator applied to the constant fields of each component; D[r]
// is the Newton diagonal (ghosts held fixed), inverted.
template <int G>
__global__ void k_coarse_rows_vec(LevelView<double> L, double* __restrict__ scratch, double* __restrict__ A,
                                  double* __restrict__ invD, int n) {
  pdl_entry();
  const int col = blockIdx.x, cells = n / 3;
  const long ng = L.sy * (L.n2 + 2 * L.three);
  double* U[3];
  for (int c = 0; c < 3; ++c) U[c] = scratch + ((long)col * 3 + c) * ng;
  for (long q = threadIdx.x; q < 3 * ng; q += blockDim.x) U[0][q] = 0.0;
  __syncthreads();
  if (col >= n) {
    for (int q = threadIdx.x; q < cells; q += blockDim.x) U[col - n][interior_p(L, q)] = 1.0;
  } else if (threadIdx.x == 0) {
    U[col / cells][interior_p(L, col % cells)] = 1.0;
  }
  __syncthreads();
  const long ngh = ghost_count(L);
  for (int c = 0; c < 3; ++c)
    for (long g = threadIdx.x; g < ngh; g += blockDim.x) fill_one_ghost(L, U[c], c, g);
  __syncthreads();
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    int i, j, k;
    L.cell(r % cells, i, j, k);
    double D;
    A[(long)col * n + r] = vec_op<double, G>(L, U[0], U[1], U[2], r / cells, i, j, L.idx(i, j, k), D);
    if (col == 0) invD[r] = 1.0 / D;
  }
}

template <int G>
__global__ void __launch_bounds__(CV_THREADS)
    k_coarse_vec_rows(LevelView<double> L, double* U, double* V, double* W, const double* f0, const double* f1,
                      const double* f2, const __grid_constant__ CoarseRows R) {
  pdl_entry();
  __shared__ CoarseShared sh;
  coarse_vec_rows<G>(sh, L, U, V, W, f0, f1, f2, R);
}

void launch_coarse_rows_vec(const LevelView<double>& L, double* scratch, double* A, double* invD, int n,
                            cudaStream_t st) {
  count_launch();
  if (L.geom == CART)
    launch_k(k_coarse_rows_vec<CART>, n + 3, 256, 0, st, L, scratch, A, invD, n);
  else if (L.geom == CYL)
    launch_k(k_coarse_rows_vec<CYL>, n + 3, 256, 0, st, L, scratch, A, invD, n);
  else
    launch_k(k_coarse_rows_vec<SPH>, n + 3, 256, 0, st, L, scratch, A, invD, n);
}

void launch_coarse_vec_rows(const LevelView<double>& L, double* const V[3], const double* const f[3],
                            const CoarseRows& R, cudaStream_t st) {
  count_launch();
  if (L.geom == CART)
    launch_k(k_coarse_vec_rows<CART>, 1, CV_THREADS, 0, st, L, V[0], V[1], V[2], f[0], f[1], f[2], R);
  else if (L.geom == CYL)
    launch_k(k_coarse_vec_rows<CYL>, 1, CV_THREADS, 0, st, L, V[0], V[1], V[2], f[0], f[1], f[2], R);
  else
    launch_k(k_coarse_vec_rows<SPH>, 1, CV_THREADS, 0, st, L, V[0], V[1], V[2], f[0], f[1], f[2], R);
}

}  // namespace gmg
