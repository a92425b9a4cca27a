// The FP64 FAS V-cycle of a scalar equation (Sec. 2.7) from a level of a few thousand cells down,
// in one launch of a thread-block cluster.
//
// On such levels a launched pass is a dependent chain of its launch (~1.2
// us), one L2 round trip and an FP64 chain of ~1500 cycles (a dependent FP64
// operation takes ~64 cycles, a division ~430): 3.3 us in the captured cycle,
// whatever the level's size, 12 of them per level and cycle.  A cluster
// rather than one block because the FP64 pipe takes ~16 cycles per warp
// instruction: 1024 cells of one colour are 23 k cycles on one SM and 1.4 k
// on sixteen.
//
// A thread owns one cell of every level, with its stencil, sources and
// prolongation weights laid out once per cycle in shared memory; every block
// holds u of all levels there too, and a new value is stored into the blocks
// that own a neighbour (distributed shared memory).  A pass is then a
// cluster barrier, six shared loads and the part of the update that depends
// on the neighbours, ~7 dependent operations; what depends on the cell's own
// value (for eq. psi the powers of 1 + u and the division) is evaluated while
// the other colour is swept.  Levels of at most FAS_SOLO_CELLS cells run on
// block 0 alone with block barriers.
//
// Eq. psi on 64 x 32 cells: 207 us per cycle launched pass by pass, 159 us in
// a cluster that passed u through global memory (3.5 - 4.9 k cycles per pass
// plus 1.1 - 1.9 k for its barrier), ~70 us so.
#include <cooperative_groups.h>

#include "mg_coarse.cuh"
#include "mg_internal.h"
#include "mg_kernels.cuh"

namespace cg = cooperative_groups;

namespace gmg {

constexpr int FAS_THREADS = 256;
constexpr int FAS_SOLO_THREADS = 128;
static_assert(FAS_SOLO_CELLS <= FAS_SOLO_THREADS && CS_CELLS <= FAS_SOLO_CELLS, "a thread per cell");

// Per-cell values a thread keeps in shared memory (slot v at v * slots + s).
enum {
  FS_E, FS_W, FS_N, FS_S, FS_Z,  // couplings to the neighbours (Z: both)
  FS_C,                          // own value: outer ghosts, - c of a linear equation
  FS_D,                          // Newton diagonal; linear equations: inverted
  FS_A, FS_B,                    // eq. psi: 2 pi U, A2 / 8
  FS_F,                          // right-hand side
  FS_UH,                         // restricted u
  FS_PX, FS_PY, FS_PZ,           // prolongation weights of the parent's neighbours
  FS_R,                          // restriction weight
  FS_COUNT
};
// Compact cell numbers: neighbours, own cell, blocks owning a neighbour (bit
// mask); the parent's neighbours and the parent.
struct __align__(8) FasIndex {
  unsigned short nb[6], q, mask, px[3], parent;
};

// Slots of a level: red cells, then black ones, each padded to whole warps
// so that a colour's pass leaves the other colour's warps alone.
__host__ __device__ __forceinline__ int fas_half(long cells, int size) {
  const int h = (int)(cells / size / 2);
  return h < 32 ? 32 : h;
}

// Where a level's slots and arrays start (in slots, in values of u and of x,
// the restricted residual and later u_H - uh_H), and its sizes.
struct FasAt {
  int slot, u, x;
  int half;    // slots of a colour
  int mine;    // cells of a colour a block owns
  int groups;  // coarse cells a block owns the children of
  int lgroups; // log2
};

__device__ __forceinline__ unsigned smem_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void remote_store(unsigned addr, int rank, double v) {
  unsigned ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(ra), "d"(v) : "memory");
}

template <int G, int KIND>
struct Fas {
  const FasLevel* lv;
  const FasAt* at;
  int nl, solo_from, rank, size, slots;
  double* slot;     // [FS_COUNT][slots]
  FasIndex* index;  // [slots]
  double *u0, *x0;  // u of all levels, x from level 1 on
  double *wr, *wu;  // [FAS_THREADS] weighted residual and u of the block's cells

  // ---- the level being visited
  int l;
  FasAt o;
  int colour, g, s;  // thread's colour, rank in the colour, slot
  bool on, three;
  double c[5], cC, D, a, b8, f, u;
  double q8, X, inv, base;  // of the own value

  __device__ __forceinline__ int team(int m) const { return m < solo_from ? size : 1; }
  __device__ __forceinline__ bool here(int m) const { return rank < team(m); }
  __device__ __forceinline__ void arrive() const { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
  __device__ __forceinline__ void wait() const { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
  __device__ __forceinline__ void solo_sync() const {
    asm volatile("bar.sync 1, %0;" ::"n"(FAS_SOLO_THREADS) : "memory");
  }
  // A barrier of the team of level m; own() runs where it costs least.
  template <typename F>
  __device__ __forceinline__ void sync(int m, F own) const {
    if (m < solo_from) {
      arrive();
      own();
      wait();
    } else {
      solo_sync();
      own();
    }
  }

  // The place of slot tid of level m, the one thread tid works on.
  __device__ __forceinline__ void go(int m, int tid = threadIdx.x) {
    l = m;
    o = at[m];
    colour = tid >= o.half;
    g = tid - colour * o.half;
    s = o.slot + tid;
    on = here(m) && tid < 2 * o.half && g < o.mine;
  }
  // Cells of a level in groups of one coarse cell's children; a block owns
  // consecutive groups.  Thread g of a colour takes pair g % pairs (same
  // (j, k): one red and one black child) of the block's group g / pairs.
  __device__ __forceinline__ void cell(int& i, int& j, int& k) const {
    const LevelView<double>& L = lv[l].v;
    if (l == nl - 1) {
      L.colour_cell(g, colour, i, j, k);
      return;
    }
    const int lp = L.three ? 2 : 1, pc = g & ((1 << lp) - 1);
    const int G0 = (rank << o.lgroups) + (g >> lp);
    const int dj = pc & 1, dk = pc >> 1;
    i = 2 * (G0 & ((L.n0 >> 1) - 1)) + (colour ^ dj ^ dk);
    j = 2 * ((G0 >> (L.ln0 - 1)) & ((L.n1 >> 1) - 1)) + dj;
    k = 2 * (G0 >> (L.ln0 + L.ln1 - 2)) + dk;
  }
  // The block that owns cell q of level m.
  __device__ __forceinline__ int owner(int m, int q) const {
    if (m >= solo_from) return 0;
    const LevelView<double>& L = lv[m].v;
    const int i = q & (L.n0 - 1), j = (q >> L.ln0) & (L.n1 - 1), k = q >> (L.ln0 + L.ln1);
    return ((i >> 1) + ((j >> 1) << (L.ln0 - 1)) + ((k >> 1) << (L.ln0 + L.ln1 - 2))) >> at[m].lgroups;
  }
  __device__ __forceinline__ double& sl(int v) const { return slot[v * slots + s]; }

  // Lay out slot sq (once per cycle, by any thread).
  __device__ __forceinline__ void setup(int sq) {
    int m = 0;
    while (m + 1 < nl && sq >= at[m + 1].slot) ++m;
    go(m, sq - at[m].slot);
    if (!on) return;
    const FasLevel& F = lv[m];
    const LevelView<double>& L = F.v;
    int i, j, k;
    cell(i, j, k);
    CoarseCell<G> cc;
    coarse_cell_load<G>(cc, L, m == 0 ? F.f : nullptr, F.s0, F.s1, i, j, k);
    const double cf[6] = {cc.cE, cc.cW, G == SPH ? cc.cC * cc.cN : cc.cN, G == SPH ? cc.cC * cc.cS : cc.cS,
                          cc.cZ, cc.cZ};
    FasIndex ix;
    ix.q = (unsigned short)cc.q;
    double C = 0.0;
    unsigned mask = 0u;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
      const bool ghost = cc.b[e] < 0;
      if (ghost && cc.g[e] != 1.0) C += cf[e] * (cc.g[e] - 1.0);
      ix.nb[e] = (unsigned short)(ghost ? cc.q : cc.b[e]);
      if (!ghost) mask |= 1u << owner(m, cc.b[e]);
    }
    ix.mask = (unsigned short)(mask & ~(1u << rank));
    for (int e = 0; e < 5; ++e) sl(FS_E + e) = cf[e];
    if (KIND == EQ_PSI) {
      sl(FS_C) = C;
      sl(FS_D) = cc.D;
      sl(FS_A) = (2 * PI_D) * cc.s0;
      sl(FS_B) = 0.125 * cc.s1;
    } else {
      sl(FS_C) = C - cc.s1;
      sl(FS_D) = 1.0 / (cc.D - cc.s1);
    }
    sl(FS_F) = cc.f;
    if (m + 1 < nl) {
      const LevelView<double>& Lc = lv[m + 1].v;
      const int I = i >> 1, J = j >> 1, K = L.three ? k >> 1 : 0;
      ix.parent = (unsigned short)(I + Lc.n0 * (J + Lc.n1 * K));
#pragma unroll
      for (int d = 0; d < 3; ++d) {
        int ci = I, cj = J, ck = K;
        double w = 0.25;
        bool out;
        if (d == 0) {
          ci += (i & 1) ? 1 : -1;
          out = ci < 0 || ci >= Lc.n0;
        } else if (d == 1) {
          cj += (j & 1) ? 1 : -1;
          out = cj < 0 || cj >= Lc.n1;
        } else {
          ck += L.three ? ((k & 1) ? 1 : -1) : 0;
          out = L.three && (ck < 0 || ck >= Lc.n2);
        }
        if (out) w *= ghost_rule(Lc, -1, d, ci, cj, ck);
        ix.px[d] = (unsigned short)(ci + Lc.n0 * (cj + Lc.n1 * ck));
        sl(FS_PX + d) = w;
      }
      const double w00 = L.TI(TI_VW, i) * L.TJ(TJ_VW, j), wi = L.TI(TI_VW, i) + L.TI(TI_VW, i ^ 1),
                   wj = L.TJ(TJ_VW, j) + L.TJ(TJ_VW, j ^ 1);
      sl(FS_R) = w00 / ((L.three ? 2.0 : 1.0) * (wi * wj));
    }
    index[s] = ix;
  }

  __device__ __forceinline__ void load(FasIndex& ix) {
    if (!on) return;
    ix = index[s];
#pragma unroll
    for (int e = 0; e < 5; ++e) c[e] = sl(FS_E + e);
    cC = sl(FS_C);
    D = sl(FS_D);
    if (KIND == EQ_PSI) {
      a = sl(FS_A);
      b8 = sl(FS_B);
    }
    f = sl(FS_F);
    u = u0[o.u + ix.q];
  }
  // What the next update takes from the own value alone.
  __device__ __forceinline__ void own_part() {
    base = fma(cC, u, -f);
    if (KIND == EQ_PSI) {
      const double q = 1.0 + u, q2 = q * q, q4 = q2 * q2, t = a * (q4 * q2);
      q8 = q4 * q4;
      X = (t + b8) * q;
      inv = 1.0 / fma(D, q8, -fma(7.0, b8, t));
    }
  }
  // lap u - c u - f, differences to the own value multiplied by the couplings.
  __device__ __forceinline__ double defect(const FasIndex& ix) const {
    const double* v = u0 + o.u;
    double A = fma(c[0], v[ix.nb[0]] - u, base), B = c[2] * (v[ix.nb[2]] - u);
    A = fma(c[1], v[ix.nb[1]] - u, A);
    B = fma(c[3], v[ix.nb[3]] - u, B);
    if (three) A = fma(c[4], (v[ix.nb[4]] - u) + (v[ix.nb[5]] - u), A);
    return A + B;
  }
  // The nonlinear term of L(u) at the own value.
  __device__ __forceinline__ double source() const {
    if (KIND != EQ_PSI) return 0.0;
    const double ip = 1.0 / (1.0 + u), ip2 = ip * ip, ip4 = ip2 * ip2;
    return a * ip + b8 * (ip4 * ip2 * ip);
  }
  __device__ __forceinline__ void put(const FasIndex& ix, bool others) const {
    double* p = u0 + o.u + ix.q;
    *p = u;
    if (others)
      for (unsigned m = ix.mask; m; m &= m - 1u) remote_store(smem_addr(p), __ffs(m) - 1, u);
  }
  __device__ __forceinline__ void update(const FasIndex& ix, bool others) {
    if (!on) return;
    const double d = defect(ix);
    u -= KIND == EQ_PSI ? fma(d, q8, X) * inv : d * D;
    put(ix, others);
  }
  // Sweeps; tail() by every thread behind the last pass, while its barrier
  // completes; the barrier is left out (with the stores into other blocks)
  // when last.  On block 0 a colour only signals that it is done and waits
  // for the other's signal: what it takes from its own values does not hold
  // up the other colour.
  template <typename F>
  __device__ __forceinline__ void sweeps(const FasIndex& ix, int n, bool last, F tail) {
    if (l < solo_from) {
      for (int h = 0; h < 2 * n; ++h) {
        const bool end = h == 2 * n - 1, mine = (h & 1) == colour;
        if (mine) update(ix, !(end && last));
        if (end && last) break;
        if (end)
          sync(l, tail);
        else
          sync(l, [&] {
            if (on && mine && h + 2 < 2 * n) own_part();
          });
      }
      return;
    }
    auto signal = [](int b) { asm volatile("bar.arrive %0, %1;" ::"r"(b), "n"(FAS_SOLO_THREADS) : "memory"); };
    auto await = [](int b) { asm volatile("bar.sync %0, %1;" ::"r"(b), "n"(FAS_SOLO_THREADS) : "memory"); };
    for (int k = 0; k < n; ++k) {
      if (colour == 0) {
        if (k > 0) await(3);  // the black cells
        update(ix, false);
        signal(2);
      } else {
        await(2);
        update(ix, false);
        if (k + 1 < n) signal(3);
      }
      if (on && k + 1 < n) own_part();
    }
    if (!last) {
      solo_sync();
      tail();
    }
  }

  // Right-hand side L_H(u_H) + R r of a level below the first.  It reads the
  // neighbours' restricted u, which the first sweep replaces: a barrier of the
  // level's team stands between the two.
  __device__ __forceinline__ void rhs(const FasIndex& ix) {
    if (!on) return;
    f = 0.0;
    base = cC * u;
    f = defect(ix) + source() + x0[o.x + ix.q];
    sl(FS_F) = f;
    sl(FS_UH) = u;
  }

  __device__ __forceinline__ void down(int m, int nu1) {
    go(m);
    FasIndex ix;
    load(ix);
    auto own = [&] {
      if (on && nu1 > 0) own_part();
    };
    if (m > 0) {
      rhs(ix);
      sync(m, own);  // every right-hand side before the first new value
    } else {
      own();
    }
    double nl_term = 0.0;
    auto before = [&] {
      if (on) {
        base = fma(cC, u, -f);
        nl_term = source();
      }
    };
    if (nu1 > 0)
      sweeps(ix, nu1, false, before);
    else
      before();
    if (on) {
      const double w = sl(FS_R);
      wr[threadIdx.x] = -w * (defect(ix) + nl_term);
      wu[threadIdx.x] = w * u;
    }
    if (m < solo_from)
      __syncthreads();
    else
      solo_sync();
    // the block's coarse cells: sums over the pairs of a group
    if ((int)threadIdx.x < o.groups) {
      const int hp = o.half, lp = three ? 2 : 1;
      const double *r = wr + (threadIdx.x << lp), *v = wu + (threadIdx.x << lp);
      double R = (r[0] + r[hp]) + (r[1] + r[hp + 1]), V = (v[0] + v[hp]) + (v[1] + v[hp + 1]);
      if (three) {
        R += (r[2] + r[hp + 2]) + (r[3] + r[hp + 3]);
        V += (v[2] + v[hp + 2]) + (v[3] + v[hp + 3]);
      }
      const int q = (rank << o.lgroups) + threadIdx.x;  // groups are numbered like the coarse cells
      double *pu = u0 + at[m + 1].u + q, *px = x0 + at[m + 1].x + q;
      const int to = owner(m + 1, q);
      if (team(m) == 1) {
        *pu = V;
        *px = R;
      } else {
        remote_store(smem_addr(px), to, R);
        for (int b = 0; b < team(m + 1); ++b) remote_store(smem_addr(pu), b, V);
      }
    }
    sync(m, [] {});
  }

  // Correction from level m + 1 (behind a barrier), post-sweeps; u - uh to
  // the blocks of the level above, or u back to HBM.
  __device__ __forceinline__ void up(int m, int nu2) {
    go(m);
    FasIndex ix;
    load(ix);
    sync(m, [] {});
    if (on) {
      const double* e = x0 + at[m + 1].x;
      double add = fma(sl(FS_PX), e[ix.px[0]], sl(FS_PY) * e[ix.px[1]]);
      if (three)
        add += fma(sl(FS_PZ), e[ix.px[2]], 0.25 * e[ix.parent]);
      else
        add = fma(0.5, e[ix.parent], add);
      u += add;
      put(ix, nu2 > 0);
    }
    if (nu2 > 0) {
      sync(m, [&] {
        if (on) own_part();
      });
      sweeps(ix, nu2, true, [] {});
    }
    finish(ix);
  }
  __device__ __forceinline__ void finish(const FasIndex& ix) const {
    if (!on) return;
    if (l == 0) {
      int i, j, k;
      cell(i, j, k);
      lv[0].u[lv[0].v.idx(i, j, k)] = u;
      return;
    }
    const double e = u - sl(FS_UH);
    double* p = x0 + o.x + ix.q;
    *p = e;
    for (int b = 0; b < team(l - 1); ++b)
      if (b != rank) remote_store(smem_addr(p), b, e);
  }
  __device__ __forceinline__ void coarsest(int n) {
    go(nl - 1);
    FasIndex ix;
    load(ix);
    rhs(ix);
    sync(nl - 1, [&] {  // every right-hand side before the first new value
      if (on) own_part();
    });
    sweeps(ix, n, true, [] {});
    finish(ix);
  }
};

// Shared memory of a cycle: levels, u, x, two values per thread, slots.
struct FasShape {
  int nu, nx, slots;
};
inline size_t fas_smem(const FasShape& S) {
  return (sizeof(FasLevel) + sizeof(FasAt)) * FAS_MAX + sizeof(double) * (S.nu + S.nx + 2 * FAS_THREADS + (size_t)FS_COUNT * S.slots) +
         sizeof(FasIndex) * S.slots;
}
inline FasShape fas_shape(const FasCycle& P, int cluster) {
  FasShape S{0, 0, 0};
  for (int l = 0; l < P.nl; ++l) {
    const int n = (int)ncells(P.lv[l].v);
    S.nu += n;
    if (l > 0) S.nx += n;
    S.slots += 2 * fas_half(n, l < P.solo_from ? cluster : 1);
  }
  return S;
}

template <int G, int KIND>
__global__ void __launch_bounds__(FAS_THREADS) k_fas_cycle(const __grid_constant__ FasCycle P, const FasShape S) {
  extern __shared__ __align__(16) unsigned char sm[];
  Fas<G, KIND> T;
  T.nl = P.nl;
  T.solo_from = P.solo_from;
  T.rank = (int)cg::this_cluster().block_rank();
  T.size = (int)cg::this_cluster().num_blocks();
  FasAt* const at = reinterpret_cast<FasAt*>(sm + sizeof(FasLevel) * FAS_MAX);
  T.lv = reinterpret_cast<const FasLevel*>(sm);
  T.at = at;
  T.three = P.lv[0].v.three;
  T.u0 = reinterpret_cast<double*>(at + FAS_MAX);
  T.x0 = T.u0 + S.nu;
  T.wr = T.x0 + S.nx;
  T.wu = T.wr + FAS_THREADS;
  T.slot = T.wu + FAS_THREADS;
  T.slots = S.slots;
  T.index = reinterpret_cast<FasIndex*>(T.slot + (size_t)FS_COUNT * S.slots);
  for (int q = threadIdx.x; q < (int)(sizeof(FasLevel) / 4) * P.nl; q += FAS_THREADS)
    reinterpret_cast<unsigned*>(sm)[q] = reinterpret_cast<const unsigned*>(P.lv)[q];
  if (threadIdx.x == 0) {
    FasAt o{};
    for (int l = 0; l < P.nl; ++l) {
      const LevelView<double>& L = P.lv[l].v;
      const int n = L.n0 * L.n1 * L.n2, team = T.team(l);
      o.half = fas_half(n, team);
      o.mine = n / team / 2;
      o.groups = n / team / (T.three ? 8 : 4);
      o.lgroups = 31 - __clz(o.groups);
      at[l] = o;
      o.slot += 2 * o.half;
      o.u += n;
      if (l > 0) o.x += n;
    }
  }
  __syncthreads();
  pdl_entry();
  const LevelView<double>& L0 = T.lv[0].v;
#pragma unroll 8
  for (int q = threadIdx.x; q < L0.n0 * L0.n1 * L0.n2; q += FAS_THREADS) T.u0[q] = T.lv[0].u[interior_p(L0, q)];
  for (int q = threadIdx.x; q < S.slots; q += FAS_THREADS) T.setup(q);
  // every block has started before the first store into another one
  T.arrive();
  T.wait();
  const int nl = P.nl;
  for (int l = 0; l + 1 < nl && T.here(l); ++l) {
    if (l >= P.solo_from && threadIdx.x >= FAS_SOLO_THREADS) break;
    T.down(l, P.nu1);
  }
  const bool solo = T.rank == 0 && threadIdx.x < FAS_SOLO_THREADS;
  if (solo) T.coarsest(P.coarse_sweeps);
  for (int l = nl - 2; l >= 0; --l) {
    if (l >= P.solo_from ? !solo : !T.here(l)) continue;
    T.up(l, P.nu2);
  }
}

using FasKernel = void (*)(FasCycle, FasShape);

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

// Most shared memory a cycle takes: levels of 4096 cells and each a quarter
// of the one before.
static size_t fas_smem_max(int cluster) {
  FasShape S{0, 0, 0};
  for (long n = FAS_CLUSTER_CELLS; n >= 4; n /= 4) {
    S.nu += (int)n;
    if (n < FAS_CLUSTER_CELLS) S.nx += (int)n;
    S.slots += 2 * fas_half(n, n > FAS_SOLO_CELLS ? cluster : 1);
  }
  return fas_smem(S);
}

static cudaLaunchConfig_t fas_config(int cluster, size_t smem, cudaStream_t st, cudaLaunchAttribute* at) {
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)cluster;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)cluster);
  cfg.blockDim = dim3(FAS_THREADS);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cfg;
}

void init_fas_attributes() {
  int best = 16;
  for (int g = 0; g < 3; ++g)
    for (int kind = EQ_PSI; kind <= EQ_LIN; ++kind) {
      FasKernel k = fas_kernel(g, kind);
      cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
      if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fas_smem_max(8)) != cudaSuccess) {
        cudaGetLastError();
        best = 0;
      }
      for (; g_fas_cluster < 0 && best >= 8; best /= 2) {
        cudaLaunchAttribute at[2];
        cudaLaunchConfig_t cfg = fas_config(best, fas_smem_max(best), nullptr, at);
        cfg.numAttrs = 1;
        int nc = 0;
        if (cudaOccupancyMaxActiveClusters(&nc, k, &cfg) == cudaSuccess && nc > 0) break;
        cudaGetLastError();
      }
    }
  if (g_fas_cluster < 0) g_fas_cluster = best >= 8 ? best : 0;
}

long fas_cycle_cells() { return std::min<long>(FAS_CLUSTER_CELLS, (long)g_fas_cluster * FAS_THREADS); }

void launch_fas_cycle(const FasCycle& P, int geom, int kind, cudaStream_t st) {
  count_launch();
  cudaLaunchAttribute at[2];
  const FasShape S = fas_shape(P, g_fas_cluster);
  const cudaLaunchConfig_t cfg = fas_config(g_fas_cluster, fas_smem(S), st, at);
  cudaLaunchKernelEx(&cfg, fas_kernel(geom, kind), P, S);
}

}  // namespace gmg
