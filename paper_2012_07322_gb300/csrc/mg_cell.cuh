// Thread-block clusters whose blocks hold a level in shared memory: stores
// into another block's shared memory, barriers, and which cell a thread owns.
#pragma once
#include "mg_internal.h"
#include "mg_kernels.cuh"

namespace gmg {

__device__ __forceinline__ unsigned cl_addr(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned cl_map(unsigned addr, int rank) {
  unsigned ra;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(ra) : "r"(addr), "r"(rank));
  return ra;
}
__device__ __forceinline__ void cl_store(unsigned addr, int rank, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cl_map(addr, rank)), "f"(v) : "memory");
}
__device__ __forceinline__ void cl_store(unsigned addr, int rank, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(cl_map(addr, rank)), "d"(v) : "memory");
}
__device__ __forceinline__ void cl_sync() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}

// The cell of a thread.  Cells are dealt in groups of one coarse cell's
// children, consecutive groups to a block, red cells to the first threads and
// black ones to the others; thread g of a colour takes pair g % pairs (same
// (j, k)) of group g / pairs.
struct ClCell {
  int tid, rank, size, half, groups, lgroups, lp, colour;
  bool on;
  int i, j, k, p;  // p: offset in the ghosted level
  template <typename LV>
  __device__ __forceinline__ ClCell(const LV& L, int r, int s) : tid(threadIdx.x), rank(r), size(s) {
    const int n = L.n0 * L.n1 * L.n2, mine = n / size / 2;
    half = max(mine, 32);  // a colour's threads, in whole warps
    lp = L.three ? 2 : 1;
    groups = (n >> (lp + 1)) / size;
    lgroups = 31 - __clz(groups);
    colour = tid >= half;
    const int g = tid - colour * half, pc = g & ((1 << lp) - 1), G0 = (rank << lgroups) + (g >> lp), dj = pc & 1, dk = pc >> 1;
    on = g < mine;
    i = 2 * (G0 & ((L.n0 >> 1) - 1)) + (colour ^ dj ^ dk);
    j = 2 * ((G0 >> (L.ln0 - 1)) & ((L.n1 >> 1) - 1)) + dj;
    k = 2 * (G0 >> (L.ln0 + L.ln1 - 2)) + dk;
    p = (int)L.idx(i, j, k);
  }
  // A barrier of the blocks that work on the level.
  __device__ __forceinline__ void sync() const {
    if (size > 1)
      cl_sync();
    else
      __syncthreads();
  }
  template <typename LV>
  __device__ __forceinline__ int owner(const LV& L, int a, int b, int c) const {
    return ((a >> 1) + ((b >> 1) << (L.ln0 - 1)) + ((c >> 1) << (L.ln0 + L.ln1 - 2))) >> lgroups;
  }
  // Restriction weight, normalised over the cell's group.
  template <typename T>
  __device__ __forceinline__ T weight(const LevelView<T>& L) const {
    const T wi = L.TI(TI_VW, i), wj = L.TJ(TJ_VW, j);
    const T si = wi + L.TI(TI_VW, i ^ 1), sj = wj + L.TJ(TJ_VW, j ^ 1);
    return wi * wj / ((L.three ? T(2) : T(1)) * (si * sj));
  }
  // Sum of a group's values w[thread].
  template <typename T>
  __device__ __forceinline__ T group_sum(const T* w, int g) const {
    const T* r = w + (g << lp);
    T s = (r[0] + r[half]) + (r[1] + r[half + 1]);
    if (lp == 2) s += (r[2] + r[half + 2]) + (r[3] + r[half + 3]);
    return s;
  }
};

}  // namespace gmg
