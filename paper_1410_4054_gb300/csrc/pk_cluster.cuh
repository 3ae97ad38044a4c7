// Reductions shared by the solvers that run a whole iteration loop on one thread-block
// cluster with their vectors in the CTAs' shared memory (pipelined CG and BiCGStab on one
// system, and the batched solver's cluster engine).
//
// A fused phase ends with a block sum of its partial inner products into the CTA's slots, a
// hardware cluster barrier, and the cluster total: every CTA reads all C CTAs' slots in rank
// order through distributed shared memory and adds them with the same butterfly, so every CTA
// holds bit-identical scalars and takes the same decisions (control flow stays uniform across
// the cluster; there is no spin-wait).
#pragma once

#include <cooperative_groups.h>

#include "pk_internal.cuh"

namespace pk {

namespace cg = cooperative_groups;

// Block sums of NV values over NT threads into slots[0 .. NV): warp sums (integer arithmetic,
// pk_internal.cuh: the FP64 pipe belongs to the row products), then warp k adds the warps' values
// of sum k.  The caller's cluster barrier publishes the slots and frees buf (NV * NT / 32 doubles).
template <int NT, int NV>
__device__ __forceinline__ void cluster_block_slots(double (&v)[NV], double* buf, double* slots) {
  constexpr int NW = NT / 32;
  static_assert(NW >= NV && NW <= 32, "one warp per sum");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  warp_sums<NV>(v);
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < NV; ++k) buf[k * NW + warp] = v[k];
  }
  __syncthreads();
  if (warp < NV) {
    const double t = warp_sum(lane < NW ? buf[warp * NW + lane] : 0.0);
    if (lane == 0) slots[warp] = t;
  }
}

// Cluster totals of slots [s0, s0 + NV) of every CTA, in warp 0 (after a cluster barrier): lane c
// reads CTA c's values from distributed shared memory; every CTA adds the same values, so all hold
// the same bits.  Thread 0 goes on with the scalar work and broadcasts its result.
template <int NV>
__device__ __forceinline__ void cluster_total(cg::cluster_group& cl, double* slots, int s0, double (&out)[NV]) {
  const int lane = threadIdx.x & 31;
  const double* rem = lane < (int)cl.num_blocks() ? cl.map_shared_rank(slots, lane) : nullptr;
#pragma unroll
  for (int k = 0; k < NV; ++k) out[k] = rem ? rem[s0 + k] : 0.0;
  warp_sums<NV>(out);
}

// Rows over a cluster: CTA k owns rows [k R, (k + 1) R).
struct ClusterRows {
  int R;
  uint32_t inv;  // ceil(2^32 / R): c / R = mulhi(c, inv) for c R < 2^32
  __device__ __forceinline__ explicit ClusterRows(int rows) : R(rows), inv(0xffffffffu / (uint32_t)rows + 1) {}
};

// Rows per CTA for n rows on C CTAs: equal shares in whole warps, at least one warp's.  (Shares of a
// power of two left up to half of the CTAs without rows.)
__host__ __device__ inline int cluster_share(int64_t n, int C) {
  const int64_t r = (n + C - 1) / C;
  return r <= 32 ? 32 : (int)((r + 31) & ~(int64_t)31);
}

// Element `c` of a vector distributed over the cluster, each CTA's part at `local` in its shared
// memory.
__device__ __forceinline__ double cluster_elem(cg::cluster_group& cl, const ClusterRows& rows, double* local, int c) {
  const int k = (int)__umulhi((uint32_t)c, rows.inv);
  return *cl.map_shared_rank(local + (c - k * rows.R), k);
}

// Row of A times a distributed vector: four entries per step with their loads
// independent, products added left to right.  j, j1: the row's entries.
__device__ __forceinline__ double cluster_row(cg::cluster_group& cl, const ClusterRows& rows,
                                              const int32_t* __restrict__ ci, const double* __restrict__ va,
                                              double* local, int j, const int j1) {
  double s = 0.0;
  for (; j + 4 <= j1; j += 4) {
    int c[4];
    double w[4], pv[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      c[k] = __ldg(ci + j + k);
      w[k] = __ldg(va + j + k);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) pv[k] = cluster_elem(cl, rows, local, c[k]);
#pragma unroll
    for (int k = 0; k < 4; ++k) s = fma(w[k], pv[k], s);
  }
  for (; j < j1; ++j) s = fma(__ldg(va + j), cluster_elem(cl, rows, local, __ldg(ci + j)), s);
  return s;
}

}  // namespace pk
