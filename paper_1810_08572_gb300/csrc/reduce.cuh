// Grid-wide reductions in one launch (device side).
#pragma once

#include "common.cuh"

namespace fvs {

constexpr int RB = 256;   // threads per reduction block

// ---------------------------------------------------------------------------
// Deterministic reductions: every block writes its partial sums; the last
// block to finish (ticket) adds the partials in block order, so the result
// does not depend on scheduling, and then applies the scalar bookkeeping.
//
// FP64 issues at two lanes a clock and SM on this part (0.53 T operations/s
// measured), so a reduction's own arithmetic shows: a block first folds its
// eight warps through shared memory (one warp per sum: seven adds and five
// shuffles) instead of shuffling in each of them (45 warp adds per sum), and
// the quotients of the Krylov recurrences (alpha, omega, beta) are formed
// once, by the thread that finishes the reduction, instead of by every
// thread of the vector kernel that uses them (311,296 threads x 2 divisions
// were 14 us a launch whatever the vector's length).  The grid follows the
// vector's length below one full wave, so short vectors have few partials.
// k_bicg_xr_dot 46.2 -> 30.8 us, k_bicg_p 20.3 -> 10.7, k_bicg_s 12.0 -> 6.8
// at 2,097,152 rows (22, 10 and 7.4 us of memory traffic); k_cg_xr_dot
// 17.2 -> 8.4, k_dot_rz 11.3 -> 7.1, k_cg_p 8.0 -> 3.2 at 422,000 rows.
// ---------------------------------------------------------------------------
struct OpSum { static __device__ __forceinline__ double f(double a, double b) { return a + b; } };
struct OpMax { static __device__ __forceinline__ double f(double a, double b) { return fmax(a, b); } };

// NS sums (1 to 3) of the RB threads of a block; result s (s < NS) is valid
// in lane 0 of warp s
template <class OP, int NS>
__device__ __forceinline__ double block_fold(const double (&a)[NS]) {
  __shared__ double sh[NS][RB];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < NS; ++k) sh[k][threadIdx.x] = a[k];
  __syncthreads();
  double v = 0.0;
  if (w < NS) {
    const double* q = sh[w] + lane;
    v = OP::f(OP::f(OP::f(q[0], q[32]), OP::f(q[64], q[96])), OP::f(OP::f(q[128], q[160]), OP::f(q[192], q[224])));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = OP::f(v, __shfl_down_sync(0xffffffffu, v, o));
  }
  return v;
}

// Grid-wide sums of a[0 .. NS - 1]: true in thread 0 of the block that
// finishes last, with the sums in a.  All partials are non-negative under
// OpMax.
template <class OP, int NS>
__device__ __forceinline__ bool grid_fold(double (&a)[NS], double* part, unsigned int* ticket) {
  __shared__ bool last;
  __shared__ double fin[NS];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double v = block_fold<OP, NS>(a);
  if (w < NS && lane == 0) {
    part[(size_t)w * gridDim.x + blockIdx.x] = v;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double x[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) x[k] = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += RB) {
#pragma unroll
    for (int k = 0; k < NS; ++k) x[k] = OP::f(x[k], __ldcg(part + (size_t)k * gridDim.x + i));
  }
  v = block_fold<OP, NS>(x);
  if (NS > 1) {
    if (w < NS && lane == 0) fin[w] = v;
    __syncthreads();
  }
  if (threadIdx.x != 0) return false;
  a[0] = v;
#pragma unroll
  for (int k = 1; k < NS; ++k) a[k] = fin[k];
  *ticket = 0u;
  return true;
}
template <class OP, int NS>
__device__ __forceinline__ bool grid_fold(double& a, double& b, double* part, unsigned int* ticket) {
  double v[NS];
  v[0] = a;
  if (NS > 1) v[NS - 1] = b;
  if (!grid_fold<OP, NS>(v, part, ticket)) return false;
  a = v[0];
  b = NS > 1 ? v[NS - 1] : 0.0;
  return true;
}

}  // namespace fvs
