// mqo_step_dense.cuh -- the fused descent step of dense member graphs on the
// tensor cores (k_step_t).  The step itself (gradient, momentum, projection,
// rounding, exact evaluation) is the one of mqo_step.cuh.
//
// Why: with 16-bit x the CSR kernels gather nnz rows of x from shared memory
// and are bound by those loads and by issue (162 us per step of 512 graphs,
// n ~ 750, p = 0.15, B = 32).  At this density the product A X is a
// contraction: A as bits is n^2/8 bytes (36 MB for the batch, L2-resident)
// and 2 n^2 B flops run on the tensor cores in a few microseconds.
//
// Why it gives the same bits: the float32 sum of a row in CSR order equals
// the exact sum whenever every partial sum is representable.  16-bit values
// |x| in [2^-t, 1] are multiples of 2^-(t+p-1) (p = 8 for bfloat16, 11 for
// float16), so all partial sums below 2^s are exact in float32 if
// s + t + p - 1 <= 24, in any order, and the tensor core's float32
// accumulation of them is exact too.  Pairs (row, trajectory) that this
// does not cover (a neighbour whose x is small, out of the box or not
// finite) are found by the same product: every x has a companion column w
// (1 if x rounds into the set, 2^10 if small, 2^14 if tiny or irregular)
// whose row sums count both the neighbours in the set and the doubtful
// ones.  Doubtful pairs (0.3 % of a BF16 MIS run) are listed and summed again
// one by one in CSR order; a warp with many of them sums its 32 rows again,
// and a block of x with many small values skips the product.
//
// Measured (BF16, one step): 512 graphs, n ~ 750, degree 112, B = 32, inside the
// machine: 162 us (sliced ELL) -> 104 us; 8 graphs (1000, 100), B = 128:
// 130 (staged) -> 24 us; 8 graphs (1000, 500), B = 128, MaxCut: 264 -> 27 us on
// binary points, 150 us with every row summed in CSR order.  Bound by the
// latency between the warps that expand A and the MMAs (tensor pipe 20 %
// active, issue 42 %): TMEM holds two chunks of A per row tile.
#pragma once

#include "mqo_step.cuh"

namespace mqo {

constexpr int kDenseThreads = 256;  // two warpgroups, each with row tiles of its own,
constexpr int kIssuer = 8;          // and a warp that issues their MMAs
constexpr int kDenseGroup = 32;     // trajectories per CTA
constexpr int kDoubtful = 1024;     // doubtful pairs a CTA lists
// of 1024 pairs of a warp and tile: with more the rows are summed again (for
// MIS most x are 0 and a listed pair skips them)
constexpr int kDoubtfulMis = 200, kDoubtfulCut = 48;
constexpr uint32_t kDenseTmem = 256;  // TMEM columns per CTA: 2 x (64 sums + 2 x 32 of A)

// geometry of the bit matrix of a member graph with ng nodes: row tiles of
// 128, columns in pieces of 128 (one uint4 per row)
__host__ __device__ __forceinline__ int dense_tiles(int ng) { return (ng + 127) >> 7; }

struct DenseArgs {
  const uint4* bits;          // all member graphs
  const int64_t* bits_off;    // per member graph: its first uint4
  int32_t parts;              // CTAs per (member graph, trajectory group)
  int32_t groups;             // trajectory groups: B / 32
  float t0, t1;               // |x| >= t0: exact up to the largest degree; >= t1: up to s1
  float s1x2;                 // 2 * s1
  float degree;               // mean degree of all member graphs
  volatile int32_t* late;       // set if a wait ran out (pinned host memory)
  uint32_t polls;               // looks of a wait
};

cudaError_t launch_step_dense(const StepArgs& a, const DensePlan& p, int x_dtype, int v_dtype, cudaStream_t s);

}  // namespace mqo
