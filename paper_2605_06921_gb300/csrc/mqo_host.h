// mqo_host.h -- launchers shared by the host runtime of the mQO library.
#pragma once

#include <cuda_runtime.h>

#include "../../include/mqo.h"
#include "mqo_dev.cuh"

namespace mqo {

constexpr int kPairThreads = 256;  // pair kernels: (node, trajectory) per thread

// The most dynamic shared memory a plan may ask of each kind of kernel, and
// what every launch of such a kernel allows it (allow_smem): the same value
// whatever the solver, so that host threads whose solvers need different
// amounts do not lower each other's limit between the call and the launch.
constexpr size_t kStepSmemLimit = 110 * 1024;     // shared-memory step kernels: the member graph's block fits
constexpr size_t kDiscSmemLimit = 160 * 1024;     // fused discrete kernel: the member graph's bit words fit
constexpr size_t kDiscBitsSmemLimit = 120 * 1024; // its form on bit matrices
constexpr size_t kSmallSmemLimit = 200 * 1024;    // multi-tick kernel: a member graph and its trajectories fit
constexpr size_t kStagedSmemLimit = 200 * 1024;   // staged-gather step kernel: a slice fits
constexpr size_t kDenseSmemLimit = 224 * 1024;    // tensor-core step: 32 trajectories of a member graph's x fit
template <typename K>
inline cudaError_t allow_smem(K kern, size_t limit) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)limit);
}

enum CtrlMode : int { CTRL_MACHINE = 0, CTRL_LS_BEGIN = 1, CTRL_LS = 2, CTRL_RESET = 3 };

struct DensePlan;
// smem > 0: the shared-memory kernel with that much dynamic shared memory,
// with the sliced-ELL neighbour stream when `ell` is given (build_ell);
// `dense`: the tensor-core kernel of dense member graphs instead
cudaError_t launch_step(const SolverDev& S, Counters* cnt, const int32_t* act, const int32_t* gflag_step,
                        size_t smem, cudaStream_t stream, const int4* ell, const int2* ell_pos,
                        const DensePlan* dense, int sms);
// the sliced-ELL stream of the shared-memory step kernel (mqo_step_smem.cuh)
// for `rpw` rows per warp and x rows `pitch` bytes apart, from the group
// table `pos` (one entry per processing position)
cudaError_t launch_ell_fill(const GraphDev& g, int rpw, int pitch, const int2* pos, int4* ell, cudaStream_t s);
// dense member graphs on the tensor cores (mqo_step_dense.cuh): their bit
// matrices, the CTAs per (member graph, 32 trajectories), the dynamic shared
// memory of a CTA and the bits of the largest degree (degree < 2^sum_bits);
// the looks of a wait inside the kernel before it gives up, and the word in
// pinned host memory that it sets then
constexpr uint32_t kDensePolls = 1u << 26;
struct DensePlan {
  const uint4* bits;
  const int64_t* bits_off;  // per member graph: first uint4
  int32_t parts;
  int32_t sum_bits;
  size_t smem;
  uint32_t polls;
  int32_t* late;
};
cudaError_t launch_dense_bits(const GraphDev& g, const int64_t* bits_off, const int2* tiles, int num_tiles,
                              uint4* bits, cudaStream_t s);
size_t dense_smem_bytes(int max_ng);
// the stream of x staged as float32 (mqo_step_f32.cu): 16-bit entries
cudaError_t launch_ell_fill16(const GraphDev& g, int rpw, int pitch, const int2* pos, int4* ell, cudaStream_t s);
bool step_wide_possible(int B, int x_dtype);
// the row-group kernel (mqo_step_rows.cu)
bool step_rows_possible(int B, int x_dtype, int problem, int objective, int max_degree);
int default_step_vec(int B, int x_dtype);
bool staged_vec_ok(int B, int x_dtype, int vec);
int default_staged_vec(int B, int x_dtype);
size_t step_smem_bytes(int B, int x_dtype, int problem, int max_ng);

// small member graphs: `count` ticks (plain == nullptr) or plain steps in one
// launch, advancing the tick number (mqo_small.cu)
size_t small_smem_bytes(int B, int x_dtype, int v_dtype, int ng, int nnz, bool weighted);
cudaError_t launch_small(const SolverDev& S, int count, Counters* plain, int threads, size_t smem, cudaStream_t s);

cudaError_t launch_ctrl(const SolverDev& S, int mode, const uint8_t* mask, cudaStream_t stream);
cudaError_t launch_apply(const SolverDev& S, cudaStream_t stream);
cudaError_t launch_disc(const SolverDev& S, int pass, cudaStream_t stream);
size_t disc_graph_smem_bytes(int B, int max_ng);
cudaError_t launch_disc_graph(const SolverDev& S, size_t smem, cudaStream_t stream);
// the same for member graphs with bit matrices (mqo_disc_bits.cu)
size_t disc_bits_smem_bytes(int problem, int max_ng);
int disc_bits_ctas(const SolverDev& S, int sms);
cudaError_t launch_disc_bits(const SolverDev& S, const uint4* bits, const int64_t* bits_off, size_t smem,
                             int sms, cudaStream_t stream);
cudaError_t launch_tick_end(const SolverDev& S, cudaStream_t stream);
cudaError_t launch_round_bits(const SolverDev& S, uint32_t* z, cudaStream_t stream);
cudaError_t launch_eval(const SolverDev& S, const uint32_t* z, Counters* out, cudaStream_t stream);
cudaError_t launch_eval_bits(const SolverDev& S, const uint4* bits, const int64_t* bits_off, int max_ng,
                             const uint32_t* z, Counters* out, cudaStream_t stream);
cudaError_t launch_counters_out(const SolverDev& S, const Counters* c, int64_t* value, int64_t* a, int64_t* b,
                                int kind, cudaStream_t stream);
cudaError_t launch_objective(const SolverDev& S, double* out, cudaStream_t stream);
cudaError_t launch_ls_merge(const SolverDev& S, const TrajState* saved, cudaStream_t stream);
cudaError_t launch_init(const SolverDev& S, Counters* plain, cudaStream_t stream);
cudaError_t launch_any_pending(const SolverDev& S, int32_t* out, cudaStream_t stream);
// device check of the CSR entries (range, no self loop, strictly ascending
// rows, weights in {-1,+1}, no edge between member graphs, a reverse entry
// with the same weight): *bad_row <- the smallest row with a bad entry
// (unchanged if none); synchronous
cudaError_t launch_validate_csr(const int32_t* rp, const int32_t* col, const int8_t* w, const int32_t* node_off,
                                int32_t G, int32_t n, int32_t* bad_row, int sms, cudaStream_t stream);
cudaError_t launch_pool_ctrl(const SolverDev& S, cudaStream_t stream);
// 16-bit member-local copies of the column indices (every member graph below 65536 nodes)
cudaError_t launch_col16(const GraphDev& g, uint16_t* col16, cudaStream_t stream);
cudaError_t launch_pool_apply(const SolverDev& S, cudaStream_t stream);

// graph-level kernels (autograd path)
struct HeavyPlan {
  const int32_t* light_rows;  // rows handled whole
  int32_t num_light;
  const int32_t* heavy_row;   // per chunk: row
  const int32_t* heavy_j0;    // per chunk: first entry
  const int32_t* heavy_j1;    // per chunk: end entry
  int32_t num_chunks;
  const int32_t* heavy_rows;  // distinct heavy rows
  const int32_t* heavy_first; // per heavy row: first chunk
  int32_t num_heavy;
  // the chunks, {row, -1 - chunk, first entry, end entry}, then the light rows in
  // segments of consecutive rows (no heavy row inside) of about kFbSegEntries
  // entries: {first row, end row, first entry, end entry}
  const int4* segs;
  int32_t num_segs;
};
constexpr int kFbSegEntries = 512;

// the shared-memory bandwidth probe (mqo_probe.cu): `grid` CTAs of
// smem_probe_threads() threads, `iters` iterations of four 16-byte loads each
cudaError_t launch_smem_probe(int grid, int32_t iters, uint32_t* sink, cudaStream_t s);
int smem_probe_threads();

cudaError_t launch_fb(const GraphDev& g, const HeavyPlan& hp, const float* X, int B, float lambda_,
                      const float* gout, float* G, float* AX, double* obj, float* scratch, int grid,
                      cudaStream_t stream);
cudaError_t launch_grad_ax(const float* AX, const float* gout, float* G, int64_t n, int B, float lambda_,
                           cudaStream_t s);
cudaError_t launch_momentum(float* x, float* v, const float* grad, int64_t n, float lr, float mu, float lo,
                            float hi, cudaStream_t stream);
cudaError_t launch_adam(float* x, float* m, float* u, const float* grad, int64_t n, float lr, float b1, float b2,
                        float eps, int64_t t, float lo, float hi, cudaStream_t stream);

// read-only view of a graph's device CSR and its long-row statistics
// (rows longer than 512 entries, and their 512-entry chunks)
struct GraphCsrView {
  const int32_t* row_ptr;
  const int32_t* col;
  const int8_t* w;
  int32_t n;
  int32_t long_rows;
  int64_t long_chunks;
  int32_t sms;  // multiprocessors of the device the graph was created on
};

}  // namespace mqo

struct mqo_graph_s;
void graph_csr_view(mqo_graph_s* g, mqo::GraphCsrView* out);
mqo_status set_last_error(mqo_status status, const char* msg);
