// mqo_api.cu -- host runtime and C ABI of the mQO library (see include/mqo.h).
//
// Graphs are validated once on the host and deep-copied to device memory.
// A solver owns all device state of its trajectories and an internal
// non-blocking stream; every call is ordered after earlier work of the
// caller's stream and before later work on it through a pair of events.
// The machine's tick (control, apply, step, three discrete passes, tick
// end) is captured once as a CUDA graph and replayed.
#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <string>
#include <thread>
#include <vector>

#include "../../include/mqo.h"
#include "mqo_host.h"
#include "mqo_step_dense.cuh"

using namespace mqo;

namespace {

thread_local std::string g_err;

mqo_status fail(mqo_status st, const char* fmt, ...) {
  char buf[512];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof(buf), fmt, ap);
  va_end(ap);
  g_err = buf;
  return st;
}

constexpr int kChunkNodes = kItemMaxNodes;  // nodes per item
constexpr int kSplit = 512;       // row length above which the f_B kernels chunk a row
constexpr int kSmallTicks = 4096;               // ticks per launch of that kernel
constexpr int kDenseMaxDegree = 1023;  // tensor-core step: neighbour counts take 10 bits
constexpr int64_t kL2Bytes = (int64_t)129 << 20;
constexpr double kDenseFill = 0.04;    // and this share of the bit matrices' cells is set (3.1 bytes per CSR entry at most)
constexpr int kDefaultSliceKB = 32;  // staged step kernel: gathered x rows per slice (KB)

}  // namespace

#define CKG(call)                                                                                   \
  do {                                                                                              \
    cudaError_t e_ = (call);                                                                        \
    if (e_ != cudaSuccess) return fail(MQO_ECUDA, "%s failed: %s", #call, cudaGetErrorString(e_)); \
  } while (0)

struct mqo_graph_s {
  int64_t n = 0, nnz = 0;
  int32_t G = 0;
  int32_t* d_rp = nullptr;
  int32_t* d_col = nullptr;
  int8_t* d_w = nullptr;
  int32_t* d_off = nullptr;
  int32_t* d_dmax = nullptr;
  Item* d_items = nullptr;
  int32_t* d_order = nullptr;
  uint16_t* d_col16 = nullptr;  // member-local column indices (every member graph below 65536 nodes)
  // bit matrices of dense member graphs (mqo_step_dense.cuh), built at creation
  uint4* d_bits = nullptr;
  int64_t* d_bits_off = nullptr;
  int32_t max_ng = 0, max_deg = 0;
  int32_t num_items = 0;
  std::vector<int32_t> h_rp;
  std::vector<int32_t> h_off;
  std::vector<Item> h_items;
  std::vector<int32_t> h_order;  // rows of every item in processing order
  // f_B kernels: chunk plan of long rows and their scratch
  bool hp_built = false;
  HeavyPlan hp{};
  int32_t* d_hp = nullptr;
  float* d_scratch = nullptr;
  size_t scratch_floats = 0;
  int sms = 152;
  // rows longer than 512 entries and their 512-entry chunks (counted once at
  // creation, for the allocation-free gradient's capacity check)
  int32_t long_rows = 0;
  int64_t long_chunks = 0;

  GraphDev dev() const {
    GraphDev g;
    g.n = (int32_t)n;
    g.num_graphs = G;
    g.nnz = nnz;
    g.row_ptr = d_rp;
    g.col = d_col;
    g.w = d_w;
    g.node_off = d_off;
    g.dmax = d_dmax;
    g.items = d_items;
    g.order = d_order;
    g.col16 = d_col16;
    g.num_items = num_items;
    return g;
  }
};

struct mqo_solver_s {
  mqo_graph g = nullptr;
  mqo_params p{};
  SolverDev S{};
  cudaStream_t user = nullptr;
  cudaStream_t work = nullptr;
  cudaEvent_t ev_in = nullptr, ev_out = nullptr;
  // second branch of a tick: the fused discrete kernel beside the step
  cudaStream_t work2 = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_join = nullptr;
  cudaGraphExec_t gx1 = nullptr, gx16 = nullptr;
  bool poisoned = false;
  size_t step_smem = 0;  // > 0: shared-memory step kernel with this much dynamic smem
  size_t disc_smem = 0;  // > 0: fused per-graph discrete kernel with this much dynamic smem
  bool rows_ok = false;      // the row-group step kernel is possible
  size_t step_smem_max = 0;  // smem the shared-memory step kernel needs (0: not possible)
  size_t disc_smem_max = 0;  // smem the fused discrete kernel needs (0: not possible)
  size_t disc_bits_max = 0;  // smem of its form on bit matrices (0: not possible)
  bool disc_bits = false;    // the current plan uses that form (disc_smem bytes)
  int64_t host_tick = 0;
  Counters* d_cnt_plain = nullptr;
  Counters* d_eval = nullptr;
  int32_t* h_pending = nullptr;  // pinned
  int32_t* d_pending = nullptr;
  int32_t* h_late = nullptr;  // pinned; set by a step kernel whose wait ran out
  // saved state around a standalone local search
  void* d_save = nullptr;
  std::vector<void*> allocs;
  size_t x_bytes = 0, v_bytes = 0, words = 0, pairs = 0;
  // staged-gather step kernel: device slice arrays per capacity (KB of
  // gathered rows of x), built on first use
  struct SliceSet {
    int cap_kb = 0;
    Slice* d = nullptr;
    int32_t count = 0, rows = 0, cols = 0;
  };
  std::vector<SliceSet> slice_sets;
  bool staged_ok = false;  // every row's neighbour rows fit the largest capacity
  // shared-memory step kernel with the sliced-ELL neighbour stream: device
  // arrays per layout (rows per warp, pitch of the staged x rows), built on
  // first use
  struct EllSet {
    int rpw = 0, pitch = 0;
    int4* d = nullptr;
    int2* pos = nullptr;
    bool ok = false;
  };
  std::vector<EllSet> ell_sets;
  bool ell_ok = false;           // the layout allows the ELL stream
  bool ell_only = false;         // the shared-memory kernel needs it (B < 32)
  bool step_ell = false;         // the current plan uses it
  const int4* ell = nullptr;     // its arrays for the current lane width
  const int2* ell_pos = nullptr;
  // tensor-core step kernel of dense member graphs
  bool dense_ok = false;         // the graph has bit matrices and the types allow it
  DensePlan dense_plan{};
  const DensePlan* dense = nullptr;  // the current plan uses it
  // many ticks of small member graphs in one launch (mqo_small.cu)
  size_t small_smem = 0;  // > 0: possible, with this much dynamic shared memory
  int small_threads = 0;
  bool small = false;     // the current plan uses it
  bool small_step = false;  // plain steps use it, whatever the plan of ticks
};

namespace {

template <typename T>
mqo_status dalloc(T** p, size_t count, std::vector<void*>* track) {
  void* q = nullptr;
  cudaError_t e = cudaMalloc(&q, std::max<size_t>(count, 1) * sizeof(T));
  if (e != cudaSuccess) cudaGetLastError();  // reported here, not by the next launch
  if (e != cudaSuccess) return fail(MQO_ENOMEM, "cudaMalloc(%zu bytes): %s", count * sizeof(T), cudaGetErrorString(e));
  *p = static_cast<T*>(q);
  if (track) track->push_back(q);
  return MQO_OK;
}

size_t dtype_size(int d) { return d == DT_F32 ? 4 : 2; }

// Slices of the staged-gather step kernel: walk every work item's rows in
// order and cut a slice before the row that would take it past `rows` rows
// or `cols` CSR entries.  False if one row alone has more than `cols` entries.
bool build_slices(const mqo_graph_s* g, int32_t rows, int32_t cols, std::vector<Slice>& out) {
  out.clear();
  for (int32_t it = 0; it < g->num_items; ++it) {
    const Item& item = g->h_items[(size_t)it];
    int32_t v0 = item.v0;
    while (v0 < item.v1) {
      int32_t v1 = v0;
      int64_t c = 0;
      while (v1 < item.v1 && v1 - v0 < rows) {
        const int64_t d = g->h_rp[(size_t)v1 + 1] - g->h_rp[(size_t)v1];
        if (d > cols) return false;
        if (c + d > cols) break;
        c += d;
        v1 += 1;
      }
      out.push_back(Slice{item.g, it, v0, v1, g->h_rp[(size_t)v0], g->h_rp[(size_t)v1], 0, 0});
      v0 = v1;
    }
  }
  return true;
}

// rows and CSR entries of one staged slice for `cap_kb` KB of gathered x rows
void slice_shape(int B, int x_dtype, int cap_kb, int32_t* rows, int32_t* cols) {
  const int rowx = B * (int)dtype_size(x_dtype);
  *cols = std::max(1, cap_kb * 1024 / rowx);
  *rows = std::min<int32_t>(128, std::max<int32_t>(8, *cols / 2));
}

// the staged kernel needs 16-byte multiples for a row of x and of V
bool staged_possible(int B, int x_dtype, int v_dtype) {
  return (B * (int)dtype_size(x_dtype)) % 16 == 0 && (B * (int)dtype_size(v_dtype)) % 16 == 0 && B <= 256 &&
         staged_vec_ok(B, x_dtype, default_staged_vec(B, x_dtype));
}

// Host checks of the CSR structure (sizes, row pointers): O(n).
mqo_status validate_structure(int64_t n, int64_t nnz, const int64_t* rp) {
  if (n < 1 || n >= (1LL << 31)) return fail(MQO_EINVAL, "n=%lld out of range [1, 2^31)", (long long)n);
  if (nnz < 0 || nnz >= (1LL << 31)) return fail(MQO_EINVAL, "nnz=%lld out of range [0, 2^31)", (long long)nnz);
  if (rp[0] != 0 || rp[n] != nnz) return fail(MQO_EGRAPH, "row_ptr[0] must be 0 and row_ptr[n] must be nnz");
  for (int64_t v = 0; v < n; ++v)
    if (rp[v + 1] < rp[v]) return fail(MQO_EGRAPH, "row_ptr decreases at row %lld", (long long)v);
  return MQO_OK;
}

// Host validation of the entries of rows [r0, r1) of symmetric CSR (see
// mqo_graph_create_csr): the message of the first bad entry of the smallest
// bad row.  Used for the whole graph when no GPU is present, and otherwise
// for the row the device check reports, to word the error.
mqo_status validate(int64_t n, int64_t nnz, const int64_t* rp, const int32_t* col, const int8_t* w,
                    const int64_t* offs, int32_t G, int64_t r0 = 0, int64_t r1 = -1) {
  mqo_status st0 = validate_structure(n, nnz, rp);
  if (st0 != MQO_OK) return st0;
  if (r1 < 0) r1 = n;
  std::vector<int32_t> graph_of;
  if (offs) {
    graph_of.resize((size_t)n);
    for (int32_t g = 0; g < G; ++g)
      for (int64_t v = offs[g]; v < offs[g + 1]; ++v) graph_of[(size_t)v] = g;
  }
  // rows are checked in parallel ranges; the reported error is the one of
  // the smallest row, as a sequential scan would find it
  struct Bad {
    int64_t row = -1;
    char msg[200] = {0};
  };
  auto check_rows = [&](int64_t v0, int64_t v1, Bad* bad) {
    for (int64_t v = v0; v < v1; ++v) {
      for (int64_t j = rp[v]; j < rp[v + 1]; ++j) {
        const int32_t u = col[j];
        const char* why = nullptr;
        char buf[200];
        if (u < 0 || u >= n) {
          snprintf(buf, sizeof(buf), "col_idx[%lld]=%d out of range", (long long)j, u);
          why = buf;
        } else if (u == v) {
          snprintf(buf, sizeof(buf), "self loop at node %lld", (long long)v);
          why = buf;
        } else if (j > rp[v] && col[j - 1] >= u) {
          snprintf(buf, sizeof(buf), "row %lld not strictly ascending at entry %lld", (long long)v, (long long)j);
          why = buf;
        } else if (w && w[j] != 1 && w[j] != -1) {
          snprintf(buf, sizeof(buf), "weight %d at entry %lld not in {-1,+1}", w[j], (long long)j);
          why = buf;
        } else if (offs && graph_of[(size_t)u] != graph_of[(size_t)v]) {
          snprintf(buf, sizeof(buf), "edge (%lld,%d) joins two member graphs", (long long)v, u);
          why = buf;
        } else {
          // symmetric: v in row u with the same weight
          const int32_t* b = col + rp[u];
          const int32_t* e = col + rp[u + 1];
          const int32_t* f = std::lower_bound(b, e, (int32_t)v);
          if (f == e || *f != v) {
            snprintf(buf, sizeof(buf), "edge (%lld,%d) has no reverse entry", (long long)v, u);
            why = buf;
          } else if (w && w[rp[u] + (f - b)] != w[j]) {
            snprintf(buf, sizeof(buf), "weight of (%lld,%d) is not symmetric", (long long)v, u);
            why = buf;
          }
        }
        if (why) {
          bad->row = v;
          snprintf(bad->msg, sizeof(bad->msg), "%s", why);
          return;
        }
      }
    }
  };
  const unsigned hw = std::thread::hardware_concurrency();
  const int64_t nr = r1 - r0;
  const int P = (int)std::max<int64_t>(1, std::min<int64_t>({(int64_t)(hw ? hw : 1), 32, nnz / 65536 + 1, nr}));
  std::vector<Bad> bad((size_t)P);
  std::vector<std::thread> pool;
  for (int p = 0; p < P; ++p) {
    const int64_t v0 = r0 + nr * p / P, v1 = r0 + nr * (p + 1) / P;
    if (p == P - 1) check_rows(v0, v1, &bad[(size_t)p]);
    else pool.emplace_back(check_rows, v0, v1, &bad[(size_t)p]);
  }
  for (auto& th : pool) th.join();
  for (const Bad& b : bad)
    if (b.row >= 0) return fail(MQO_EGRAPH, "%s", b.msg);
  return MQO_OK;
}

// Bit matrices of the member graphs (mqo_step_dense.cuh) where the step of
// dense member graphs may use them: no weights, degrees that fit the
// companion counts, an x block of 32 trajectories that fits in shared memory,
// and at least kDenseFill of the matrices' cells set.  They only make calls
// faster: where there is no memory for them the graph stays without.
mqo_status build_dense_bits(mqo_graph g, const std::vector<int32_t>& dmax, cudaStream_t stream) {
  for (int32_t k = 0; k < g->G; ++k) {
    g->max_ng = std::max(g->max_ng, g->h_off[(size_t)k + 1] - g->h_off[(size_t)k]);
    g->max_deg = std::max(g->max_deg, dmax[(size_t)k]);
  }
  if (g->d_w || g->nnz == 0 || g->max_deg > kDenseMaxDegree || dense_smem_bytes(g->max_ng) > kDenseSmemLimit)
    return MQO_OK;
  std::vector<int64_t> off((size_t)g->G);
  std::vector<int2> tiles;
  int64_t vecs = 0;
  for (int32_t k = 0; k < g->G; ++k) {
    const int64_t nt = (g->h_off[(size_t)k + 1] - g->h_off[(size_t)k] + 127) / 128;
    off[(size_t)k] = vecs;
    for (int64_t t = 0; t < nt; ++t) tiles.push_back(make_int2(k, (int)t));
    vecs += nt * nt * 128;
  }
  if ((double)g->nnz < kDenseFill * 128.0 * (double)vecs) return MQO_OK;
  int2* d_tiles = nullptr;
  mqo_status st = dalloc(&g->d_bits, (size_t)vecs, nullptr);
  if (st == MQO_OK) st = dalloc(&g->d_bits_off, (size_t)g->G, nullptr);
  if (st == MQO_OK) st = dalloc(&d_tiles, tiles.size(), nullptr);
  if (st != MQO_OK) {
    cudaFree(g->d_bits);
    cudaFree(g->d_bits_off);
    g->d_bits = nullptr;
    g->d_bits_off = nullptr;
    return MQO_OK;
  }
  cudaError_t e = cudaMemcpy(g->d_bits_off, off.data(), sizeof(int64_t) * off.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(d_tiles, tiles.data(), sizeof(int2) * tiles.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = launch_dense_bits(g->dev(), g->d_bits_off, d_tiles, (int)tiles.size(), g->d_bits, stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  cudaFree(d_tiles);
  if (e != cudaSuccess) return fail(MQO_ECUDA, "graph bit matrices: %s", cudaGetErrorString(e));
  return MQO_OK;
}

mqo_status build_graph(int32_t G, const int64_t* offs, int64_t n, int64_t nnz, const int64_t* rp_in,
                       const int32_t* col_in, const int8_t* w_in, int32_t is_dev, cudaStream_t stream,
                       mqo_graph* out) {
  if (!out || !rp_in || (nnz > 0 && !col_in)) return fail(MQO_EINVAL, "null pointer argument");
  *out = nullptr;
  std::vector<int64_t> rp_h;
  const int64_t* rp = rp_in;
  const int32_t* col = col_in;
  const int8_t* w = w_in;
  if (is_dev) {
    int nd = 0;
    if (cudaGetDeviceCount(&nd) != cudaSuccess || nd < 1) return fail(MQO_EINVAL, "device arrays need a GPU");
    // row pointers to the host (items, degree order); the entries are
    // copied device to device and checked on the device
    if (n < 1 || n >= (1LL << 31)) return fail(MQO_EINVAL, "n out of range");
    rp_h.resize((size_t)n + 1);
    CKG(cudaStreamSynchronize(stream));
    CKG(cudaMemcpy(rp_h.data(), rp_in, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToHost));
    rp = rp_h.data();
  }
  std::vector<int64_t> offs_own;
  if (!offs) {
    offs_own = {0, n};
    offs = offs_own.data();
    G = 1;
  } else {
    if (G < 1) return fail(MQO_EINVAL, "num_graphs must be >= 1");
    if (offs[0] != 0) return fail(MQO_EGRAPH, "node_offsets[0] must be 0");
    for (int32_t g = 0; g < G; ++g)
      if (offs[g + 1] <= offs[g]) return fail(MQO_EGRAPH, "member graph %d is empty", g);
    n = offs[G];
  }
  // With a GPU the entries are checked by a kernel after the upload (the
  // host checks only the structure); without one, on the host.
  int ndev = 0;
  const bool on_gpu = cudaGetDeviceCount(&ndev) == cudaSuccess && ndev > 0;
  if (!on_gpu) cudaGetLastError();  // clear the error of the query
  mqo_status st = on_gpu ? validate_structure(n, nnz, rp) : validate(n, nnz, rp, col, w, G > 1 ? offs : nullptr, G);
  if (st != MQO_OK) return st;

  auto* g = new mqo_graph_s();
  g->n = n;
  g->nnz = nnz;
  g->G = G;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&g->sms, cudaDevAttrMultiProcessorCount, dev);
  g->h_rp.resize((size_t)n + 1);
  for (int64_t v = 0; v <= n; ++v) g->h_rp[(size_t)v] = (int32_t)rp[v];
  for (int64_t v = 0; v < n; ++v) {
    const int64_t d = rp[v + 1] - rp[v];
    if (d > 512) {
      g->long_rows += 1;
      g->long_chunks += (d + 511) / 512;
    }
  }
  std::vector<int32_t> off32((size_t)G + 1), dmax((size_t)G, 0);
  std::vector<Item> items;
  for (int32_t k = 0; k <= G; ++k) off32[(size_t)k] = (int32_t)offs[k];
  for (int32_t k = 0; k < G; ++k) {
    for (int64_t v = offs[k]; v < offs[k + 1]; ++v)
      dmax[(size_t)k] = std::max<int32_t>(dmax[(size_t)k], (int32_t)(rp[v + 1] - rp[v]));
    for (int64_t v0 = offs[k]; v0 < offs[k + 1]; v0 += kChunkNodes) {
      Item it;
      it.g = k;
      it.v0 = (int32_t)v0;
      it.v1 = (int32_t)std::min<int64_t>(v0 + kChunkNodes, offs[k + 1]);
      it.pad = 0;
      items.push_back(it);
    }
  }
  // rows of every item by decreasing degree (ties by node id): rows that
  // walk their neighbour lists in lockstep then have nearly equal lengths
  std::vector<int32_t> order((size_t)n);
  {
    auto sort_items = [&](size_t i0, size_t i1) {
      for (size_t i = i0; i < i1; ++i) {
        const Item& it = items[i];
        int32_t* o = order.data() + it.v0;
        for (int32_t v = it.v0; v < it.v1; ++v) o[v - it.v0] = v;
        std::stable_sort(o, o + (it.v1 - it.v0),
                         [&](int32_t x, int32_t y) { return rp[x + 1] - rp[x] > rp[y + 1] - rp[y]; });
      }
    };
    const unsigned hw = std::thread::hardware_concurrency();
    const size_t P = std::max<size_t>(1, std::min<size_t>({(size_t)(hw ? hw : 1), 32, items.size() / 64 + 1}));
    std::vector<std::thread> th;
    for (size_t p = 1; p < P; ++p) th.emplace_back(sort_items, items.size() * p / P, items.size() * (p + 1) / P);
    sort_items(0, items.size() / P);
    for (auto& t : th) t.join();
  }
  g->num_items = (int32_t)items.size();
  g->h_items = items;
  g->h_off = off32;
  auto cleanup = [&](mqo_status s) {
    mqo_graph_destroy(g);
    return s;
  };
  if ((st = dalloc(&g->d_rp, (size_t)n + 1, nullptr)) != MQO_OK) return cleanup(st);
  if ((st = dalloc(&g->d_col, (size_t)nnz, nullptr)) != MQO_OK) return cleanup(st);
  if (w && (st = dalloc(&g->d_w, (size_t)nnz, nullptr)) != MQO_OK) return cleanup(st);
  if ((st = dalloc(&g->d_off, (size_t)G + 1, nullptr)) != MQO_OK) return cleanup(st);
  if ((st = dalloc(&g->d_dmax, (size_t)G, nullptr)) != MQO_OK) return cleanup(st);
  if ((st = dalloc(&g->d_items, items.size(), nullptr)) != MQO_OK) return cleanup(st);
  if ((st = dalloc(&g->d_order, (size_t)n, nullptr)) != MQO_OK) return cleanup(st);
  cudaError_t e = cudaSuccess;
  e = cudaMemcpy(g->d_rp, g->h_rp.data(), sizeof(int32_t) * (n + 1), cudaMemcpyHostToDevice);
  if (e == cudaSuccess && nnz) e = cudaMemcpy(g->d_col, col, sizeof(int32_t) * nnz, cudaMemcpyDefault);
  if (e == cudaSuccess && w && nnz) e = cudaMemcpy(g->d_w, w, nnz, cudaMemcpyDefault);
  if (e == cudaSuccess) e = cudaMemcpy(g->d_off, off32.data(), sizeof(int32_t) * (G + 1), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(g->d_dmax, dmax.data(), sizeof(int32_t) * G, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(g->d_items, items.data(), sizeof(Item) * items.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(g->d_order, order.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cleanup(fail(MQO_ECUDA, "graph upload: %s", cudaGetErrorString(e)));
  g->h_order = std::move(order);
  if (on_gpu && nnz > 0) {
    int32_t* d_bad = nullptr;
    if ((st = dalloc(&d_bad, 1, nullptr)) != MQO_OK) return cleanup(st);
    int32_t bad = (int32_t)n;
    e = cudaMemcpy(d_bad, &bad, sizeof(int32_t), cudaMemcpyHostToDevice);
    if (e == cudaSuccess)
      e = launch_validate_csr(g->d_rp, g->d_col, g->d_w, g->d_off, G, (int32_t)n, d_bad, g->sms, stream);
    if (e == cudaSuccess) e = cudaMemcpy(&bad, d_bad, sizeof(int32_t), cudaMemcpyDeviceToHost);
    cudaFree(d_bad);
    if (e != cudaSuccess) return cleanup(fail(MQO_ECUDA, "graph validation: %s", cudaGetErrorString(e)));
    if (bad < n) {
      // word the error from the host copy of the smallest bad row
      if (is_dev) {
        std::vector<int32_t> colh((size_t)nnz);
        std::vector<int8_t> wh(w ? (size_t)nnz : 0);
        cudaMemcpy(colh.data(), g->d_col, sizeof(int32_t) * nnz, cudaMemcpyDeviceToHost);
        if (w) cudaMemcpy(wh.data(), g->d_w, nnz, cudaMemcpyDeviceToHost);
        st = validate(n, nnz, rp, colh.data(), w ? wh.data() : nullptr, G > 1 ? offs : nullptr, G, bad, bad + 1);
      } else {
        st = validate(n, nnz, rp, col, w, G > 1 ? offs : nullptr, G, bad, bad + 1);
      }
      if (st == MQO_OK) st = fail(MQO_EGRAPH, "row %d failed validation", bad);
      return cleanup(st);
    }
  }
  // 16-bit member-local column indices for the shared-memory step kernel
  // when every member graph (and its zero dummy row) fits in them
  if (on_gpu && nnz > 0) {
    int32_t max_ng = 0;
    for (int32_t k = 0; k < G; ++k) max_ng = std::max<int32_t>(max_ng, off32[(size_t)k + 1] - off32[(size_t)k]);
    if (max_ng < 65535) {
      if ((st = dalloc(&g->d_col16, (size_t)nnz, nullptr)) != MQO_OK) return cleanup(st);
      e = launch_col16(g->dev(), g->d_col16, stream);
      if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
      if (e != cudaSuccess) return cleanup(fail(MQO_ECUDA, "graph upload: %s", cudaGetErrorString(e)));
    }
  }
  if (on_gpu && (st = build_dense_bits(g, dmax, stream)) != MQO_OK) return cleanup(st);
  *out = g;
  return MQO_OK;
}

mqo_status build_heavy_plan(mqo_graph g) {
  if (g->hp_built) return MQO_OK;
  std::vector<int32_t> light, hrow, hj0, hj1, hrows, hfirst;
  for (int64_t v = 0; v < g->n; ++v) {
    const int32_t a = g->h_rp[(size_t)v], b = g->h_rp[(size_t)v + 1];
    if (b - a <= kSplit) {
      light.push_back((int32_t)v);
    } else {
      hrows.push_back((int32_t)v);
      hfirst.push_back((int32_t)hrow.size());
      for (int32_t j = a; j < b; j += kSplit) {
        hrow.push_back((int32_t)v);
        hj0.push_back(j);
        hj1.push_back(std::min(j + kSplit, b));
      }
    }
  }
  hfirst.push_back((int32_t)hrow.size());
  // segments of consecutive light rows, cut before a heavy row or once a
  // segment holds kFbSegEntries entries
  std::vector<int32_t> segs;
  for (size_t c = 0; c < hrow.size(); ++c) {
    segs.push_back(hrow[c]);
    segs.push_back(-1 - (int32_t)c);
    segs.push_back(hj0[c]);
    segs.push_back(hj1[c]);
  }
  {
    int64_t r0 = -1;
    auto close = [&](int64_t r1) {
      if (r0 >= 0 && r1 > r0) {
        segs.push_back((int32_t)r0);
        segs.push_back((int32_t)r1);
        segs.push_back(g->h_rp[(size_t)r0]);
        segs.push_back(g->h_rp[(size_t)r1]);
      }
      r0 = -1;
    };
    for (int64_t v = 0; v < g->n; ++v) {
      const int32_t d = g->h_rp[(size_t)v + 1] - g->h_rp[(size_t)v];
      if (d > kSplit) {
        close(v);
        continue;
      }
      if (r0 < 0) r0 = v;
      if (g->h_rp[(size_t)v + 1] - g->h_rp[(size_t)r0] >= kFbSegEntries) close(v + 1);
    }
    close(g->n);
  }
  const size_t total = light.size() + 3 * hrow.size() + hrows.size() + hfirst.size() + segs.size() + 4;
  mqo_status st = dalloc(&g->d_hp, total, nullptr);
  if (st != MQO_OK) return st;
  int32_t* p = g->d_hp;
  auto put = [&](const std::vector<int32_t>& v) -> int32_t* {
    int32_t* q = p;
    if (!v.empty()) cudaMemcpy(q, v.data(), v.size() * sizeof(int32_t), cudaMemcpyHostToDevice);
    p += v.size();
    return q;
  };
  g->hp.light_rows = put(light);
  g->hp.num_light = (int32_t)light.size();
  g->hp.heavy_row = put(hrow);
  g->hp.heavy_j0 = put(hj0);
  g->hp.heavy_j1 = put(hj1);
  g->hp.num_chunks = (int32_t)hrow.size();
  g->hp.heavy_rows = put(hrows);
  g->hp.heavy_first = put(hfirst);
  g->hp.num_heavy = (int32_t)hrows.size();
  // the segment records are int4: start them on a 16-byte boundary
  while (((uintptr_t)p & 15u) != 0) ++p;
  g->hp.segs = reinterpret_cast<const int4*>(put(segs));
  g->hp.num_segs = (int32_t)(segs.size() / 4);
  CKG(cudaGetLastError());
  g->hp_built = true;
  return MQO_OK;
}

struct Scope {
  mqo_solver s;
  explicit Scope(mqo_solver s_) : s(s_) {
    cudaEventRecord(s->ev_in, s->user);
    cudaStreamWaitEvent(s->work, s->ev_in, 0);
  }
  ~Scope() {
    cudaEventRecord(s->ev_out, s->work);
    cudaStreamWaitEvent(s->user, s->ev_out, 0);
  }
};

mqo_status poison(mqo_solver s, cudaError_t e, const char* what) {
  s->poisoned = true;
  return fail(MQO_ECUDA, "%s: %s", what, cudaGetErrorString(e));
}

#define CKS(call)                                 \
  do {                                            \
    cudaError_t e_ = (call);                      \
    if (e_ != cudaSuccess) return poison(s, e_, #call); \
  } while (0)

// A wait of the step kernel ran out: the x and V it left are no step's.
mqo_status look_late(mqo_solver s) {
  if (!s->h_late || *static_cast<volatile int32_t*>(s->h_late) == 0) return MQO_OK;
  s->poisoned = true;
  return fail(MQO_ETIMEOUT, "a wait of the step kernel ran out");
}

// after the work the caller waits for
#define CHECK_LATE(s)                                  \
  do {                                                 \
    const mqo_status late_ = look_late(s);             \
    if (late_ != MQO_OK) return late_;                 \
  } while (0)

#define CHECK_SOLVER(s)                                                             \
  do {                                                                              \
    if (!(s)) return fail(MQO_EINVAL, "null solver");                               \
    if ((s)->poisoned) return fail(MQO_ESTATE, "solver poisoned by an earlier error"); \
    CHECK_LATE(s);                                                                  \
  } while (0)

// The staged kernel's slices for `cap_kb` KB of gathered x rows, built and
// uploaded on first use; count < 0 if some row has too many entries for it.
mqo_solver_s::SliceSet slice_set(mqo_solver s, int cap_kb) {
  for (const auto& ss : s->slice_sets)
    if (ss.cap_kb == cap_kb) return ss;
  mqo_solver_s::SliceSet ss;
  ss.cap_kb = cap_kb;
  slice_shape(s->S.B, s->S.p.x_dtype, cap_kb, &ss.rows, &ss.cols);
  std::vector<Slice> h;
  const size_t smem = staged_layout(s->S.B, (int)dtype_size(s->S.p.x_dtype), (int)dtype_size(s->S.p.v_dtype), ss.cols,
                                    ss.rows, true)
                          .total;
  if (smem > kStagedSmemLimit || !build_slices(s->g, ss.rows, ss.cols, h) || h.empty()) {
    ss.count = -1;
  } else if (dalloc(&ss.d, h.size(), &s->allocs) != MQO_OK ||
             cudaMemcpy(ss.d, h.data(), h.size() * sizeof(Slice), cudaMemcpyHostToDevice) != cudaSuccess) {
    ss.count = -1;
  } else {
    ss.count = (int32_t)h.size();
  }
  s->slice_sets.push_back(ss);
  return ss;
}

void use_slices(mqo_solver s, const mqo_solver_s::SliceSet& ss) {
  s->S.slices = ss.d;
  s->S.num_slices = ss.count;
  s->S.slice_rows = ss.rows;
  s->S.slice_cols = ss.cols;
}

int slice_kb(mqo_solver s) {
  for (const auto& ss : s->slice_sets)
    if (ss.d == s->S.slices && ss.count > 0) return ss.cap_kb;
  return 0;
}

// Rows per warp and pitch (bytes between staged rows of x) of the
// shared-memory step kernel: 2-byte x: 4 trajectories per lane, or 8 with wide
// lanes; rows of 64 bytes are stored with a 128-byte pitch; float32, and every type
// below 32 trajectories: 4, staged as float32.
void ell_shape(int B, int x_dtype, bool wide, int* rpw, int* pitch) {
  const int vec = wide && x_dtype != DT_F32 && B >= 32 ? 8 : 4;
  *rpw = 32 / (B / vec);
  *pitch = x_dtype == DT_F32 || B < 32 ? B * 4 : std::max(B * 2, 128);
}

// The sliced-ELL arrays for the current batch and lane width, built and
// uploaded on first use (ok = false if they could not be).  Group table on
// the host: the rows of every item in groups of rpw positions, each padded
// to the group's longest row rounded up to 4 entries; vectors on the device.
mqo_solver_s::EllSet ell_set(mqo_solver s, bool wide) {
  int rpw = 0, pitch = 0;
  ell_shape(s->S.B, s->S.p.x_dtype, wide, &rpw, &pitch);
  for (const auto& es : s->ell_sets)
    if (es.rpw == rpw && es.pitch == pitch) return es;
  const bool e16 = s->S.p.x_dtype == DT_F32 || s->S.B < 32;  // eight 16-bit entries per vector
  mqo_solver_s::EllSet es;
  es.rpw = rpw;
  es.pitch = pitch;
  const mqo_graph g = s->g;
  std::vector<int2> pos((size_t)g->n);
  int64_t total = 0;
  for (const Item& it : g->h_items)
    for (int32_t p0 = it.v0; p0 < it.v1; p0 += rpw) {
      const int32_t p1 = std::min<int32_t>(p0 + rpw, it.v1);
      int32_t dmax = 0;
      for (int32_t p = p0; p < p1; ++p) {
        const int32_t v = g->h_order[(size_t)p];
        dmax = std::max<int32_t>(dmax, g->h_rp[(size_t)v + 1] - g->h_rp[(size_t)v]);
      }
      const int32_t nvec = (dmax + 3) / 4;
      for (int32_t p = p0; p < p1; ++p) pos[(size_t)p] = make_int2((int32_t)std::min<int64_t>(total, INT32_MAX), nvec);
      total += (int64_t)(e16 ? (nvec + 1) / 2 : nvec) * rpw;
    }
  if (total < INT32_MAX && dalloc(&es.d, (size_t)total, &s->allocs) == MQO_OK &&
      dalloc(&es.pos, (size_t)g->n, &s->allocs) == MQO_OK &&
      cudaMemcpy(es.pos, pos.data(), sizeof(int2) * (size_t)g->n, cudaMemcpyHostToDevice) == cudaSuccess &&
      (e16 ? launch_ell_fill16 : launch_ell_fill)(g->dev(), rpw, pitch, es.pos, es.d, s->work) == cudaSuccess &&
      cudaStreamSynchronize(s->work) == cudaSuccess)
    es.ok = true;
  else
    cudaGetLastError();
  s->ell_sets.push_back(es);
  return es;
}

// Discrete rounds follow one another: descents are cut off after a few steps
// (MIS repairs each), or few of them lie between two local searches.
bool rounds_often(const mqo_params& p) {
  return (p.problem == PROB_MIS && p.repair && p.descent_cap < 20) ||
         (p.local_search && ((int64_t)p.t_gs + 1) * p.descent_cap < 300);
}

// Is a tick of the machine in the multi-tick kernel no slower than one of the
// tick's kernels?  Ticks with discrete rounds cost it more than steps do (a
// CTA walks all lists of its member graph), so where descents are short, so that
// rounds follow one another, and for MIS, whose capped descents are repaired,
// both times are estimated: us of a tick, the multi-tick kernel per wave of CTAs
// from the largest member graph's nodes, pairs and work, the tick's kernels
// from all pairs and work.  The coefficients are fitted to 1952 machine runs (14
// sizes and degrees, 1 to 300 graphs, B = 1 to 128, both problems, descents of 50
// steps and of 2 and 6; the plan taken is 0.5 % behind the better one on
// average).  Multi-tick against the tick's kernels, us: n = 200, degree 10, B = 1:
// 2.0 and 13; MIS, n = 100, degree 10, one graph: B = 16 7.4 and 13, B = 32 15.8 and
// 13.2 to 15.1, B = 64 33 and 14.7; n = 100, degree 4, B = 64, t_gs = 1, cap 6: 44 and 33.
bool tick_small_faster(mqo_solver s, const mqo_params& p, int pairs, int64_t work, int waves) {
  const mqo_graph g = s->g;
  const bool mis = p.problem == PROB_MIS, bits = g->d_bits != nullptr && p.batch >= 32;
  const bool rounds = rounds_often(p);
  if (!mis && !rounds) return true;
  struct Cost {
    double base, pair, work, node;                        // multi-tick kernel
    double kernels, all_narrow, all_wide, all_work, b, n, one;  // tick's kernels (narrow: B < 32; one: largest graph's pairs)
  };
  static const Cost kDescent[2] = {{1.5, 1.9e-3, 0.086e-3, 0, 14.5, 13.8e-6, 7.4e-6, 1.1e-6, 0.092, 0, 0},
                                   {0, 4.5e-3, 0.032e-3, 0, 14.7, 0, 12.8e-6, 0, 0.013, 0, 0.05e-3}};
  static const Cost kMis[2] = {{3.5, 6.3e-3, 0, 5.4e-3, 21.7, 59e-6, 15.8e-6, 0.1e-6, 0.04, 0, 0.5e-3},
                               {3.9, 3.9e-3, 0.025e-3, 8.1e-3, 27.5, 0, 33e-6, 0, 0.03, 0, 0}};
  static const Cost kCut[2] = {{3.0, 5.6e-3, 0.23e-3, 0, 21.2, 51e-6, 21e-6, 2.3e-6, 0.029, 0, 0.84e-3},
                               {8.7, 6.9e-3, 0.047e-3, 17e-3, 24.9, 0, 42e-6, 0, 0.027, 0.038, 0}};
  const Cost& c = (!rounds ? kDescent : mis ? kMis : kCut)[bits];
  const double n = g->max_ng, all = (double)g->n * p.batch, all_work = (double)g->nnz * p.batch;
  const bool narrow = p.batch < 32;
  const double small = waves * (c.base + c.pair * pairs + c.work * (double)work + c.node * n);
  const double ticks = c.kernels + (narrow ? c.all_narrow : c.all_wide) * all + (narrow ? c.all_work * all_work : 0.0) +
                       c.b * p.batch + c.n * n + c.one * pairs;
  return small <= ticks;
}

// selects the CSR (on = false) or the sliced-ELL stream for the current lane
// width; the CSR one when the ELL arrays are not available
void use_ell(mqo_solver s, bool on) {
  s->step_ell = false;
  s->ell = nullptr;
  s->ell_pos = nullptr;
  if (!on || !s->ell_ok || (s->S.p.x_dtype == DT_F32 && !s->S.step_wide)) return;  // float32: 16-byte lanes only
  const mqo_solver_s::EllSet es = ell_set(s, s->S.step_wide != 0);
  if (!es.ok) return;
  s->step_ell = true;
  s->ell = es.d;
  s->ell_pos = es.pos;
}

// MQO_SERIAL_TICK=1: the step and the discrete kernels one after the other
// (read at every enqueue, so that a test can compare the two orders)
bool serial_tick() {
  const char* e = getenv("MQO_SERIAL_TICK");
  return e && strcmp(e, "1") == 0;
}

// Do the plan's step and fused discrete kernel run one after the other?  A
// shared-memory step of one wave (a CTA on each SM) that starts beside the
// discrete kernel's CTAs finds their SMs taken and puts two of its own on
// others, which halves the step's speed where gathers bound it (16-byte lanes,
// float32); with rare rounds the discrete CTAs end at once and nothing is
// gained by the overlap.  Measured (us of a tick, beside and after; rounds
// rare, bit matrices): MaxCut, 75 graphs, n = 300, degree 60, float16: B = 64
// 71.2 and 47.5, B = 128 129.9 and 82.0; MIS, 76 graphs, n = 200, degree 36, B = 128
// 51.1 and 40.7; float32, 100 graphs, n = 120, degree 40, B = 128 65.7 and 43.8.
// 8-byte lanes 0.98 to 1.04, more items than SMs 0.94 to 1.06, rounds often
// 1.05 to 1.4: beside.
bool one_wave(mqo_solver s) {
  const mqo_graph g = s->g;
  const SolverDev& S = s->S;
  if (s->disc_smem == 0 || s->step_smem == 0 || s->dense || rounds_often(s->p)) return false;
  if (!S.step_wide && S.p.x_dtype != DT_F32) return false;
  const int disc = s->disc_bits ? disc_bits_ctas(S, g->sms) : g->G;
  return g->num_items <= g->sms && g->num_items + disc > g->sms;
}

// the discrete passes fused into one launch
cudaError_t launch_disc_fused(mqo_solver s, cudaStream_t stream) {
  if (s->disc_bits) return launch_disc_bits(s->S, s->g->d_bits, s->g->d_bits_off, s->disc_smem, s->g->sms, stream);
  return launch_disc_graph(s->S, s->disc_smem, stream);
}

cudaError_t enqueue_tick(mqo_solver s) {
  cudaError_t e;
  const SolverDev& S = s->S;
  const int G = S.g.num_graphs;
  if (S.K > 0) {  // pmQO: the graphs' pool decisions come first
    if ((e = launch_pool_ctrl(S, s->work)) != cudaSuccess) return e;
    if ((e = launch_pool_apply(S, s->work)) != cudaSuccess) return e;
  }
  if ((e = launch_ctrl(S, CTRL_MACHINE, nullptr, s->work)) != cudaSuccess) return e;
  if ((e = launch_apply(S, s->work)) != cudaSuccess) return e;
  if (s->work2 && !serial_tick() && !one_wave(s)) {
    // The step (x, V, rounding words; counters of stepping trajectories) and
    // the discrete passes (work, auxiliary, free and drop bit sets and the
    // move arrays; counters of trajectories in a round, integer atomics)
    // touch disjoint state and both follow k_apply: two branches, so that
    // step CTAs fill the SMs the discrete kernels leave idle.
    if ((e = cudaEventRecord(s->ev_fork, s->work)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(s->work2, s->ev_fork, 0)) != cudaSuccess) return e;
    if (s->disc_smem > 0) {
      if ((e = launch_disc_fused(s, s->work2)) != cudaSuccess) return e;
    } else {
      for (int pass = 0; pass < 3; ++pass)
        if ((e = launch_disc(S, pass, s->work2)) != cudaSuccess) return e;
    }
    if ((e = launch_step(S, S.cnt, S.act, S.gflag + 2 * G, s->step_smem, s->work, s->ell, s->ell_pos, s->dense, s->g->sms)) != cudaSuccess)
      return e;
    if ((e = cudaEventRecord(s->ev_join, s->work2)) != cudaSuccess) return e;
    if ((e = cudaStreamWaitEvent(s->work, s->ev_join, 0)) != cudaSuccess) return e;
    return launch_tick_end(S, s->work);
  }
  if ((e = launch_step(S, S.cnt, S.act, S.gflag + 2 * G, s->step_smem, s->work, s->ell, s->ell_pos, s->dense, s->g->sms)) != cudaSuccess) return e;
  if (s->disc_smem > 0) {
    if ((e = launch_disc_fused(s, s->work)) != cudaSuccess) return e;
  } else {
    for (int pass = 0; pass < 3; ++pass)
      if ((e = launch_disc(S, pass, s->work)) != cudaSuccess) return e;
  }
  return launch_tick_end(S, s->work);
}

cudaError_t enqueue_ls_tick(mqo_solver s, int mode) {
  cudaError_t e;
  const SolverDev& S = s->S;
  if ((e = launch_ctrl(S, mode, nullptr, s->work)) != cudaSuccess) return e;
  if ((e = launch_apply(S, s->work)) != cudaSuccess) return e;
  if (s->disc_smem > 0) {
    if ((e = launch_disc_fused(s, s->work)) != cudaSuccess) return e;
  } else {
    for (int pass = 0; pass < 3; ++pass)
      if ((e = launch_disc(S, pass, s->work)) != cudaSuccess) return e;
  }
  return launch_tick_end(S, s->work);
}

cudaError_t capture(mqo_solver s, int ticks, cudaGraphExec_t* out) {
  cudaGraph_t graph = nullptr;
  cudaError_t e = cudaStreamBeginCapture(s->work, cudaStreamCaptureModeThreadLocal);
  if (e != cudaSuccess) return e;
  cudaError_t ek = cudaSuccess;
  for (int i = 0; i < ticks && ek == cudaSuccess; ++i) ek = enqueue_tick(s);
  e = cudaStreamEndCapture(s->work, &graph);
  if (ek != cudaSuccess) {
    if (graph) cudaGraphDestroy(graph);
    return ek;
  }
  if (e != cudaSuccess) return e;
  e = cudaGraphInstantiate(out, graph, 0);
  cudaGraphDestroy(graph);
  return e;
}

}  // namespace

void graph_csr_view(mqo_graph_s* g, GraphCsrView* out) {
  out->row_ptr = g->d_rp;
  out->col = g->d_col;
  out->w = g->d_w;
  out->n = (int32_t)g->n;
  out->long_rows = g->long_rows;
  out->long_chunks = g->long_chunks;
  out->sms = g->sms;
}

mqo_status set_last_error(mqo_status status, const char* msg) {
  g_err = msg;
  return status;
}

extern "C" {

const char* mqo_last_error(void) { return g_err.c_str(); }

const char* mqo_version(void) { return "mqo-gb300 0.1 (sm_103a)"; }

mqo_status mqo_graph_create_csr(int64_t n, int64_t nnz, const int64_t* row_ptr, const int32_t* col_idx,
                                const int8_t* weights, int32_t is_device_ptr, void* cuda_stream, mqo_graph* out) {
  return build_graph(1, nullptr, n, nnz, row_ptr, col_idx, weights, is_device_ptr, (cudaStream_t)cuda_stream, out);
}

mqo_status mqo_graph_create_packed(int32_t num_graphs, const int64_t* node_offsets, int64_t nnz,
                                   const int64_t* row_ptr, const int32_t* col_idx, const int8_t* weights,
                                   int32_t is_device_ptr, void* cuda_stream, mqo_graph* out) {
  if (!node_offsets) return fail(MQO_EINVAL, "null node_offsets");
  if (num_graphs < 1) return fail(MQO_EINVAL, "num_graphs must be >= 1");
  std::vector<int64_t> offs(node_offsets, node_offsets + num_graphs + 1);
  return build_graph(num_graphs, offs.data(), offs.back(), nnz, row_ptr, col_idx, weights, is_device_ptr,
                     (cudaStream_t)cuda_stream, out);
}

mqo_status mqo_graph_destroy(mqo_graph g) {
  if (!g) return MQO_OK;
  cudaFree(g->d_rp);
  cudaFree(g->d_col);
  cudaFree(g->d_w);
  cudaFree(g->d_off);
  cudaFree(g->d_dmax);
  cudaFree(g->d_items);
  cudaFree(g->d_order);
  cudaFree(g->d_col16);
  cudaFree(g->d_bits);
  cudaFree(g->d_bits_off);
  cudaFree(g->d_hp);
  cudaFree(g->d_scratch);
  delete g;
  return MQO_OK;
}

mqo_status mqo_graph_info(mqo_graph g, int64_t* n, int64_t* nnz, int32_t* num_graphs) {
  if (!g) return fail(MQO_EINVAL, "null graph");
  if (n) *n = g->n;
  if (nnz) *nnz = g->nnz;
  if (num_graphs) *num_graphs = g->G;
  return MQO_OK;
}

mqo_status mqo_solver_create(mqo_graph g, const mqo_params* p, void* cuda_stream, mqo_solver* out) {
  if (!g || !p || !out) return fail(MQO_EINVAL, "null argument");
  *out = nullptr;
  const int B = p->batch;
  if (B < 1 || B > 128 || (B & (B - 1))) return fail(MQO_EINVAL, "batch=%d must be a power of two in [1,128]", B);
  if (p->problem != MQO_MIS && p->problem != MQO_MAXCUT) return fail(MQO_EINVAL, "unknown problem %d", p->problem);
  if (p->problem == MQO_MIS && g->d_w) return fail(MQO_EINVAL, "MIS needs an unweighted graph");
  if (p->problem == MQO_MIS && !(p->gamma > 1.0f)) return fail(MQO_EINVAL, "gamma must be > 1");
  if (p->problem == MQO_MAXCUT && !(p->lambda_ > 0.0f && p->lambda_ < 2.0f))
    return fail(MQO_EINVAL, "lambda must lie in (0,2)");
  if (p->x_dtype < 0 || p->x_dtype > 2) return fail(MQO_EINVAL, "bad x_dtype");
  if (!(p->v_dtype == MQO_F32 || p->v_dtype == p->x_dtype)) return fail(MQO_EINVAL, "v_dtype must be F32 or x_dtype");
  if (p->descent_cap < 1) return fail(MQO_EINVAL, "descent_cap must be >= 1");
  if (p->t_gs < 0) return fail(MQO_EINVAL, "t_gs must be >= 0");
  if (!(p->rho >= 0.0 && p->rho < 1.0)) return fail(MQO_EINVAL, "rho must lie in [0,1)");
  if (p->init_kind != 0 && p->init_kind != 1) return fail(MQO_EINVAL, "init_kind must be 0 or 1");
  if (p->objective < MQO_OBJ_FB || p->objective > MQO_OBJ_FA) return fail(MQO_EINVAL, "unknown objective %d", p->objective);
  if (p->problem == MQO_MIS && p->objective != MQO_OBJ_FB) return fail(MQO_EINVAL, "objective applies to MaxCut only");
  if (p->pool_k < 0 || p->pool_k > kPoolMax) return fail(MQO_EINVAL, "pool_k=%d must lie in [0,%d]", p->pool_k, kPoolMax);

  auto* s = new mqo_solver_s();
  s->g = g;
  s->p = *p;
  s->user = (cudaStream_t)cuda_stream;
  auto bail = [&](mqo_status st) {
    mqo_solver_destroy(s);
    return st;
  };
  if (cudaStreamCreateWithFlags(&s->work, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&s->ev_in, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&s->ev_out, cudaEventDisableTiming) != cudaSuccess ||
      cudaStreamCreateWithFlags(&s->work2, cudaStreamNonBlocking) != cudaSuccess ||
      cudaEventCreateWithFlags(&s->ev_fork, cudaEventDisableTiming) != cudaSuccess ||
      cudaEventCreateWithFlags(&s->ev_join, cudaEventDisableTiming) != cudaSuccess)
    return bail(fail(MQO_ECUDA, "stream/event creation failed"));
  SolverDev& S = s->S;
  S.g = g->dev();
  S.p.problem = p->problem;
  S.p.B = B;
  S.p.x_dtype = p->x_dtype;
  S.p.v_dtype = p->v_dtype;
  S.p.alpha = p->alpha;
  S.p.momentum = p->momentum;
  S.p.gamma = p->gamma;
  S.p.lambda_ = p->lambda_;
  S.p.rho = p->rho;
  S.p.sigma = p->sigma;
  S.p.t_gs = p->t_gs;
  S.p.cap = p->descent_cap;
  S.p.init_kind = p->init_kind;
  S.p.local_search = p->local_search;
  S.p.repair = p->repair;
  S.p.seed = p->seed;
  S.p.objective = p->objective;
  S.p.pool_k = p->pool_k;
  S.B = B;
  S.Bw = (B + 31) / 32;
  const int64_t n = g->n, T = (int64_t)g->G * B;
  s->pairs = (size_t)n * B;
  s->words = (size_t)n * S.Bw;
  s->x_bytes = s->pairs * dtype_size(p->x_dtype);
  s->v_bytes = s->pairs * dtype_size(p->v_dtype);
  mqo_status st;
  char *x0, *x1, *vv;
  if ((st = dalloc(&x0, s->x_bytes, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&x1, s->x_bytes, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&vv, s->v_bytes, &s->allocs)) != MQO_OK) return bail(st);
  S.X0 = x0;
  S.X1 = x1;
  S.V = vv;
  uint32_t** wbufs[] = {&S.ZX0, &S.ZX1, &S.Zbest, &S.Zwork, &S.Zaux, &S.Zfree, &S.Zdrop};
  for (auto pp : wbufs)
    if ((st = dalloc(pp, s->words, &s->allocs)) != MQO_OK) return bail(st);
  int32_t** ibufs[] = {&S.owner, &S.pa, &S.pb, &S.gain};
  for (auto pp : ibufs)
    if ((st = dalloc(pp, s->pairs, &s->allocs)) != MQO_OK) return bail(st);
  // counter replicas: enough that one replica sees at most ~8 items of a graph
  {
    int max_items = 1, max_ng = 1;
    std::vector<int32_t> per(g->G, 0);
    for (const Item& it : g->h_items) per[it.g] += 1;
    for (int32_t k = 0; k < g->G; ++k) max_items = std::max(max_items, per[k]);
    for (int32_t k = 0; k < g->G; ++k) max_ng = std::max(max_ng, g->h_off[k + 1] - g->h_off[k]);
    int R = 1;
    while (R < 64 && R * 8 < max_items) R *= 2;
    S.R = R;
    const size_t need = step_smem_bytes(B, p->x_dtype, p->problem, max_ng);
    // Default step kernel: the shared-memory one when every member graph's
    // block of x fits, else the staged-gather one when its slices fit, else
    // the plain global-memory one.  MQO_STEP_KERNEL=generic | staged selects
    // either global-memory kernel even when the member graphs fit in shared
    // memory (staged: where possible).
    const char* force = getenv("MQO_STEP_KERNEL");
    const bool generic = force && strcmp(force, "generic") == 0;
    const bool staged = force && strcmp(force, "staged") == 0;
    const bool ell_plain = p->problem == PROB_MIS || g->d_w == nullptr;
    s->ell_only = (B == 4 || B == 8 || B == 16) && ell_plain;
    s->step_smem_max = ((B >= 32 || s->ell_only) && need <= kStepSmemLimit) ? need : 0;
    s->step_smem = (generic || staged || (s->ell_only && force)) ? 0 : s->step_smem_max;
    if (staged_possible(B, p->x_dtype, p->v_dtype)) {
      // the smallest slice capacity from the default up that holds every row
      for (int kb = kDefaultSliceKB; kb <= 128 && !s->staged_ok; kb *= 2) {
        const mqo_solver_s::SliceSet ss = slice_set(s, kb);
        if (ss.count > 0) {
          s->staged_ok = true;
          use_slices(s, ss);
        }
      }
    }
    s->S.step_staged = (s->staged_ok && !generic) ? 1 : 0;
    // 16-bit column indices in the shared-memory step kernel where the graph
    // has them (MQO_COL16=0: the 32-bit ones)
    const char* c16 = getenv("MQO_COL16");
    s->S.step_c16 = g->d_col16 != nullptr && !(c16 && strcmp(c16, "0") == 0) ? 1 : 0;
    // MQO_STEP_KERNEL=wide: the shared-memory kernel with 16-byte lanes
    s->S.step_wide = force && strcmp(force, "wide") == 0 && step_wide_possible(B, p->x_dtype) ? 1 : 0;
    // the sliced-ELL neighbour stream of the shared-memory kernel where the
    // layout allows it (MIS: bfloat16 or float32 x; MaxCut: no weights; float32:
    // B <= 64, from B = 4, where below 32 there is no CSR form); MQO_STEP_ELL=0: the
    // CSR arrays.
    s->ell_ok = s->step_smem_max > 0 &&
                (s->ell_only || ((B == 32 || B == 64 || (B == 128 && p->x_dtype != DT_F32)) &&
                                 (p->problem == PROB_MIS ? p->x_dtype != DT_F16 : g->d_w == nullptr)));
    // Default: 16-byte lanes with the ELL stream (the fewest instructions
    // per gathered byte).  MQO_STEP_ELL=1: the ELL stream with the lanes
    // MQO_STEP_KERNEL selects (8-byte unless "wide"); MQO_STEP_KERNEL=wide
    // alone keeps the CSR indices.
    const char* ellv = getenv("MQO_STEP_ELL");
    const bool ell_forced = ellv && strcmp(ellv, "1") == 0;
    const bool ell_off = ellv && strcmp(ellv, "0") == 0;
    if (!ellv && !force && s->ell_ok && step_wide_possible(B, p->x_dtype)) s->S.step_wide = 1;
    if (s->ell_only) s->S.step_wide = 1;
    // Dense member graphs: the tensor-core kernel, unless an environment
    // variable above selects one of the others (MQO_STEP_KERNEL=dense: this
    // one where possible).  Its time grows with n per row, theirs with the
    // degree, and it works in row tiles of 128 times groups of 32 trajectories,
    // which have to fill the GPU.  Measured (BF16, us of a step among 8 or 64 graphs
    // after some ticks, other kernel in brackets):
    //  * MIS against the shared-memory kernel from a mean degree of 32 + n / 20
    //    (n = 400, 64 graphs, B = 32, degree 48: 19.5 (20.6); n = 800, degree 64: 28.5
    //    (28.9), degree 96: 28.8 (33.4)), with fewer tiles than SMs from 38 + n / 18
    //    (ticks, 16 graphs: n = 600, degree 64 1.13 of the other's time, 100: 0.9);
    //  * MIS where x does not fit there, against the staged and row-group kernels,
    //    from 16 + n / 25 (64 graphs, B = 128: n = 600, degree 48: 51 (99); n = 800: 76
    //    (132); B = 32, n = 1000, degree 64: 37 (61)); below the line it would win too
    //    at n = 1200 and 1400, degree 64 (B = 128: 142 (293) and 173 (300));
    //  * with few tiles from 32 + n / 20 up, by 14 / tiles higher below 100 tiles, and
    //    not below 24 (ticks, one graph: n = 1000, degree 100, B = 32 1.56 of the
    //    staged kernel's time, B = 128 1.02; n = 850, 4 graphs, degree 110 1.20, 160 1.08);
    //  * MaxCut meets x inside the box for longer, whose rows it sums in CSR order:
    //    against the shared-memory kernel from 48 + n / 16 (64 graphs, B = 32: n = 600,
    //    degree 96: 38.5 (57); ticks 0.8 and late ones 0.6 of the other's time; plain
    //    steps from x all over the box 1.05 to 1.4), not for the smallest graphs at
    //    B = 32 (n = 160: 1.2); else from 16 + n / 25 (B = 128, n = 800, degree 48: 114
    //    (146), n = 1000, degree 64: 189 (181), n = 1700, degree 96: 392 (480); float16
    //    676 (505)), with few tiles as below (ticks, one graph, B = 32: n = 1000, degree
    //    200 2.3 of the staged kernel's time, B = 128, n = 800, degree 110 1.5, 160 0.95).
    s->dense_ok = g->d_bits != nullptr && p->x_dtype != DT_F32 && B % kDenseGroup == 0;
    if (s->dense_ok) {
      s->dense_plan.bits = g->d_bits;
      s->dense_plan.bits_off = g->d_bits_off;
      s->dense_plan.smem = dense_smem_bytes(g->max_ng);
      int bits = 1;
      while ((1 << bits) <= g->max_deg) ++bits;
      s->dense_plan.sum_bits = bits;
      // a CTA works two row tiles at a time; a graph's tiles go to more CTAs
      // until there are about three waves of them (2 CTAs per SM), which evens
      // out the last wave (512 graphs of 6 tiles: 2 parts 147 us a tick, 1 part
      // 151, 3 parts, each staging x again, 155)
      const int pairs = (dense_tiles(g->max_ng) + 1) / 2;
      const int ctas = g->G * (B / kDenseGroup);
      s->dense_plan.parts = std::max(1, std::min(pairs, (6 * g->sms + ctas - 1) / ctas));
      const double degree = (double)g->nnz / (double)g->n, n = g->max_ng;
      const int64_t tiles = (int64_t)ctas * dense_tiles(g->max_ng);
      const bool fills = tiles >= g->sms, smem = s->step_smem_max > 0;
      // 11-bit significands leave fewer sums exact: MaxCut in float16 stays with the
      // shared-memory kernel (407 graphs, n = 164, degree 46, B = 128: 164 us a tick
      // against 142)
      const bool cut = p->problem == PROB_MAXCUT;
      double from;
      if (smem && cut) from = n <= 256 && B == 32 ? 1e9 : 48.0 + n / 16.0;
      else if (smem) from = fills ? 32.0 + n / 20.0 : 38.0 + n / 18.0;
      else if (fills) from = 16.0 + n / 25.0;
      else if (cut) from = tiles < 28 ? 1e9 : std::max(48.0 + n / 16.0, tiles < 76 ? 0.18 * n : 0.0);
      else from = tiles < 24 ? 1e9 : (32.0 + n / 20.0) * (tiles < 100 ? 1.0 + 14.0 / (double)tiles : 1.0);
      const bool few_exact = cut && p->x_dtype == DT_F16 && smem;
      if ((!force && !ellv && !c16 && degree >= from && !few_exact) || (force && strcmp(force, "dense") == 0))
        s->dense = &s->dense_plan;
    }
    // Small member graphs: the multi-tick kernel, unless an environment
    // variable selects one of the tick's kernels (MQO_TICK_KERNEL=ticks: never,
    // small: wherever it is possible).
    {
      int64_t work = 0;
      int pairs = 0;
      size_t smem = 0;
      for (int32_t k = 0; k < g->G; ++k) {
        const int32_t ng = g->h_off[k + 1] - g->h_off[k];
        const int32_t nz = g->h_rp[(size_t)g->h_off[k + 1]] - g->h_rp[(size_t)g->h_off[k]];
        work = std::max(work, (int64_t)nz * B);
        pairs = (int)std::max<int64_t>(pairs, std::min<int64_t>((int64_t)ng * B, 1 << 20));
        if (ng >= 65536 || (int64_t)ng * B > (1 << 20)) smem = SIZE_MAX;
        else smem = std::max(smem, small_smem_bytes(B, p->x_dtype, p->v_dtype, ng, nz, g->d_w != nullptr));
      }
      if (p->pool_k == 0 && S.R == 1 && smem <= kSmallSmemLimit) {
        s->small_smem = smem;
        s->small_threads = std::min(1024, std::max(128, (pairs + 127) / 128 * 128));
        const char* tk = getenv("MQO_TICK_KERNEL");
        const bool other = force || ellv || c16 || getenv("MQO_DISC_KERNEL") || getenv("MQO_SERIAL_TICK");
        // A plain step takes about 0.8 us, 0.8 ns per (node, trajectory) pair and
        // 0.06 ns per (entry, trajectory) pair of the largest member graph, and
        // there is one CTA per SM; a step of the kernels takes 11 us and up (n = 200,
        // B = 1: 1.0 against 11.7; n = 400, degree 24, B = 8: 8.3 against 12.8;
        // n = 200, degree 24, B = 32: 12.9 against 19.5, 300 graphs 26 against 28;
        // n = 400, degree 24, B = 32: 25 against 21).
        const double us = 0.8 + 0.8e-3 * pairs + 0.06e-3 * (double)work;
        const int waves = (g->G + g->sms - 1) / g->sms;
        const bool faster = us <= 11.0 && us * waves <= 22.0;
        s->small_step = tk ? strcmp(tk, "small") == 0 : !other && faster;
        s->small = s->small_step && (tk || tick_small_faster(s, *p, pairs, work, waves));
      }
    }
    // 16-bit x, MIS or MaxCut on f_B: the row-group kernel, unless an environment
    // variable selects one of the others (MQO_STEP_KERNEL=rows: this one where
    // possible).  A row's neighbours are read a few at a time, so the longest row
    // is a chain of L2 latencies (about 0.15 us per entry beyond what the staged
    // kernel takes), to be covered by the time of the whole step at about 5 TB/s of
    // L2 reads.  Measured, rows against staged: n = 10^4, degree 20 (longest 40),
    // B = 32 23.7 us against 19.7, B = 64 23.6 against 25.5, B = 128 29 against 36;
    // n = 5 10^4, longest row 864, B = 32: 227 against 30.  Rows of 64 bytes from an
    // x far larger than L2 wait for DRAM, which the staged kernel's deeper queue
    // serves better (10^7 nodes, B = 32: 3.25 ms against 3.42; 4 10^6: the same).
    s->rows_ok = step_rows_possible(B, p->x_dtype, p->problem, p->objective, g->max_deg);
    const bool none_forced = !force && !ellv && !c16;
    {
      const bool covered = (double)(g->nnz + 4 * g->n) * B >= 375e3 * g->max_deg;
      const bool dram = B == 32 && g->n * B * 2 > 2 * kL2Bytes && p->v_dtype != DT_F32;
      bool rows = s->rows_ok && covered && !dram;
      if (none_forced && s->step_smem > 0) {
        // Member graphs that fit in shared memory: that kernel runs one CTA per item
        // and leaves the GPU idle below about a third as many items as SMs (n = 300,
        // degree 20, B = 128, MIS: 8 items 34 us against 15 of the staged kernel, 32
        // items 35 against 23, 100 items 35 against 41), but not where an item has
        // little to gather (us of a tick with a pool, BF16, MIS: 33 items of 60 nodes,
        // degree 10, B = 32: 21.5 of the staged kernel against 18.2; 48 items of 30,
        // degree 4, B = 128: 23.2 against 20.2; 16 items of 60, degree 10, B = 32: 19.3
        // against 17.1, MaxCut 17.8 and 18.2), nor with float32 x and many long rows (48
        // items of 250, degree 30, B = 64: 44 against 30; of 60, B = 128: 33.5 against
        // 26.6).  MaxCut's longer tail moves its line against the row groups.  They share
        // all rows out over the GPU, so their time grows with items and degree, the
        // other's with the degree alone.  Row
        // groups against shared memory, us of a plain step (BF16, n = 400): 72 items,
        // B = 32, degree 48: 29.6 and 30.0, degree 96: 42 and 38.5; B = 64, degree 96:
        // 45 and 61; 100 items, B = 64, degree 96: 65 and 61; B = 128, degree 96: 92 and
        // 108; 128 items, B = 32, degree 16: 23.6 and 23.8, degree 96: 48 and 38.5;
        // B = 128, degree 32: 59 and 62, degree 64: 94 and 86.  At a mean degree of 8 they
        // win with many items too (1000 items of 250 nodes, B = 128: 0.83 of the time;
        // 300 items, B = 32: 1.02).
        const int items = (int)g->h_items.size();
        const double degree = (double)g->nnz / (double)g->n, load = (double)items / g->sms;
        const bool f32 = p->x_dtype == DT_F32;
        const bool mis = p->problem == PROB_MIS;
        const double least = items <= 32 || B < 32 ? (!mis || (B != 32 && B != 64) ? 0.0 : B == 64 ? 20e3 : 28e3)
                                         : (B == 32 ? (mis ? 50e3 : 30e3) : B == 64 ? 28e3 : f32 ? 0.0 : 31e3);
        const double gathered = (double)g->nnz * B / items;
        const bool long_rows = f32 && B >= 32 && items > 32 &&
                               (B < 128 ? items * degree > 900.0 : items * degree > 1300.0 && gathered < 300e3);
        const bool few = 3 * items < g->sms && (s->staged_ok || rows) && gathered >= least && !long_rows;
        const double most = load < 0.5    ? (B == 32 ? 48.0 : 1e9)
                            : load < 0.75 ? (B == 32 ? 32.0 : B == 64 ? 48.0 : 1e9)
                                          : B / 4.0;
        const bool cut = !mis && rows && ((items < g->sms && degree <= most) || degree <= 8.0);
        if (few || cut) s->step_smem = 0;
        else rows = false;
      }
      if ((none_forced && rows && !s->dense) || (s->rows_ok && force && strcmp(force, "rows") == 0)) {
        s->step_smem = 0;
        s->S.step_staged = 2;
      }
      // float32 x: the staged kernel copies every neighbour row through shared
      // memory, where 512-byte rows leave a slice few of them, and long steps wait
      // for the copies' issue; the global-memory kernel reads the rows from L2.  Measured
      // (staged against global, us): B = 128: 10^4 nodes, degree 10 (51 MB of neighbour
      // rows) 31 and 31, degree 40 123 and 58, 10^6 nodes, degree 12 2636 and 1889;
      // B = 64: 3 10^4 nodes, degree 20 (154 MB) 61 and 74, 10^5, degree 30 (769 MB) 271
      // and 198; B = 32: 10^5, degree 30 (384 MB) 133 and 117; x of 128 MB and more
      // 688 and 854.
      const double gathered = (double)g->nnz * B * 4;
      const bool direct = (B == 128 && gathered >= 50e6) ||
                          ((B == 32 || B == 64) && gathered >= 300e6 && g->n * B * 4 <= kL2Bytes / 2);
      if (none_forced && p->x_dtype == DT_F32 && s->S.step_staged == 1 && covered && direct) s->S.step_staged = 0;
    }
    if (s->step_smem > 0 && !s->dense) use_ell(s, ell_forced || (!ell_off && !force));
    if (s->ell_only && !s->step_ell) {  // switched off, or its arrays could not be built
      if (!ell_off && s->step_smem > 0) s->step_smem_max = 0;
      s->step_smem = 0;
    }
    // The fused per-graph discrete kernel runs one CTA per member graph, so
    // it is the default only with at least half as many member graphs as
    // SMs; with fewer, the node-parallel passes (several CTAs per item) fill
    // the GPU.  MQO_DISC_KERNEL=pairs | graph forces either when possible.
    const char* dforce = getenv("MQO_DISC_KERNEL");
    const bool pairs = dforce && strcmp(dforce, "pairs") == 0;
    const bool fused = dforce && strcmp(dforce, "graph") == 0;
    const size_t dneed = disc_graph_smem_bytes(B, max_ng);
    const bool few = 2 * g->G < g->sms;
    s->disc_smem_max = (B >= 32 && dneed <= kDiscSmemLimit && (!few || fused)) ? dneed : 0;
    s->disc_smem = pairs ? 0 : s->disc_smem_max;
    // Member graphs with bit matrices: the form that follows the trajectories in
    // a round (MQO_DISC_KERNEL=bits where possible; the others exclude it).  Where
    // rounds follow one another most trajectories are in one, which the lists serve
    // a word at a time.  Measured (us of a tick, descents of 6 steps, bits against
    // the fused lists): MIS, 152 graphs, B = 64: n = 100, degree 10 66 and 41, degree 30
    // 56 and 40, n = 200, degree 36 78 and 63, degree 80 1.0 of the other's time, n = 400,
    // degree 30 up to 1.3, MaxCut 0.3 to 1.2 of it; against the node-parallel lists:
    // one graph, B = 32: n = 800, degree 120 60 and 48, MaxCut 102 and 45, n = 1200,
    // degree 200 104 and 64, 178 and 59; n = 400 and below 0.2 to 1.3 of it.
    const double degree = (double)g->nnz / (double)g->n;
    const bool mis = p->problem == PROB_MIS;
    const bool lists = rounds_often(*p) && (few ? max_ng >= 700 && g->G <= 16 && (B == 32 || (B == 64 && !mis && degree >= 100.0))
                                                : mis && s->disc_smem_max > 0 && degree < 48.0);
    s->disc_bits_max = g->d_bits != nullptr && B >= 32 ? disc_bits_smem_bytes(p->problem, max_ng) : 0;
    if (s->disc_bits_max > kDiscBitsSmemLimit) s->disc_bits_max = 0;
    if (s->disc_bits_max > 0 && (dforce ? strcmp(dforce, "bits") == 0 : !lists)) {
      s->disc_bits = true;
      s->disc_smem = s->disc_bits_max;
    }
  }
  const size_t TR = (size_t)T * S.R;
  S.K = p->pool_k;
  S.Kw = (p->pool_k + 31) / 32;
  if (S.K > 0) {
    if ((st = dalloc(&S.Pool, (size_t)n * S.Kw, &s->allocs)) != MQO_OK) return bail(st);
    if ((st = dalloc(&S.pool, (size_t)g->G, &s->allocs)) != MQO_OK) return bail(st);
    if ((st = dalloc(&S.psrc, (size_t)g->G * S.K, &s->allocs)) != MQO_OK) return bail(st);
    if ((st = dalloc(&S.pval, (size_t)g->G * S.K, &s->allocs)) != MQO_OK) return bail(st);
    if ((st = dalloc(&S.pbase, (size_t)T, &s->allocs)) != MQO_OK) return bail(st);
  }
  if ((st = dalloc(&S.st, (size_t)T, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&S.act, (size_t)T, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&S.rnd, (size_t)T, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&S.bestv, (size_t)T, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&S.cnt, TR, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&s->d_cnt_plain, TR, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&s->d_eval, TR, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&S.tick, 1, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&S.gflag, (size_t)3 * g->G, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&S.any, 4, &s->allocs)) != MQO_OK) return bail(st);
  if ((st = dalloc(&s->d_pending, 1, &s->allocs)) != MQO_OK) return bail(st);
  if (cudaMallocHost(&s->h_pending, 2 * sizeof(int32_t)) != cudaSuccess) return bail(fail(MQO_ENOMEM, "pinned alloc"));
  s->h_late = s->h_pending + 1;
  *s->h_late = 0;
  s->dense_plan.late = s->h_late;
  // MQO_DENSE_POLLS: the looks of a wait inside the tensor-core step (0: every wait runs out)
  const char* polls = getenv("MQO_DENSE_POLLS");
  s->dense_plan.polls = polls ? (uint32_t)std::min<unsigned long>(strtoul(polls, nullptr, 10), kDensePolls) : kDensePolls;
  {
    // node-parallel kernels take several CTAs per item when there are few
    // items, so that about four CTAs' worth of nodes reach every SM
    const int target = g->sms * 4;
    S.split = g->num_items >= target ? 1 : std::min(8, (target + g->num_items - 1) / g->num_items);
  }
  {
    cudaEventRecord(s->ev_in, s->user);
    cudaStreamWaitEvent(s->work, s->ev_in, 0);
    cudaMemsetAsync(S.tick, 0, sizeof(int64_t), s->work);
    cudaMemsetAsync(S.gflag, 0, sizeof(int32_t) * 3 * g->G, s->work);
    cudaMemsetAsync(S.any, 0, sizeof(int32_t) * 4, s->work);
    cudaMemsetAsync(x1, 0, s->x_bytes, s->work);
    cudaEventRecord(s->ev_out, s->work);
    cudaStreamWaitEvent(s->user, s->ev_out, 0);
  }
  if (cudaGetLastError() != cudaSuccess) return bail(fail(MQO_ECUDA, "solver setup failed"));
  *out = s;
  return mqo_init(s);
}

mqo_status mqo_solver_destroy(mqo_solver s) {
  if (!s) return MQO_OK;
  if (s->work) cudaStreamSynchronize(s->work);
  if (s->gx1) cudaGraphExecDestroy(s->gx1);
  if (s->gx16) cudaGraphExecDestroy(s->gx16);
  for (void* q : s->allocs) cudaFree(q);
  cudaFree(s->d_save);
  if (s->h_pending) cudaFreeHost(s->h_pending);
  if (s->ev_in) cudaEventDestroy(s->ev_in);
  if (s->ev_out) cudaEventDestroy(s->ev_out);
  if (s->ev_fork) cudaEventDestroy(s->ev_fork);
  if (s->ev_join) cudaEventDestroy(s->ev_join);
  if (s->work2) cudaStreamDestroy(s->work2);
  if (s->work) cudaStreamDestroy(s->work);
  delete s;
  return MQO_OK;
}

mqo_status mqo_init(mqo_solver s) {
  CHECK_SOLVER(s);
  Scope sc(s);
  SolverDev& S = s->S;
  if (S.K > 0) {
    CKS(cudaMemsetAsync(S.Pool, 0, (size_t)S.g.n * S.Kw * sizeof(uint32_t), s->work));
    CKS(cudaMemsetAsync(S.pval, 0, (size_t)S.g.num_graphs * S.K * sizeof(int64_t), s->work));
    CKS(cudaMemsetAsync(S.psrc, 0, (size_t)S.g.num_graphs * S.K * sizeof(int32_t), s->work));
    CKS(cudaMemsetAsync(S.pbase, 0xff, (size_t)S.g.num_graphs * S.B * sizeof(int32_t), s->work));
  }
  CKS(launch_init(S, s->d_cnt_plain, s->work));
  return MQO_OK;
}

mqo_status mqo_run(mqo_solver s, int64_t nticks) {
  CHECK_SOLVER(s);
  if (nticks < 0) return fail(MQO_EINVAL, "nticks < 0");
  Scope sc(s);
  if (s->small) {
    for (int64_t left = nticks; left > 0; left -= kSmallTicks)
      CKS(launch_small(s->S, (int)std::min<int64_t>(left, kSmallTicks), nullptr, s->small_threads, s->small_smem, s->work));
    s->host_tick += nticks;
    return MQO_OK;
  }
  if (!s->gx1) {
    CKS(capture(s, 1, &s->gx1));
    CKS(capture(s, 16, &s->gx16));
  }
  int64_t left = nticks;
  while (left >= 16) {
    CKS(cudaGraphLaunch(s->gx16, s->work));
    left -= 16;
  }
  while (left-- > 0) CKS(cudaGraphLaunch(s->gx1, s->work));
  s->host_tick += nticks;
  return MQO_OK;
}

mqo_status mqo_run_timed(mqo_solver s, int64_t nticks, double* phase_ms, int64_t* launches) {
  CHECK_SOLVER(s);
  if (nticks < 0) return fail(MQO_EINVAL, "nticks < 0");
  constexpr int kPhases = 7;
  std::vector<cudaEvent_t> ev((size_t)(kPhases + 1) * nticks);
  for (auto& e : ev) CKS(cudaEventCreate(&e));
  cudaError_t err = cudaSuccess;
  {
    // the nticks ticks are captured as one CUDA graph (as mqo_run replays
    // them) with an event-record node between consecutive kernels
    Scope sc(s);
    const SolverDev& S = s->S;
    const int G = S.g.num_graphs;
    cudaGraph_t graph = nullptr;
    cudaGraphExec_t exec = nullptr;
    err = cudaStreamBeginCapture(s->work, cudaStreamCaptureModeThreadLocal);
    cudaError_t ek = cudaSuccess;
    for (int64_t k = 0; k < nticks && err == cudaSuccess && ek == cudaSuccess; ++k) {
      cudaEvent_t* e = &ev[(size_t)(kPhases + 1) * k];
      int i = 0;
      ek = cudaEventRecordWithFlags(e[i++], s->work, cudaEventRecordExternal);
      if (ek == cudaSuccess && S.K > 0) ek = launch_pool_ctrl(S, s->work);  // pool kernels count as control
      if (ek == cudaSuccess && S.K > 0) ek = launch_pool_apply(S, s->work);
      if (ek == cudaSuccess) ek = launch_ctrl(S, CTRL_MACHINE, nullptr, s->work);
      if (ek == cudaSuccess) ek = cudaEventRecordWithFlags(e[i++], s->work, cudaEventRecordExternal);
      if (ek == cudaSuccess) ek = launch_apply(S, s->work);
      if (ek == cudaSuccess) ek = cudaEventRecordWithFlags(e[i++], s->work, cudaEventRecordExternal);
      if (ek == cudaSuccess) ek = launch_step(S, S.cnt, S.act, S.gflag + 2 * G, s->step_smem, s->work, s->ell, s->ell_pos, s->dense, s->g->sms);
      if (ek == cudaSuccess) ek = cudaEventRecordWithFlags(e[i++], s->work, cudaEventRecordExternal);
      for (int pass = 0; pass < 3 && ek == cudaSuccess; ++pass) {
        if (s->disc_smem > 0) {
          if (pass == 0) ek = launch_disc_fused(s, s->work);  // all three passes fused
        } else {
          ek = launch_disc(S, pass, s->work);
        }
        if (ek == cudaSuccess) ek = cudaEventRecordWithFlags(e[i++], s->work, cudaEventRecordExternal);
      }
      if (ek == cudaSuccess) ek = launch_tick_end(S, s->work);
      if (ek == cudaSuccess) ek = cudaEventRecordWithFlags(e[i++], s->work, cudaEventRecordExternal);
    }
    if (err == cudaSuccess) err = cudaStreamEndCapture(s->work, &graph);
    if (err == cudaSuccess) err = ek;
    if (err == cudaSuccess) err = cudaGraphInstantiate(&exec, graph, 0);
    if (err == cudaSuccess) err = cudaGraphLaunch(exec, s->work);
    if (exec) cudaGraphExecDestroy(exec);
    if (graph) cudaGraphDestroy(graph);
  }
  if (err == cudaSuccess) err = cudaStreamSynchronize(s->work);
  double tot[kPhases] = {0};
  for (int64_t k = 0; k < nticks && err == cudaSuccess; ++k) {
    const cudaEvent_t* e = &ev[(size_t)(kPhases + 1) * k];
    for (int p = 0; p < kPhases && err == cudaSuccess; ++p) {
      float ms = 0.0f;
      err = cudaEventElapsedTime(&ms, e[p], e[p + 1]);
      tot[p] += ms;
    }
  }
  for (auto& e : ev) cudaEventDestroy(e);
  if (err != cudaSuccess) return poison(s, err, "mqo_run_timed");
  CHECK_LATE(s);
  s->host_tick += nticks;
  if (phase_ms)
    for (int p = 0; p < kPhases; ++p) phase_ms[p] = tot[p];
  // five kernels per tick with the fused discrete kernel, seven with the
  // three node-parallel passes
  if (launches) *launches = (int64_t)((s->disc_smem > 0 ? 5 : 7) + (s->S.K > 0 ? 2 : 0)) * nticks;
  return MQO_OK;
}

mqo_status mqo_solve(mqo_solver s, int64_t nticks) {
  mqo_status st = mqo_init(s);
  if (st != MQO_OK) return st;
  return mqo_run(s, nticks);
}

mqo_status mqo_step(mqo_solver s, int32_t nsteps) {
  CHECK_SOLVER(s);
  if (nsteps < 0) return fail(MQO_EINVAL, "nsteps < 0");
  Scope sc(s);
  const SolverDev& S = s->S;
  if (s->small || s->small_step) {
    for (int32_t left = nsteps; left > 0; left -= kSmallTicks)
      CKS(launch_small(S, std::min(left, kSmallTicks), s->d_cnt_plain, s->small_threads, s->small_smem, s->work));
    s->host_tick += nsteps;
    return MQO_OK;
  }
  for (int32_t i = 0; i < nsteps; ++i) {
    CKS(cudaMemsetAsync(s->d_cnt_plain, 0, sizeof(Counters) * (size_t)S.g.num_graphs * S.B * S.R, s->work));
    CKS(launch_step(S, s->d_cnt_plain, nullptr, nullptr, s->step_smem, s->work, s->ell, s->ell_pos, s->dense, s->g->sms));
    CKS(launch_tick_end(S, s->work));
  }
  s->host_tick += nsteps;
  return MQO_OK;
}

mqo_status mqo_step_stats(mqo_solver s, int64_t* value, int64_t* a, int64_t* b) {
  CHECK_SOLVER(s);
  Scope sc(s);
  CKS(launch_counters_out(s->S, s->d_cnt_plain, value, a, b, 0, s->work));
  return MQO_OK;
}

mqo_status mqo_reset(mqo_solver s, const uint8_t* traj_mask) {
  CHECK_SOLVER(s);
  if (s->S.K > 0) return fail(MQO_EINVAL, "mqo_reset is not available in pool mode (the pool machine resets)");
  Scope sc(s);
  CKS(launch_ctrl(s->S, CTRL_RESET, traj_mask, s->work));
  CKS(launch_apply(s->S, s->work));
  return MQO_OK;
}

mqo_status mqo_round(mqo_solver s, uint32_t* z_bits) {
  CHECK_SOLVER(s);
  if (!z_bits) return fail(MQO_EINVAL, "null z_bits");
  Scope sc(s);
  CKS(launch_round_bits(s->S, z_bits, s->work));
  return MQO_OK;
}

mqo_status mqo_evaluate(mqo_solver s, const uint32_t* z_bits, int64_t* value, int64_t* conflicts,
                        int64_t* uncovered) {
  CHECK_SOLVER(s);
  if (!z_bits) return fail(MQO_EINVAL, "null z_bits");
  Scope sc(s);
  const SolverDev& S = s->S;
  CKS(cudaMemsetAsync(s->d_eval, 0, sizeof(Counters) * (size_t)S.g.num_graphs * S.B * S.R, s->work));
  if (s->g->d_bits && S.B >= 32)
    CKS(launch_eval_bits(S, s->g->d_bits, s->g->d_bits_off, s->g->max_ng, z_bits, s->d_eval, s->work));
  else
    CKS(launch_eval(S, z_bits, s->d_eval, s->work));
  CKS(launch_counters_out(S, s->d_eval, value, conflicts, uncovered, 1, s->work));
  return MQO_OK;
}

mqo_status mqo_local_search(mqo_solver s, int32_t max_rounds) {
  CHECK_SOLVER(s);
  if (max_rounds < 1) return fail(MQO_EINVAL, "max_rounds must be >= 1");
  if (s->S.K > 0) return fail(MQO_EINVAL, "mqo_local_search is not available in pool mode (the pool machine searches)");
  Scope sc(s);
  SolverDev& S = s->S;
  const size_t T = (size_t)S.g.num_graphs * S.B;
  const size_t wb = s->words * sizeof(uint32_t), pbytes = s->pairs * sizeof(int32_t);
  const size_t TR = T * (size_t)S.R;
  const size_t save_bytes = T * sizeof(TrajState) + TR * sizeof(Counters) + 4 * wb + 4 * pbytes;
  if (!s->d_save) CKS(cudaMalloc(&s->d_save, save_bytes));
  char* q = static_cast<char*>(s->d_save);
  TrajState* sv_st = reinterpret_cast<TrajState*>(q);
  q += T * sizeof(TrajState);
  struct Pair {
    void* dst;
    void* src;
    size_t n;
  };
  std::vector<Pair> saves = {{q, S.cnt, TR * sizeof(Counters)}};
  q += TR * sizeof(Counters);
  for (uint32_t* w : {S.Zwork, S.Zaux, S.Zfree, S.Zdrop}) {
    saves.push_back({q, w, wb});
    q += wb;
  }
  for (int32_t* w : {S.owner, S.pa, S.pb, S.gain}) {
    saves.push_back({q, w, pbytes});
    q += pbytes;
  }
  CKS(cudaMemcpyAsync(sv_st, S.st, T * sizeof(TrajState), cudaMemcpyDeviceToDevice, s->work));
  for (auto& pr : saves) CKS(cudaMemcpyAsync(pr.dst, pr.src, pr.n, cudaMemcpyDeviceToDevice, s->work));
  int64_t ticks = 0;
  CKS(enqueue_ls_tick(s, CTRL_LS_BEGIN));
  ++ticks;
  for (int32_t r = 0; r < max_rounds; ++r) {
    CKS(enqueue_ls_tick(s, CTRL_LS));
    ++ticks;
    CKS(launch_any_pending(S, s->d_pending, s->work));
    CKS(cudaMemcpyAsync(s->h_pending, s->d_pending, sizeof(int32_t), cudaMemcpyDeviceToHost, s->work));
    CKS(cudaStreamSynchronize(s->work));
    CHECK_LATE(s);
    if (*s->h_pending == 0) break;
  }
  if (ticks & 1) {  // keep the parity of the x buffers
    CKS(launch_tick_end(S, s->work));
    ++ticks;
  }
  s->host_tick += ticks;
  CKS(launch_ls_merge(S, sv_st, s->work));
  for (auto& pr : saves) CKS(cudaMemcpyAsync(pr.src, pr.dst, pr.n, cudaMemcpyDeviceToDevice, s->work));
  return MQO_OK;
}

mqo_status mqo_best(mqo_solver s, int64_t* values, uint32_t* z_bits) {
  CHECK_SOLVER(s);
  const SolverDev& S = s->S;
  const size_t T = (size_t)S.g.num_graphs * S.B;
  {
    Scope sc(s);
    if (z_bits) CKS(cudaMemcpyAsync(z_bits, S.Zbest, s->words * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s->work));
    if (values) CKS(cudaMemcpyAsync(values, S.bestv, T * sizeof(int64_t), cudaMemcpyDeviceToHost, s->work));
  }
  CKS(cudaStreamSynchronize(s->work));
  CKS(cudaStreamSynchronize(s->user));
  CHECK_LATE(s);
  return MQO_OK;
}

mqo_status mqo_solver_info(mqo_solver s, int32_t* step_kernel, int64_t* smem_bytes, int32_t* items,
                           int32_t* replicas) {
  if (!s) return fail(MQO_EINVAL, "null solver");
  const int B = s->S.B;
  const bool staged = s->step_smem == 0 && s->S.step_staged == 1 && !s->dense;
  const bool rows = s->step_smem == 0 && s->S.step_staged == 2 && !s->dense;
  const bool smem = s->step_smem > 0 || s->dense;
  const int vec = smem   ? 0
                  : rows ? 8
                  : (s->S.step_vec > 0 ? s->S.step_vec
                                       : (staged ? default_staged_vec(B, s->S.p.x_dtype)
                                                 : default_step_vec(B, s->S.p.x_dtype)));
  if (step_kernel)
    *step_kernel = (smem ? 1 : 0) | (s->disc_smem > 0 ? 2 : 0) |
                   (s->step_smem > 0 && s->S.step_wide && !s->dense ? 4 : 0) | (staged ? 8 : 0) | (vec << 4) |
                   ((staged ? slice_kb(s) : 0) << 8) |
                   ((s->step_smem > 0 && s->S.step_c16 && !s->dense) ? (1 << 16) : 0) |
                   ((s->step_smem > 0 && s->step_ell && !s->dense) ? (1 << 17) : 0) | (s->dense ? (1 << 18) : 0) |
                   (s->small ? (1 << 19) : 0) | (rows ? (1 << 20) : 0) | (s->disc_bits ? (1 << 21) : 0) |
                   (one_wave(s) ? (1 << 22) : 0);
  if (smem_bytes) *smem_bytes = (int64_t)(s->dense ? s->dense->smem : s->step_smem);
  if (items) *items = s->S.g.num_items;
  if (replicas) *replicas = s->S.R;
  return MQO_OK;
}

mqo_status mqo_pool_state(mqo_solver s, int32_t* counts, int64_t* values, int64_t* merges, uint32_t* bits) {
  CHECK_SOLVER(s);
  const SolverDev& S = s->S;
  if (S.K == 0) return fail(MQO_EINVAL, "the solver is not in pool mode (pool_k = 0)");
  const int G = S.g.num_graphs;
  std::vector<PoolState> ps((size_t)G);
  {
    Scope sc(s);
    if (bits)
      CKS(cudaMemcpyAsync(bits, S.Pool, (size_t)S.g.n * S.Kw * sizeof(uint32_t), cudaMemcpyDeviceToDevice, s->work));
    CKS(cudaMemcpyAsync(ps.data(), S.pool, (size_t)G * sizeof(PoolState), cudaMemcpyDeviceToHost, s->work));
    if (values)
      CKS(cudaMemcpyAsync(values, S.pval, (size_t)G * S.K * sizeof(int64_t), cudaMemcpyDeviceToHost, s->work));
  }
  CKS(cudaStreamSynchronize(s->work));
  CKS(cudaStreamSynchronize(s->user));
  CHECK_LATE(s);
  for (int g = 0; g < G; ++g) {
    if (counts) counts[g] = ps[(size_t)g].count;
    if (merges) merges[g] = ps[(size_t)g].merges;
  }
  return MQO_OK;
}

mqo_status mqo_traj_state(mqo_solver s, mqo_traj_info* out) {
  CHECK_SOLVER(s);
  if (!out) return fail(MQO_EINVAL, "null out");
  const size_t T = (size_t)s->S.g.num_graphs * s->S.B;
  std::vector<TrajState> h(T);
  const int R = s->S.R;
  std::vector<Counters> c(T * R);
  CKS(cudaStreamSynchronize(s->user));
  CKS(cudaStreamSynchronize(s->work));
  CKS(cudaMemcpy(h.data(), s->S.st, T * sizeof(TrajState), cudaMemcpyDeviceToHost));
  CKS(cudaMemcpy(c.data(), s->S.cnt, T * R * sizeof(Counters), cudaMemcpyDeviceToHost));
  CHECK_LATE(s);
  const bool mis = s->p.problem == MQO_MIS;
  for (size_t i = 0; i < T; ++i) {
    // the counters of the last tick are folded into the state by the next
    // control pass; report them as the latest evaluation
    Counters sum{0ull, 0ull, 0ull, 0ull};
    for (int r = 0; r < R; ++r) {
      sum.value += c[i * R + r].value;
      sum.a += c[i * R + r].a;
      sum.b += c[i * R + r].b;
      sum.commits += c[i * R + r].commits;
    }
    // (in pool mode only if the trajectory worked in that tick: a waiting
    // trajectory keeps its last evaluation)
    if (s->S.K == 0 || (h[i].act & ACT_STEP) || h[i].round != RD_NONE) {
      const int64_t cv = (int64_t)sum.value;
      h[i].ev_value = mis ? cv : cv / 2;
      h[i].ev_a = (int64_t)sum.a;
      h[i].ev_b = (int64_t)sum.b;
      h[i].last_commits = (int64_t)sum.commits;
    }
    mqo_traj_info& o = out[i];
    const TrajState& t = h[i];
    o.phase = t.phase;
    o.s = t.s;
    o.r = t.r;
    o.o = t.o;
    o.best = t.best;
    o.ticks = t.ticks;
    o.last_round = t.last_round;
    o.pad0 = 0;
    o.last_commits = t.last_commits;
    o.ev_value = t.ev_value;
    o.ev_a = t.ev_a;
    o.ev_b = t.ev_b;
    o.accepts = t.accepts;
    o.descents = t.descents;
    o.held = t.held;
    o.first_value = t.first_value;
    o.gain_descent = t.gain_descent;
    o.gain_ls = t.gain_ls;
    o.steps = t.steps;
  }
  return MQO_OK;
}

mqo_status mqo_get_x(mqo_solver s, void* x_out) {
  CHECK_SOLVER(s);
  if (!x_out) return fail(MQO_EINVAL, "null x_out");
  Scope sc(s);
  const void* src = (s->host_tick & 1) ? s->S.X1 : s->S.X0;
  CKS(cudaMemcpyAsync(x_out, src, s->x_bytes, cudaMemcpyDeviceToDevice, s->work));
  return MQO_OK;
}

mqo_status mqo_set_x(mqo_solver s, const void* x_in) {
  CHECK_SOLVER(s);
  if (!x_in) return fail(MQO_EINVAL, "null x_in");
  Scope sc(s);
  void* dst = (s->host_tick & 1) ? s->S.X1 : s->S.X0;
  uint32_t* zdst = (s->host_tick & 1) ? s->S.ZX1 : s->S.ZX0;
  CKS(cudaMemcpyAsync(dst, x_in, s->x_bytes, cudaMemcpyDeviceToDevice, s->work));
  CKS(launch_round_bits(s->S, zdst, s->work));
  return MQO_OK;
}

mqo_status mqo_get_v(mqo_solver s, void* v_out) {
  CHECK_SOLVER(s);
  if (!v_out) return fail(MQO_EINVAL, "null v_out");
  Scope sc(s);
  CKS(cudaMemcpyAsync(v_out, s->S.V, s->v_bytes, cudaMemcpyDeviceToDevice, s->work));
  return MQO_OK;
}

mqo_status mqo_objective_f64(mqo_solver s, double* out) {
  CHECK_SOLVER(s);
  if (!out) return fail(MQO_EINVAL, "null out");
  Scope sc(s);
  const size_t T = (size_t)s->S.g.num_graphs * s->S.B;
  CKS(cudaMemsetAsync(out, 0, T * sizeof(double), s->work));
  CKS(launch_objective(s->S, out, s->work));
  return MQO_OK;
}

namespace {

// Arguments of the f_B kernels: the chunk plan and its scratch, made on first use
mqo_status fb_ready(mqo_graph g, const float* X, int32_t B) {
  if (B < 1 || B > 256 || (B & (B - 1))) return fail(MQO_EINVAL, "B=%d must be a power of two in [1,256]", B);
  // B >= 32: rows of X are read in 16-byte pieces
  if (B >= 32 && ((uintptr_t)X & 15u) != 0) return fail(MQO_EINVAL, "X must be 16-byte aligned for B >= 32");
  mqo_status st = build_heavy_plan(g);
  if (st != MQO_OK) return st;
  const size_t need = (size_t)g->hp.num_chunks * B;
  if (need > g->scratch_floats) {
    cudaFree(g->d_scratch);
    g->d_scratch = nullptr;
    g->scratch_floats = 0;
    if ((st = dalloc(&g->d_scratch, need, nullptr)) != MQO_OK) return st;
    g->scratch_floats = need;
  }
  return MQO_OK;
}

}  // namespace

mqo_status mqo_fb_forward(mqo_graph g, const float* X, int32_t B, float lambda_, double* obj, void* cuda_stream) {
  if (!g || !X || !obj) return fail(MQO_EINVAL, "null argument");
  const mqo_status st = fb_ready(g, X, B);
  if (st != MQO_OK) return st;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  CKG(cudaMemsetAsync(obj, 0, sizeof(double) * B, s));
  CKG(launch_fb(g->dev(), g->hp, X, B, lambda_, nullptr, nullptr, nullptr, obj, g->d_scratch, g->sms * 8, s));
  return MQO_OK;
}

mqo_status mqo_fb_forward_ax(mqo_graph g, const float* X, int32_t B, float lambda_, double* obj, float* AX,
                             void* cuda_stream) {
  if (!g || !X || !obj || !AX) return fail(MQO_EINVAL, "null argument");
  const mqo_status st = fb_ready(g, X, B);
  if (st != MQO_OK) return st;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  CKG(cudaMemsetAsync(obj, 0, sizeof(double) * B, s));
  CKG(launch_fb(g->dev(), g->hp, X, B, lambda_, nullptr, nullptr, AX, obj, g->d_scratch, g->sms * 8, s));
  return MQO_OK;
}

mqo_status mqo_fb_grad_ax(mqo_graph g, const float* AX, const float* gout, float* G, int32_t B, float lambda_,
                          void* cuda_stream) {
  if (!g || !AX || !G) return fail(MQO_EINVAL, "null argument");
  if (B < 1 || B > 256 || (B & (B - 1))) return fail(MQO_EINVAL, "B=%d must be a power of two in [1,256]", B);
  CKG(launch_grad_ax(AX, gout, G, g->n * B, B, lambda_, (cudaStream_t)cuda_stream));
  return MQO_OK;
}

mqo_status mqo_spmm_grad(mqo_graph g, const float* X, const float* gout, float* G, int32_t B, float lambda_,
                         void* cuda_stream) {
  if (!g || !X || !G) return fail(MQO_EINVAL, "null argument");
  const mqo_status st = fb_ready(g, X, B);
  if (st != MQO_OK) return st;
  CKG(launch_fb(g->dev(), g->hp, X, B, lambda_, gout, G, nullptr, nullptr, g->d_scratch, g->sms * 8,
                (cudaStream_t)cuda_stream));
  return MQO_OK;
}

mqo_status mqo_measure_smem_gbs(int32_t iters, double* gbs) {
  if (!gbs || iters < 1) return fail(MQO_EINVAL, "bad argument");
  int dev = 0, sms = 0;
  CKG(cudaGetDevice(&dev));
  CKG(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int grid = 2 * sms;  // two CTAs per SM
  uint32_t* sink = nullptr;
  cudaStream_t s = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t err = cudaMalloc(&sink, sizeof(uint32_t) * (size_t)grid);
  if (err == cudaSuccess) err = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking);
  if (err == cudaSuccess) err = cudaEventCreate(&e0);
  if (err == cudaSuccess) err = cudaEventCreate(&e1);
  if (err == cudaSuccess) err = launch_smem_probe(grid, iters, sink, s);  // untimed
  if (err == cudaSuccess) err = cudaEventRecord(e0, s);
  if (err == cudaSuccess) err = launch_smem_probe(grid, iters, sink, s);
  if (err == cudaSuccess) err = cudaEventRecord(e1, s);
  if (err == cudaSuccess) err = cudaEventSynchronize(e1);
  float ms = 0.0f;
  if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e0, e1);
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  if (s) cudaStreamDestroy(s);
  if (sink) cudaFree(sink);
  if (err != cudaSuccess) return fail(MQO_ECUDA, "shared-memory probe: %s", cudaGetErrorString(err));
  if (ms <= 0.0f) return fail(MQO_ECUDA, "shared-memory probe: no elapsed time");
  const double bytes = (double)grid * smem_probe_threads() * 4.0 * (double)iters * 16.0;
  *gbs = bytes / (ms * 1e-3) / 1e9;
  return MQO_OK;
}

mqo_status mqo_pga_momentum_step(float* x, float* v, const float* grad, int64_t count, float lr, float mu, float lo,
                                 float hi, void* cuda_stream) {
  if (count < 0 || (count > 0 && (!x || !v || !grad))) return fail(MQO_EINVAL, "bad argument");
  CKG(launch_momentum(x, v, grad, count, lr, mu, lo, hi, (cudaStream_t)cuda_stream));
  return MQO_OK;
}

mqo_status mqo_pga_adam_step(float* x, float* m, float* u, const float* grad, int64_t count, float lr, float b1,
                             float b2, float eps, int64_t t, float lo, float hi, void* cuda_stream) {
  if (count < 0 || (count > 0 && (!x || !m || !u || !grad)) || t < 1) return fail(MQO_EINVAL, "bad argument");
  CKG(launch_adam(x, m, u, grad, count, lr, b1, b2, eps, t, lo, hi, (cudaStream_t)cuda_stream));
  return MQO_OK;
}

mqo_status mqo_autotune(mqo_solver s, int32_t ticks, int32_t* plan_out, double* best_ms_per_tick) {
  CHECK_SOLVER(s);
  if (ticks < 1) return fail(MQO_EINVAL, "ticks must be >= 1");
  SolverDev& S = s->S;
  const int B = S.B;
  const size_t T = (size_t)S.g.num_graphs * B;
  // every mutable device buffer of the solver, saved and restored around
  // each trial so that tuning leaves the trajectories where they were
  struct Buf {
    void* p;
    size_t n;
  };
  const std::vector<Buf> bufs = {
      {S.X0, s->x_bytes}, {S.X1, s->x_bytes}, {S.V, s->v_bytes},
      {S.ZX0, s->words * 4}, {S.ZX1, s->words * 4}, {S.Zbest, s->words * 4}, {S.Zwork, s->words * 4},
      {S.Zaux, s->words * 4}, {S.Zfree, s->words * 4}, {S.Zdrop, s->words * 4},
      {S.owner, s->pairs * 4}, {S.pa, s->pairs * 4}, {S.pb, s->pairs * 4}, {S.gain, s->pairs * 4},
      {S.st, T * sizeof(TrajState)}, {S.act, T * 4}, {S.rnd, T * 4}, {S.bestv, T * 8},
      {S.cnt, T * S.R * sizeof(Counters)}, {S.tick, 8}, {S.gflag, (size_t)3 * S.g.num_graphs * 4}, {S.any, 16},
      {S.Pool, (size_t)S.g.n * S.Kw * 4}, {S.pool, (size_t)(S.K > 0 ? S.g.num_graphs : 0) * sizeof(PoolState)},
      {S.psrc, (size_t)S.g.num_graphs * S.K * 4}, {S.pval, (size_t)S.g.num_graphs * S.K * 8},
      {S.pbase, (size_t)(S.K > 0 ? T : 0) * 4}};
  size_t total = 0;
  for (const Buf& b : bufs) total += (b.n + 255) & ~(size_t)255;
  char* snap = nullptr;
  CKS(cudaMalloc(&snap, total));
  struct Plan {
    size_t step_smem;
    int vec;
    int wide;
    size_t disc_smem;
    int staged;   // 1: staged-gather step kernel, 2: row groups
    int slice_kb; // its slice capacity
    int c16;      // shared-memory step kernel with 16-bit column indices
    int ell;      // shared-memory step kernel with the sliced-ELL stream
    int dense;    // tensor-core step kernel of dense member graphs
    int small;    // the multi-tick kernel runs the ticks
    int dbits;    // fused discrete passes on bit matrices
  };
  std::vector<Plan> plans;
  std::vector<size_t> steps = {0};
  if (s->step_smem_max > 0) steps.push_back(s->step_smem_max);
  std::vector<size_t> discs = {0};
  if (s->disc_smem_max > 0) discs.push_back(s->disc_smem_max);
  const bool wide_ok = step_wide_possible(B, S.p.x_dtype);
  for (size_t st : steps)
    for (size_t dc : discs) {
      if (st > 0) {
        for (int c16 : {0, 1}) {
          if (s->ell_only || (c16 && !s->g->d_col16)) continue;
          plans.push_back({st, 0, 0, dc, 0, 0, c16, 0, 0});
          if (wide_ok) plans.push_back({st, 0, 1, dc, 0, 0, c16, 0, 0});
        }
        if (s->ell_ok) {
          if (S.p.x_dtype != DT_F32 && !s->ell_only) plans.push_back({st, 0, 0, dc, 0, 0, 0, 1, 0});
          if (wide_ok || s->ell_only) plans.push_back({st, 0, 1, dc, 0, 0, 0, 1, 0});
        }
      } else {
        for (int v : {1, 2, 4, 8}) {
          // 16-byte lanes (8 trajectories) only for 16-bit x and momentum
          if (v == 8 && (S.p.x_dtype == DT_F32 || S.p.v_dtype == DT_F32)) continue;
          if (B % v == 0 && B / v <= 32 && 32 % (B / v) == 0) plans.push_back({0, v, 0, dc, 0, 0, 0, 0, 0});
        }
        if (s->staged_ok)
          for (int kb : {16, 32, 64, 128}) {
            if (slice_set(s, kb).count <= 0) continue;
            for (int v : {2, 4, 8})
              if (staged_vec_ok(B, S.p.x_dtype, v)) plans.push_back({0, v, 0, dc, 1, kb, 0, 0, 0});
          }
        if (s->rows_ok) plans.push_back({0, 0, 0, dc, 2, 0, 0, 0, 0});
      }
    }
  if (s->dense_ok)
    for (size_t dc : discs) plans.push_back({steps.back(), 0, 0, dc, 0, 0, 0, 0, 1});
  for (Plan& pl : plans) pl.small = pl.dbits = 0;
  if (s->disc_bits_max > 0) {
    // every step plan also with the discrete passes on bit matrices
    const size_t count = plans.size();
    for (size_t i = 0; i < count; ++i)
      if (plans[i].disc_smem == 0) {
        Plan pl = plans[i];
        pl.disc_smem = s->disc_bits_max;
        pl.dbits = 1;
        plans.push_back(pl);
      }
  }
  const Plan keep{s->step_smem, S.step_vec, S.step_wide, s->disc_smem, S.step_staged, slice_kb(s), S.step_c16,
                  s->step_ell ? 1 : 0, s->dense ? 1 : 0, s->small ? 1 : 0, s->disc_bits ? 1 : 0};
  if (s->small_smem > 0 && !s->small) {
    Plan pl = keep;
    pl.small = 1;
    plans.push_back(pl);
  }
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  cudaError_t err = cudaEventCreate(&e0);
  if (err == cudaSuccess) err = cudaEventCreate(&e1);
  // the current plan is timed first and stays unless another is faster by
  // more than kTuneMargin: a few ticks cannot see kernels that have no work
  // yet (early in a run no trajectory is in a discrete round), and noise
  // alone should not move the plan
  constexpr double kTuneMargin = 0.03;
  plans.insert(plans.begin(), keep);
  double best = 1e300;
  Plan chosen = keep;
  {
    Scope sc(s);
    size_t off = 0;
    for (const Buf& b : bufs) {
      if (err == cudaSuccess && b.n > 0) err = cudaMemcpyAsync(snap + off, b.p, b.n, cudaMemcpyDeviceToDevice, s->work);
      off += (b.n + 255) & ~(size_t)255;
    }
    for (const Plan& pl : plans) {
      if (err != cudaSuccess) break;
      off = 0;
      for (const Buf& b : bufs) {
        if (err == cudaSuccess && b.n > 0) err = cudaMemcpyAsync(b.p, snap + off, b.n, cudaMemcpyDeviceToDevice, s->work);
        off += (b.n + 255) & ~(size_t)255;
      }
      s->step_smem = pl.step_smem;
      S.step_vec = pl.vec;
      S.step_wide = pl.wide;
      s->disc_smem = pl.disc_smem;
      s->disc_bits = pl.dbits != 0;
      S.step_staged = pl.staged;
      S.step_c16 = pl.c16;
      if (pl.staged == 1) use_slices(s, slice_set(s, pl.slice_kb));
      use_ell(s, pl.step_smem > 0 && pl.ell);
      s->dense = pl.dense ? &s->dense_plan : nullptr;
      if (pl.ell && !s->step_ell) continue;  // its arrays could not be built
      auto run = [&](int32_t n) {
        if (pl.small) return launch_small(S, n, nullptr, s->small_threads, s->small_smem, s->work);
        cudaError_t e = cudaSuccess;
        for (int32_t k = 0; k < n && e == cudaSuccess; ++k) e = enqueue_tick(s);
        return e;
      };
      if (err == cudaSuccess) err = run(1);  // untimed first tick
      if (err == cudaSuccess) err = cudaEventRecord(e0, s->work);
      if (err == cudaSuccess) err = run(ticks);
      if (err == cudaSuccess) err = cudaEventRecord(e1, s->work);
      if (err == cudaSuccess) err = cudaEventSynchronize(e1);
      float ms = 0.0f;
      if (err == cudaSuccess) err = cudaEventElapsedTime(&ms, e0, e1);
      if (err == cudaSuccess && (best == 1e300 || ms < best * (1.0 - kTuneMargin))) {
        best = ms;
        chosen = pl;
      }
    }
    off = 0;
    for (const Buf& b : bufs) {
      if (err == cudaSuccess && b.n > 0) err = cudaMemcpyAsync(b.p, snap + off, b.n, cudaMemcpyDeviceToDevice, s->work);
      off += (b.n + 255) & ~(size_t)255;
    }
    if (err == cudaSuccess) err = cudaStreamSynchronize(s->work);
  }
  if (e0) cudaEventDestroy(e0);
  if (e1) cudaEventDestroy(e1);
  cudaFree(snap);
  auto apply = [&](const Plan& pl) {
    s->step_smem = pl.step_smem;
    S.step_vec = pl.vec;
    S.step_wide = pl.wide;
    s->disc_smem = pl.disc_smem;
    s->disc_bits = pl.dbits != 0;
    S.step_staged = pl.staged;
    S.step_c16 = pl.c16;
    if (pl.slice_kb > 0) use_slices(s, slice_set(s, pl.slice_kb));
    use_ell(s, pl.step_smem > 0 && pl.ell);
    s->dense = pl.dense ? &s->dense_plan : nullptr;
    s->small = pl.small != 0;
  };
  if (err != cudaSuccess) {
    apply(keep);
    return poison(s, err, "mqo_autotune");
  }
  if (look_late(s) != MQO_OK) {
    apply(keep);
    return MQO_ETIMEOUT;
  }
  apply(chosen);
  // the captured tick graphs hold the old launch configuration
  if (s->gx1) cudaGraphExecDestroy(s->gx1);
  if (s->gx16) cudaGraphExecDestroy(s->gx16);
  s->gx1 = s->gx16 = nullptr;
  if (plan_out) {
    const bool stg = chosen.step_smem == 0 && chosen.staged == 1 && !chosen.dense;
    const bool rows = chosen.step_smem == 0 && chosen.staged == 2 && !chosen.dense;
    if (rows) chosen.vec = 8;
    else if (chosen.step_smem == 0 && !chosen.dense && chosen.vec == 0)
      chosen.vec = stg ? default_staged_vec(B, S.p.x_dtype) : default_step_vec(B, S.p.x_dtype);
    if (chosen.dense) chosen.wide = chosen.c16 = chosen.ell = chosen.vec = 0;
    *plan_out = (chosen.step_smem > 0 || chosen.dense ? 1 : 0) | (chosen.dense ? (1 << 18) : 0) |
                (chosen.small ? (1 << 19) : 0) | (chosen.disc_smem > 0 ? 2 : 0) | (chosen.wide ? 4 : 0) |
                (stg ? 8 : 0) | (chosen.vec << 4) | ((stg ? chosen.slice_kb : 0) << 8) |
                ((chosen.step_smem > 0 && chosen.c16) ? (1 << 16) : 0) |
                ((chosen.step_smem > 0 && chosen.ell) ? (1 << 17) : 0) | (rows ? (1 << 20) : 0) |
                (chosen.dbits ? (1 << 21) : 0) | (one_wave(s) ? (1 << 22) : 0);
  }
  if (best_ms_per_tick) *best_ms_per_tick = best / ticks;
  return MQO_OK;
}

}  // extern "C"
