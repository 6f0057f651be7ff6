// mqo_tick.cu -- the per-trajectory machine of Alg. 1 / Alg. 2 on the GPU.
//
// One tick = (pool mode: the graphs' pool decisions, mqo_pool.cu ->)
// control (one thread, or one warp, per trajectory) -> apply (accept copies,
// resets, initialisations) -> fused descent step -> discrete round passes
// A, B and the count pass C (or the fused per-graph kernel,
// mqo_disc_graph.cu) -> tick end.  The control kernel decides, from the
// exact counters of the previous tick, what each trajectory does now; the
// node-parallel kernels then act on (node, trajectory) pairs.  Member
// graphs with nothing to do in a pass are skipped through per-graph tick
// stamps written by the control kernel.
//
// Pair kernels map thread -> (node v, trajectory b), trajectory fastest,
// one CTA per item (<= 256 nodes of one member graph), or a slice of an item
// per CTA when there are few items (item_slice).  The lanes that
// share one bit word of a node (G = min(B,32) lanes) form a group; MIS set
// logic is done on whole words: the group splits v's neighbour list, ORs
// (or once/twice-accumulates) the neighbours' words and reduces by shuffles.
#include <algorithm>

#include "mqo_machine.cuh"

namespace mqo {

// ---------------------------------------------------------------- control
struct CtrlArgs {
  SolverDev S;
  int mode;
  const uint8_t* mask;
};

// The control step of trajectory tau; c = its counters of the previous tick
// (all replicas summed; not used by a forced reset).
__device__ __forceinline__ void ctrl_one(const CtrlArgs& A, int64_t tau, const Counters& c) {
  const SolverDev& S = A.S;
  const int64_t t = *S.tick;
  const int g = (int)(tau / S.B);
  const int32_t n_g = S.g.node_off[g + 1] - S.g.node_off[g];
  const Params& p = S.p;
  TrajState st = S.st[tau];
  int act = 0;
  int round = RD_NONE;

  if (A.mode == CTRL_RESET) {
    // forced reset (mqo_reset): round r+1 from the best set, new descent;
    // the counters of the last tick stay in place
    if (A.mask == nullptr || A.mask[tau]) {
      st.r += 1;
      st.s = 0;
      st.phase = PH_DESCENT;
      reset_keys(p, tau, st.o, st.r, n_g, st);
      act = ACT_RESET;
    }
    st.act = act;
    st.round = RD_NONE;
    S.st[tau] = st;
    S.act[tau] = act;
    S.rnd[tau] = RD_NONE;
    if (act) {
      S.gflag[g] = (int32_t)(t + 1);
      S.any[0] = (int32_t)(t + 1);
    }
    return;
  }

  ctrl_decide(S, A.mode, tau, g, n_g, c, st, act, round);
  st.act = act;
  st.round = round;
  S.st[tau] = st;
  S.act[tau] = act;
  S.rnd[tau] = round;
  S.bestv[tau] = st.best;
  const int32_t stamp = (int32_t)(t + 1);
  const int G = S.g.num_graphs;
  if (act & ACT_APPLY_MASK) {
    S.gflag[g] = stamp;
    S.any[0] = stamp;
  }
  if (round != RD_NONE) {
    S.gflag[G + g] = stamp;
    S.any[1] = stamp;
  }
  if (act & ACT_STEP) {
    S.gflag[2 * G + g] = stamp;
    S.any[2] = stamp;
  }
}

// one thread per trajectory: few counter replicas
__global__ void k_ctrl(CtrlArgs A) {
  const SolverDev& S = A.S;
  const int64_t T = (int64_t)S.g.num_graphs * S.B;
  const int64_t tau = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (tau >= T) return;
  Counters c{0ull, 0ull, 0ull, 0ull};
  if (A.mode != CTRL_RESET) {  // a forced reset leaves the counters in place
    c = sum_replicas(S.cnt, tau, S.R);
    for (int r = 0; r < S.R; ++r) S.cnt[tau * S.R + r] = Counters{0ull, 0ull, 0ull, 0ull};
  }
  ctrl_one(A, tau, c);
}

// one warp per trajectory: the lanes sum and clear the R replicas together
__global__ void k_ctrl_w(CtrlArgs A) {
  const SolverDev& S = A.S;
  const int64_t T = (int64_t)S.g.num_graphs * S.B;
  const int64_t tau = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (tau >= T) return;
  Counters c{0ull, 0ull, 0ull, 0ull};
  if (A.mode != CTRL_RESET) {
    for (int r = lane; r < S.R; r += 32) {
      const Counters x = S.cnt[tau * S.R + r];
      c.value += x.value;
      c.a += x.a;
      c.b += x.b;
      c.commits += x.commits;
      S.cnt[tau * S.R + r] = Counters{0ull, 0ull, 0ull, 0ull};
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      c.value += __shfl_xor_sync(0xffffffffu, c.value, o);
      c.a += __shfl_xor_sync(0xffffffffu, c.a, o);
      c.b += __shfl_xor_sync(0xffffffffu, c.b, o);
      c.commits += __shfl_xor_sync(0xffffffffu, c.commits, o);
    }
  }
  if (lane == 0) ctrl_one(A, tau, c);
}

cudaError_t launch_ctrl(const SolverDev& S, int mode, const uint8_t* mask, cudaStream_t stream) {
  const int64_t T = (int64_t)S.g.num_graphs * S.B;
  CtrlArgs a{S, mode, mask};
  if (S.R >= 8) k_ctrl_w<<<(unsigned)((T * 32 + 255) / 256), 256, 0, stream>>>(a);
  else k_ctrl<<<(unsigned)((T + 127) / 128), 128, 0, stream>>>(a);
  return cudaGetLastError();
}

__global__ void k_tick_end(int64_t* tick) { *tick += 1; }

cudaError_t launch_tick_end(const SolverDev& S, cudaStream_t stream) {
  k_tick_end<<<1, 1, 0, stream>>>(S.tick);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- apply
// Each CTA (a slice of one item) reads the actions of its member graph's
// trajectories once.  The bit sets then change a word at a time (a node's words
// belong to one CTA): accepted bits, work sets and the base of a reset by masks
// of the trajectories with each action.  x, V and the rounding bits are written
// only for the (node, trajectory) pairs of a reset or an initialisation, listed
// in increasing order and visited trajectory fastest, so that one node's writes
// are adjacent.  Bound by latency
// (chains of small loads, then 2-byte writes to sectors of x and V).  Taking every
// pair of every action through its own loads and atomics measured 26 us a tick
// against 21 (512 graphs of about 750 nodes, B = 32); queueing the pairs that need
// their place in the permutation, so that whole warps compute it, gained nothing.
__global__ void __launch_bounds__(kPairThreads, 8) k_apply(SolverDev S) {
  __shared__ int s_list[128];
  __shared__ int s_act[128];
  __shared__ uint32_t s_keys[128][6];
  __shared__ int64_t s_rk[128];
  __shared__ int32_t s_o[128];
  __shared__ int32_t s_pb[128];   // pool member that is trajectory b's base (< 0: the empty set)
  __shared__ uint32_t s_mask[4][5];
  __shared__ int s_wcnt[4];
  __shared__ uint32_t s_base[kItemMaxNodes * 4];
  // loads that do not depend on one another go out together
  const int64_t t = *S.tick;
  const int32_t any = S.any[0];
  int it;
  Item item;
  const bool mine = item_slice(S, it, item);
  if (any != (int32_t)(t + 1) || !mine) return;
  const int B = S.B, Bw = S.Bw;
  const int g = item.g;
  const int32_t flag = S.gflag[g];
  const int myact = threadIdx.x < B ? S.act[(int64_t)g * B + threadIdx.x] : 0;
  if (flag != (int32_t)(t + 1)) return;
  // masks of the actions, and the trajectories whose x is written, in order
  // (B <= 128: warps 0..3)
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < 4) {
    const bool on = myact & (ACT_RESET | ACT_INIT);
    const unsigned bal = __ballot_sync(0xffffffffu, on);
    const unsigned zx = __ballot_sync(0xffffffffu, myact & ACT_ACC_ZX);
    const unsigned wk = __ballot_sync(0xffffffffu, (myact & (ACT_ACC_WORK | ACT_ACC_ZX)) == ACT_ACC_WORK);
    const unsigned wzx = __ballot_sync(0xffffffffu, myact & ACT_WORK_ZX);
    const unsigned wb = __ballot_sync(0xffffffffu, (myact & (ACT_WORK_BEST | ACT_WORK_ZX)) == ACT_WORK_BEST);
    const unsigned pool = __ballot_sync(0xffffffffu, myact & ACT_POOL);
    if (lane == 0) {
      s_wcnt[warp] = __popc(bal);
      s_mask[warp][0] = zx;
      s_mask[warp][1] = wk;
      s_mask[warp][2] = wzx;
      s_mask[warp][3] = wb;
      s_mask[warp][4] = pool;
    }
    if (myact & ACT_POOL) s_pb[threadIdx.x] = S.pbase[(int64_t)g * B + threadIdx.x];
    asm volatile("bar.sync 1, 128;\n" ::: "memory");  // s_wcnt of warps 0..3
    if (on) {
      int pos = __popc(bal & ((1u << lane) - 1u));
      for (int w = 0; w < warp; ++w) pos += s_wcnt[w];
      const TrajState& st = S.st[(int64_t)g * B + threadIdx.x];
      s_list[pos] = threadIdx.x;
      s_act[pos] = myact;
      if (myact & ACT_RESET) {
#pragma unroll
        for (int i = 0; i < 6; ++i) s_keys[pos][i] = st.rkeys[i];
        s_rk[pos] = st.rk;
      }
      if (myact & ACT_INIT) s_o[pos] = st.o;
    }
  }
  __syncthreads();
  const int nset = s_wcnt[0] + s_wcnt[1] + s_wcnt[2] + s_wcnt[3];
  const int nodes = item.v1 - item.v0;
  void* Xc = (t & 1) ? S.X1 : S.X0;
  uint32_t* Zc = (t & 1) ? S.ZX1 : S.ZX0;
  const uint32_t* Zp = (t & 1) ? S.ZX0 : S.ZX1;  // rounding of the x the last step evaluated
  for (int idx = threadIdx.x; idx < nodes * Bw; idx += blockDim.x) {
    const int w = idx % Bw;
    const int64_t i = (int64_t)item.v0 * Bw + idx;
    const uint32_t zx = s_mask[w][0], wk = s_mask[w][1], wzx = s_mask[w][2], wb = s_mask[w][3];
    const uint32_t zbest = S.Zbest[i];
    const uint32_t zp = (zx | wzx) ? Zp[i] : 0u;
    const uint32_t zwork = (wk | wzx | wb) ? S.Zwork[i] : 0u;
    const uint32_t zb = (zbest & ~(zx | wk)) | (zp & zx) | (zwork & wk);
    if (zb != zbest) S.Zbest[i] = zb;
    // pool mode: the base of a reset / local search is pool member pbase[tau]
    uint32_t base = zb;
    if (uint32_t pool = s_mask[w][4]) {
      base &= ~pool;
      const uint32_t* member = S.Pool + (i / Bw) * S.Kw;
      for (; pool; pool &= pool - 1u) {
        const int b = __ffs(pool) - 1, k = s_pb[32 * w + b];
        if (k >= 0) base |= ((member[k >> 5] >> (k & 31)) & 1u) << b;
      }
    }
    if (wzx | wb) S.Zwork[i] = (zwork & ~(wzx | wb)) | (zp & wzx) | (base & wb);
    s_base[idx] = base;
  }
  if (nset == 0) return;
  __syncthreads();
  const bool mis = S.p.problem == PROB_MIS;
  const float thr = mis ? 0.5f : 0.0f;
  const int32_t off = S.g.node_off[g];
  const uint32_t n_g = (uint32_t)(S.g.node_off[g + 1] - off);
  for (int idx = threadIdx.x; idx < nset * nodes; idx += blockDim.x) {
    const int vi = idx / nset, j = idx - vi * nset;
    const int b = s_list[j];
    const int64_t v = item.v0 + vi;
    const uint32_t vl = (uint32_t)(v - off);
    float x;
    if (s_act[j] & ACT_RESET) {
      x = reset_x(mis, (s_base[vi * Bw + (b >> 5)] >> (b & 31)) & 1u, n_g, s_keys[j], s_rk[j], vl);
    } else {
      x = init_x(S.p, s_o[j], vl, (int64_t)g * B + b, S.g.row_ptr[v + 1] - S.g.row_ptr[v], S.g.dmax[g]);
    }
    const int64_t e = v * B + b;
    if (S.p.x_dtype == DT_F32) {
      static_cast<float*>(Xc)[e] = x;
    } else if (S.p.x_dtype == DT_BF16) {
      const __nv_bfloat16 h = __float2bfloat16_rn(x);
      static_cast<__nv_bfloat16*>(Xc)[e] = h;
      x = __bfloat162float(h);
    } else {
      const __half h = __float2half_rn(x);
      static_cast<__half*>(Xc)[e] = h;
      x = __half2float(h);
    }
    if (S.p.v_dtype == DT_F32) static_cast<float*>(S.V)[e] = 0.0f;
    else if (S.p.v_dtype == DT_BF16) static_cast<__nv_bfloat16*>(S.V)[e] = __float2bfloat16_rn(0.0f);
    else static_cast<__half*>(S.V)[e] = __float2half_rn(0.0f);
    set_bit_atomic(Zc, v, Bw, b, x > thr);
  }
}

cudaError_t launch_apply(const SolverDev& S, cudaStream_t stream) {
  k_apply<<<S.g.num_items * S.split, kPairThreads, 0, stream>>>(S);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- discrete rounds
__device__ __forceinline__ void flush_pair_counters(const SolverDev& S, unsigned long long* s_cnt, int g, int it,
                                                    Counters* dst) {
  __syncthreads();
  const int B = S.B;
  const int rep = it % S.R;
  for (int i = threadIdx.x; i < 4 * B; i += blockDim.x) {
    const unsigned long long val = s_cnt[i];
    if (val) {
      Counters* c = dst + ((int64_t)g * B + i / 4) * S.R + rep;
      const int k = i & 3;
      unsigned long long* p = k == 0 ? &c->value : k == 1 ? &c->a : k == 2 ? &c->b : &c->commits;
      atomicAdd(p, val);
    }
  }
}

__global__ void __launch_bounds__(kPairThreads) k_disc(SolverDev S, int pass) {
  __shared__ unsigned long long s_cnt[4 * 128];
  const int64_t t = *S.tick;
  if (S.any[1] != (int32_t)(t + 1)) return;
  int it;
  Item item;
  if (!item_slice(S, it, item)) return;
  const int G = S.g.num_graphs;
  if (S.gflag[G + item.g] != (int32_t)(t + 1)) return;
  const int B = S.B;
  for (int i = threadIdx.x; i < 4 * B; i += blockDim.x) s_cnt[i] = 0ull;
  __syncthreads();
  disc_pass(S, item, pass, s_cnt);
  flush_pair_counters(S, s_cnt, item.g, it, S.cnt);
}

cudaError_t launch_disc(const SolverDev& S, int pass, cudaStream_t stream) {
  k_disc<<<S.g.num_items * S.split, kPairThreads, 0, stream>>>(S, pass);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- readouts
__global__ void __launch_bounds__(kPairThreads) k_round_bits(SolverDev S, uint32_t* z) {
  const int64_t t = *S.tick;
  const void* Xc = (t & 1) ? S.X1 : S.X0;
  const bool mis = S.p.problem == PROB_MIS;
  const float thr = mis ? 0.5f : 0.0f;
  const Item item = S.g.items[blockIdx.x];
  item_pairs(S, item, [&](const PairCtx& c) {
    float x = 0.0f;
    if (c.in) {
      const int64_t e = c.v * S.B + c.b;
      if (S.p.x_dtype == DT_F32) x = static_cast<const float*>(Xc)[e];
      else if (S.p.x_dtype == DT_BF16) x = __bfloat162float(static_cast<const __nv_bfloat16*>(Xc)[e]);
      else x = __half2float(static_cast<const __half*>(Xc)[e]);
    }
    update_word(z, c.v, S.Bw, c.b, S.B, x > thr, c.in);
  });
}

cudaError_t launch_round_bits(const SolverDev& S, uint32_t* z, cudaStream_t stream) {
  k_round_bits<<<S.g.num_items, kPairThreads, 0, stream>>>(S, z);
  return cudaGetLastError();
}

// The readout kernels sum a pair's neighbours kAhead at a time, so that many
// loads are in flight, and split the items until every SM has about eight
// CTAs (64 graphs of 750 nodes, 32 trajectories: objective, evaluation and
// rounding together 430 us -> 144 us; one neighbour at a time and a CTA per item
// they waited for one L2 load after the other).
constexpr int kAhead = 8;
static SolverDev split_items(const SolverDev& S, int sms) {
  SolverDev D = S;
  const int target = 8 * sms;
  D.split = S.g.num_items >= target ? 1 : std::min(16, (target + S.g.num_items - 1) / S.g.num_items);
  return D;
}
static int sm_count() {
  int dev = 0, sms = 152;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// exact evaluation of given bits: MIS (size, conflicting edges x2, uncovered);
// MaxCut (2*cut, non-fixed, positive gain)
__global__ void __launch_bounds__(kPairThreads) k_eval(SolverDev S, const uint32_t* __restrict__ z, Counters* out) {
  __shared__ unsigned long long s_cnt[4 * 128];
  const int B = S.B, Bw = S.Bw;
  const bool mis = S.p.problem == PROB_MIS;
  const int32_t* __restrict__ rp = S.g.row_ptr;
  const int32_t* __restrict__ col = S.g.col;
  const int8_t* __restrict__ wts = S.g.w;
  int it;
  Item item;
  if (!item_slice(S, it, item)) return;
  for (int i = threadIdx.x; i < 4 * B; i += blockDim.x) s_cnt[i] = 0ull;
  __syncthreads();
  long long a0 = 0, a1 = 0, a2 = 0;
  const int my_b = (int)(threadIdx.x % B);
  item_pairs(S, item, [&](const PairCtx& c) {
    if (!c.in) return;
    const int64_t v = c.v;
    const int b = c.b;
    const bool zv = get_bit(z, v, Bw, b);
    // neighbours (their weights) in the set, and all of them
    const int32_t j1 = rp[v + 1];
    int32_t j = rp[v];
    int P = 0, W = wts ? 0 : j1 - j;
    for (; j + kAhead <= j1; j += kAhead) {
      bool in[kAhead];
#pragma unroll
      for (int k = 0; k < kAhead; ++k) in[k] = get_bit(z, col[j + k], Bw, b);
#pragma unroll
      for (int k = 0; k < kAhead; ++k) {
        const int w = wts ? (int)wts[j + k] : 1;
        if (wts) W += w;
        P += in[k] ? w : 0;
      }
    }
    for (; j < j1; ++j) {
      const int w = wts ? (int)wts[j] : 1;
      if (wts) W += w;
      P += get_bit(z, col[j], Bw, b) ? w : 0;
    }
    if (mis) {
      a0 += zv;
      a1 += zv ? P : 0;
      a2 += !zv && P == 0;
    } else {
      const int as = 2 * P - W;
      a0 += zv ? (W - P) : P;
      a1 += !(zv ? (as <= -1) : (as >= 0));
      a2 += (zv ? as : -as) > 0;
    }
  });
  if (a0) atomicAdd(&s_cnt[4 * my_b + 0], (unsigned long long)a0);
  if (a1) atomicAdd(&s_cnt[4 * my_b + 1], (unsigned long long)a1);
  if (a2) atomicAdd(&s_cnt[4 * my_b + 2], (unsigned long long)a2);
  flush_pair_counters(S, s_cnt, item.g, it, out);
}

cudaError_t launch_eval(const SolverDev& S, const uint32_t* z, Counters* out, cudaStream_t stream) {
  const SolverDev D = split_items(S, sm_count());
  k_eval<<<D.g.num_items * D.split, kPairThreads, 0, stream>>>(D, z, out);
  return cudaGetLastError();
}

// counters (R replicas) -> user arrays. kind 0: step/machine counters
// (MaxCut value is 2*cut); kind 1: evaluation counters (MIS a = 2*edges,
// MaxCut value = 2*cut)
__global__ void k_counters_out(const Counters* c, int64_t T, int R, int mis, int kind, int64_t* value, int64_t* a,
                               int64_t* b) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= T) return;
  const Counters x = sum_replicas(c, i, R);
  int64_t v = (int64_t)x.value, aa = (int64_t)x.a;
  if (!mis) v /= 2;
  if (mis && kind == 1) aa /= 2;
  if (value) value[i] = v;
  if (a) a[i] = aa;
  if (b) b[i] = (int64_t)x.b;
}

cudaError_t launch_counters_out(const SolverDev& S, const Counters* c, int64_t* value, int64_t* a, int64_t* b,
                                int kind, cudaStream_t stream) {
  const int64_t T = (int64_t)S.g.num_graphs * S.B;
  k_counters_out<<<(unsigned)((T + 255) / 256), 256, 0, stream>>>(c, T, S.R, S.p.problem == PROB_MIS, kind, value,
                                                                  a, b);
  return cudaGetLastError();
}

// relaxed objective per trajectory in double: (Ax)_v in float32 (CSR order),
// then the node's terms in double (MIS h; MaxCut f_B, f_L = 1/4 x'(D-A)x,
// f_P = x'(D-A+lambda I)x or f_A = -x'Ax), accumulated per thread and
// reduced per item in shared memory
template <typename TX>
__global__ void __launch_bounds__(kPairThreads) k_objective(SolverDev S, double* out) {
  __shared__ double s_obj[128];
  const int64_t t = *S.tick;
  const TX* __restrict__ Xc = static_cast<const TX*>((t & 1) ? S.X1 : S.X0);
  const int32_t* __restrict__ rp = S.g.row_ptr;
  const int32_t* __restrict__ col = S.g.col;
  const int8_t* __restrict__ wts = S.g.w;
  const int B = S.B;
  const bool mis = S.p.problem == PROB_MIS;
  auto ld = [&](int64_t e) -> float { return to_f(Xc[e]); };
  int it;
  Item item;
  if (!item_slice(S, it, item)) return;
  for (int i = threadIdx.x; i < B; i += blockDim.x) s_obj[i] = 0.0;
  __syncthreads();
  double part = 0.0;
  item_pairs(S, item, [&](const PairCtx& c) {
    if (!c.in) return;
    const int32_t j1 = rp[c.v + 1];
    int32_t j = rp[c.v];
    float acc = 0.0f;
    int d = wts ? 0 : j1 - j;
    for (; j + kAhead <= j1; j += kAhead) {
      float f[kAhead];
#pragma unroll
      for (int k = 0; k < kAhead; ++k) f[k] = ld((int64_t)col[j + k] * B + c.b);
#pragma unroll
      for (int k = 0; k < kAhead; ++k) {
        const int w = wts ? (int)wts[j + k] : 1;
        if (wts) d += w;
        acc = w >= 0 ? acc + f[k] : acc - f[k];
      }
    }
    for (; j < j1; ++j) {
      const float xu = ld((int64_t)col[j] * B + c.b);
      const int w = wts ? (int)wts[j] : 1;
      if (wts) d += w;
      acc = w >= 0 ? acc + xu : acc - xu;
    }
    const double xv = (double)ld(c.v * B + c.b);
    const double xax = xv * (double)acc, lam = (double)S.p.lambda_;
    if (mis) {
      part += xv - 0.5 * (double)S.p.gamma * xax;
    } else {
      const double xdx = (double)d * xv * xv;
      switch (S.p.objective) {
        case OBJ_FL: part += 0.25 * (xdx - xax); break;
        case OBJ_FP: part += (xdx - xax) + lam * xv * xv; break;
        case OBJ_FA: part += -xax; break;
        default: part += -lam * xv - xax; break;
      }
    }
  });
  if (part != 0.0) atomicAdd(&s_obj[threadIdx.x % B], part);
  __syncthreads();
  for (int i = threadIdx.x; i < B; i += blockDim.x)
    if (s_obj[i] != 0.0) atomicAdd(&out[(int64_t)item.g * B + i], s_obj[i]);
}

// The same with pieces of VEC values of x: a lane holds VEC
// trajectories, B / VEC lanes a node, so one load serves 32 / (B / VEC) nodes; the
// ids of a node's neighbours come one per lane and go round by shuffles.
template <typename TX, int VEC, bool WEIGHTED>
__global__ void __launch_bounds__(kPairThreads, 4) k_objective_v(SolverDev S, double* out) {
  __shared__ double s_obj[128];
  const int64_t t = *S.tick;
  const TX* __restrict__ Xc = static_cast<const TX*>((t & 1) ? S.X1 : S.X0);
  const int32_t* __restrict__ rp = S.g.row_ptr;
  const int32_t* __restrict__ col = S.g.col;
  const int8_t* __restrict__ wts = S.g.w;
  const int B = S.B, lpr = B / VEC, rpw = 32 / lpr;
  const bool mis = S.p.problem == PROB_MIS;
  int it;
  Item item;
  if (!item_slice(S, it, item)) return;
  for (int i = threadIdx.x; i < B; i += blockDim.x) s_obj[i] = 0.0;
  __syncthreads();
  const int lane = threadIdx.x & 31, sub = lane / lpr, l = lane - sub * lpr, warp = threadIdx.x >> 5;
  const double lam = (double)S.p.lambda_;
  double part[VEC];
#pragma unroll
  for (int e = 0; e < VEC; ++e) part[e] = 0.0;
  for (int v0 = item.v0 + warp * rpw; v0 < item.v1; v0 += (kPairThreads / 32) * rpw) {
    const int v = v0 + sub;
    const bool in = v < item.v1;
    const int32_t j0 = in ? rp[v] : 0, len = in ? rp[v + 1] - j0 : 0;
    const int longest = __reduce_max_sync(0xffffffffu, len);
    const Pack<TX, VEC> xv = ld_pack<TX, VEC>(Xc + (int64_t)(in ? v : item.v0) * B + l * VEC);
    float acc[VEC];
    int d = WEIGHTED ? 0 : len;
#pragma unroll
    for (int e = 0; e < VEC; ++e) acc[e] = 0.0f;
    // ids (weights) of 4 lpr entries per round, one round ahead
    int u[4], w[4], un[4], wn[4];
    auto ids = [&](int k0, int* uu, int* ww) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = k0 + i * lpr + l;
        uu[i] = k < len ? col[j0 + k] : -1;
        if (WEIGHTED) ww[i] = k < len ? (int)wts[j0 + k] : 0;
      }
    };
    ids(0, u, w);
    for (int k0 = 0; k0 < longest; k0 += 4 * lpr) {
      ids(k0 + 4 * lpr, un, wn);
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        for (int k = 0; k < lpr && k0 + i * lpr + k < longest; k += 4) {
          Pack<TX, VEC> p[4];
          int uk[4], wk[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uk[q] = __shfl_sync(0xffffffffu, u[i], (k + q) & (lpr - 1), lpr);
            if (WEIGHTED) wk[q] = __shfl_sync(0xffffffffu, w[i], (k + q) & (lpr - 1), lpr);
            if (k + q >= lpr) uk[q] = -1;
            if (uk[q] >= 0) p[q] = ld_pack<TX, VEC>(Xc + (int64_t)uk[q] * B + l * VEC);
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            if (uk[q] < 0) continue;
            if (WEIGHTED) d += wk[q];
#pragma unroll
            for (int e = 0; e < VEC; ++e)
              acc[e] = !WEIGHTED || wk[q] >= 0 ? acc[e] + to_f(p[q].e[e]) : acc[e] - to_f(p[q].e[e]);
          }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        u[i] = un[i];
        if (WEIGHTED) w[i] = wn[i];
      }
    }
    if (!in) continue;
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
      const double x = (double)to_f(xv.e[e]);
      const double xax = x * (double)acc[e];
      if (mis) {
        part[e] += x - 0.5 * (double)S.p.gamma * xax;
      } else {
        const double xdx = (double)d * x * x;
        switch (S.p.objective) {
          case OBJ_FL: part[e] += 0.25 * (xdx - xax); break;
          case OBJ_FP: part[e] += (xdx - xax) + lam * x * x; break;
          case OBJ_FA: part[e] += -xax; break;
          default: part[e] += -lam * x - xax; break;
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < VEC; ++e) {
    for (int o = lpr; o < 32; o <<= 1) part[e] += __shfl_xor_sync(0xffffffffu, part[e], o);
    if (sub == 0 && part[e] != 0.0) atomicAdd(&s_obj[l * VEC + e], part[e]);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < B; i += blockDim.x)
    if (s_obj[i] != 0.0) atomicAdd(&out[(int64_t)item.g * B + i], s_obj[i]);
}

cudaError_t launch_objective(const SolverDev& S, double* out, cudaStream_t stream) {
  SolverDev D = split_items(S, sm_count());
  constexpr int vec = 4;
  if (S.B >= vec) D.split = std::max(1, std::min(D.split, S.B / vec));  // every warp of a CTA has rows
  const int grid = D.g.num_items * D.split;
  // (eight values per lane need more registers than four CTAs per SM have)
  auto run = [&](auto tx) {
    using TX = decltype(tx);
    if (S.g.w) k_objective_v<TX, vec, true><<<grid, kPairThreads, 0, stream>>>(D, out);
    else k_objective_v<TX, vec, false><<<grid, kPairThreads, 0, stream>>>(D, out);
    return cudaGetLastError();
  };
  if (S.B >= vec) {
    if (S.p.x_dtype == DT_F32) return run(float{});
    if (S.p.x_dtype == DT_BF16) return run(__nv_bfloat16{});
    return run(__half{});
  }
  if (S.p.x_dtype == DT_F32) k_objective<float><<<grid, kPairThreads, 0, stream>>>(D, out);
  else if (S.p.x_dtype == DT_BF16) k_objective<__nv_bfloat16><<<grid, kPairThreads, 0, stream>>>(D, out);
  else k_objective<__half><<<grid, kPairThreads, 0, stream>>>(D, out);
  return cudaGetLastError();
}

// after a standalone local search: restore the machine state, keep best
__global__ void k_ls_merge(TrajState* st, const TrajState* saved, int64_t* bestv, int64_t T) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= T) return;
  TrajState s = saved[i];
  s.best = st[i].best;
  s.accepts = st[i].accepts;
  s.first_value = st[i].first_value;
  s.gain_descent = st[i].gain_descent;
  s.gain_ls = st[i].gain_ls;
  st[i] = s;
  bestv[i] = s.best;
}

cudaError_t launch_ls_merge(const SolverDev& S, const TrajState* saved, cudaStream_t stream) {
  const int64_t T = (int64_t)S.g.num_graphs * S.B;
  k_ls_merge<<<(unsigned)((T + 255) / 256), 256, 0, stream>>>(S.st, saved, S.bestv, T);
  return cudaGetLastError();
}

// fresh machine state for every trajectory: first descent of outer
// iteration 0, no best set, the initial x (Alg. 1/2 step 2), V = 0 and empty bit
// sets, all in one launch (twelve memsets and two kernels before: 65 us for 24
// graphs of up to 300 nodes, 8 trajectories; 313 us for 512 graphs of 750, 32
// trajectories).  The move arrays (owner, pa, pb, gain) need no fill: every
// local search and repair begins with a counting round, whose pass C writes
// owner and gain, and pa / pb are written by pass A of the tick that reads
// them.  Bound by Philox4x64-10 (twenty 64-bit products per value).
__global__ void __launch_bounds__(kPairThreads) k_init(SolverDev S, Counters* plain) {
  const int64_t T = (int64_t)S.g.num_graphs * S.B;
  const int64_t t = *S.tick;
  const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = first; i < T * S.R; i += step) {
    S.cnt[i] = Counters{0ull, 0ull, 0ull, 0ull};
    plain[i] = Counters{0ull, 0ull, 0ull, 0ull};
  }
  for (int64_t tau = first; tau < T; tau += step) {
    TrajState st;
    st.phase = PH_DESCENT;
    st.s = 0;
    st.r = 0;
    st.o = 0;
    st.best = (int64_t)(-9223372036854775807LL - 1);
    st.ticks = 0;
    st.last_round = RD_NONE;
    st.round = RD_NONE;
    st.last_commits = 0;
    st.ev_value = st.ev_a = st.ev_b = 0;
    st.accepts = st.descents = 0;
    st.act = ACT_INIT;
    st.ls_done = 0;
    for (int i = 0; i < 6; ++i) st.rkeys[i] = 0u;
    st.rk = 0;
    st.held = (int64_t)(-9223372036854775807LL - 1);
    st.first_value = st.held;
    st.gain_descent = st.gain_ls = 0;
    st.steps = 0;
    S.st[tau] = st;
    if (S.K > 0 && tau < S.g.num_graphs) {
      PoolState ps;
      ps.epoch = EP_DESCENT;
      ps.count = 0;
      ps.best = st.best;
      ps.merges = 0;
      ps.dec = DEC_NONE;
      ps.best_src = -1;
      ps.merged = 0;
      ps.stamp = 0;
      S.pool[tau] = ps;
    }
    S.act[tau] = ACT_INIT;
    S.rnd[tau] = RD_NONE;
    S.bestv[tau] = st.best;
  }
  int it;
  Item item;
  if (!item_slice(S, it, item)) return;
  const bool mis = S.p.problem == PROB_MIS;
  const float thr = mis ? 0.5f : 0.0f;
  void* Xc = (t & 1) ? S.X1 : S.X0;
  uint32_t* Zc = (t & 1) ? S.ZX1 : S.ZX0;
  uint32_t* Zo = (t & 1) ? S.ZX0 : S.ZX1;
  const int32_t off = S.g.node_off[item.g], dmax = S.g.dmax[item.g];
  item_pairs(S, item, [&](const PairCtx& c) {
    float x = 0.0f;
    if (c.in) {
      const int64_t e = c.v * S.B + c.b;
      x = init_x(S.p, 0, (uint32_t)(c.v - off), c.tau, S.g.row_ptr[c.v + 1] - S.g.row_ptr[c.v], dmax);
      if (S.p.x_dtype == DT_F32) {
        static_cast<float*>(Xc)[e] = x;
      } else if (S.p.x_dtype == DT_BF16) {
        const __nv_bfloat16 h = __float2bfloat16_rn(x);
        static_cast<__nv_bfloat16*>(Xc)[e] = h;
        x = __bfloat162float(h);
      } else {
        const __half h = __float2half_rn(x);
        static_cast<__half*>(Xc)[e] = h;
        x = __half2float(h);
      }
      if (S.p.v_dtype == DT_F32) static_cast<float*>(S.V)[e] = 0.0f;
      else static_cast<uint16_t*>(S.V)[e] = 0;
    }
    const unsigned m = __ballot_sync(0xffffffffu, c.in && x > thr);
    if (c.in && c.gl == 0) {
      const int64_t w = c.v * S.Bw + c.wk;
      Zc[w] = (m & c.gmask) >> ((threadIdx.x & 31) & ~(c.G - 1));
      Zo[w] = 0u;
      S.Zbest[w] = 0u;
      S.Zwork[w] = 0u;
      S.Zaux[w] = 0u;
      S.Zfree[w] = 0u;
      S.Zdrop[w] = 0u;
    }
  });
}

cudaError_t launch_init(const SolverDev& S, Counters* plain, cudaStream_t stream) {
  k_init<<<S.g.num_items * S.split, kPairThreads, 0, stream>>>(S, plain);
  return cudaGetLastError();
}

// out = number of trajectories still running a standalone local search
__global__ void k_any_pending(SolverDev S, int32_t* out) {
  const int64_t T = (int64_t)S.g.num_graphs * S.B;
  int c = 0;
  for (int64_t i = threadIdx.x; i < T; i += blockDim.x) c += S.st[i].ls_done == 0;
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  __shared__ int s[32];
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = c;
  __syncthreads();
  if (threadIdx.x == 0) {
    int tot = 0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) tot += s[i];
    *out = tot;
  }
}

cudaError_t launch_any_pending(const SolverDev& S, int32_t* out, cudaStream_t stream) {
  k_any_pending<<<1, 1024, 0, stream>>>(S, out);
  return cudaGetLastError();
}

}  // namespace mqo
