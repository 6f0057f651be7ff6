// mqo_small.cu -- many ticks (or plain steps) of small member graphs in one
// launch (k_small): one CTA per member graph holds its CSR, iterates, momentum,
// bit sets and machine states in shared memory and runs the tick -- control,
// apply, step, discrete passes -- with block barriers in between.
//
// Why: a tick of the kernels in mqo_tick.cu is five to seven dependent launches
// of about 2 us each, whatever the size: 13 us for one graph of 200 nodes and
// one trajectory.  Member graphs do not interact, so a CTA needs nothing but
// barriers.  Bound by latency: the control decision of a thread, then the
// longest row's chain of shared-memory loads.
// Same decisions, sums and bit sets as the tick kernels: a thread sums its
// (node, trajectory) pair's neighbours in CSR order.
#include "mqo_machine.cuh"
#include "mqo_step.cuh"

namespace mqo {

// byte offsets of a CTA's shared memory
struct SmallLayout {
  size_t st, cnt, step, act, list, rnd, rp, col, w, x0, x1, v, z, total;
};

__host__ __device__ __forceinline__ SmallLayout small_layout(int B, int sx, int sv, int ng, int nnz, bool weighted) {
  SmallLayout L;
  const size_t pairs = (size_t)ng * B, words = (size_t)ng * ((B + 31) / 32);
  L.st = 0;
  L.cnt = L.st + align16(sizeof(TrajState) * B);
  L.step = L.cnt + align16((size_t)4 * B * 8);
  L.act = L.step + align16((size_t)3 * B * 4);
  L.list = L.act + align16((size_t)B * 4);
  L.rnd = L.list + align16((size_t)B * 4);
  L.rp = L.rnd + align16((size_t)B * 4);
  L.col = L.rp + align16((size_t)(ng + 1) * 4);
  L.w = L.col + align16((size_t)nnz * 2);
  L.x0 = L.w + (weighted ? align16((size_t)nnz) : 0);
  L.x1 = L.x0 + align16(pairs * sx);
  L.v = L.x1 + align16(pairs * sx);
  L.z = L.v + align16(pairs * sv);
  L.total = L.z + align16(7 * words * 4);
  return L;
}

size_t small_smem_bytes(int B, int x_dtype, int v_dtype, int ng, int nnz, bool weighted) {
  return small_layout(B, x_dtype == DT_F32 ? 4 : 2, v_dtype == DT_F32 ? 4 : 2, ng, nnz, weighted).total;
}

// count > 0 ticks of the machine, or plain steps of every trajectory whose
// last evaluation goes to `plain` (when not null); the caller advances the
// tick number afterwards
template <typename TX, typename TV, bool MIS>
__global__ void __launch_bounds__(1024) k_small(SolverDev S, int count, Counters* plain) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ int s_flag[2];
  __shared__ int s_nact;
  const int g = blockIdx.x;
  const int B = S.B, Bw = S.Bw;
  const int tid = threadIdx.x, lane = tid & 31, nt = blockDim.x;
  const int64_t t0 = *S.tick;
  const int32_t off = S.g.node_off[g];
  const int32_t ng = S.g.node_off[g + 1] - off;
  const int32_t j0 = S.g.row_ptr[off];
  const int32_t nnz = S.g.row_ptr[off + ng] - j0;
  const bool weighted = S.g.w != nullptr;
  const SmallLayout L = small_layout(B, (int)sizeof(TX), (int)sizeof(TV), ng, nnz, weighted);
  TrajState* st = reinterpret_cast<TrajState*>(smem + L.st);
  unsigned long long* s_cnt = reinterpret_cast<unsigned long long*>(smem + L.cnt);
  int* s_step = reinterpret_cast<int*>(smem + L.step);
  int* s_act = reinterpret_cast<int*>(smem + L.act);
  int* s_list = reinterpret_cast<int*>(smem + L.list);
  int* s_rnd = reinterpret_cast<int*>(smem + L.rnd);
  int32_t* rp = reinterpret_cast<int32_t*>(smem + L.rp);
  uint16_t* col = reinterpret_cast<uint16_t*>(smem + L.col);
  int8_t* wts = reinterpret_cast<int8_t*>(smem + L.w);
  TX* X[2] = {reinterpret_cast<TX*>(smem + L.x0), reinterpret_cast<TX*>(smem + L.x1)};
  TV* V = reinterpret_cast<TV*>(smem + L.v);
  const int words = ng * Bw, pairs = ng * B;
  uint32_t* Z = reinterpret_cast<uint32_t*>(smem + L.z);  // ZX0, ZX1, best, work, aux, free, drop
  uint32_t* gZ[7] = {S.ZX0, S.ZX1, S.Zbest, S.Zwork, S.Zaux, S.Zfree, S.Zdrop};
  const int64_t tau0 = (int64_t)g * B;
  const int64_t poff = (int64_t)off * B, woff = (int64_t)off * Bw;

  for (int i = tid; i <= ng; i += nt) rp[i] = S.g.row_ptr[off + i] - j0;
  for (int i = tid; i < nnz; i += nt) {
    col[i] = (uint16_t)(S.g.col[j0 + i] - off);
    if (weighted) wts[i] = S.g.w[j0 + i];
  }
  for (int i = tid; i < pairs; i += nt) {
    X[0][i] = static_cast<const TX*>(S.X0)[poff + i];
    X[1][i] = static_cast<const TX*>(S.X1)[poff + i];
    V[i] = static_cast<const TV*>(S.V)[poff + i];
  }
#pragma unroll
  for (int k = 0; k < 7; ++k)
    for (int i = tid; i < words; i += nt) Z[k * words + i] = gZ[k][woff + i];
  if (tid < B) {
    if (!plain) {
      st[tid] = S.st[tau0 + tid];
      const Counters c = S.cnt[tau0 + tid];
      s_cnt[4 * tid] = c.value, s_cnt[4 * tid + 1] = c.a, s_cnt[4 * tid + 2] = c.b, s_cnt[4 * tid + 3] = c.commits;
    }
    s_act[tid] = ACT_STEP;
#pragma unroll
    for (int k = 0; k < 3; ++k) s_step[3 * tid + k] = 0;
  }
  if (tid < 2) s_flag[tid] = 0;
  __syncthreads();

  // the solver with the graph's bit sets and rounds in shared memory, for the
  // discrete passes (global node and trajectory numbers)
  SolverDev D = S;
  D.Zbest = Z + 2 * words - woff;
  D.Zwork = Z + 3 * words - woff;
  D.Zaux = Z + 4 * words - woff;
  D.Zfree = Z + 5 * words - woff;
  D.Zdrop = Z + 6 * words - woff;
  D.rnd = s_rnd - tau0;
  const Item item{g, off, off + ng, 0};

  const float thr = MIS ? 0.5f : 0.0f, lo = MIS ? 0.0f : -1.0f;
  StepArgs a;
  a.objective = S.p.objective;
  a.alpha = S.p.alpha;
  a.momentum = S.p.momentum;
  a.gamma = S.p.gamma;
  a.lambda_ = S.p.lambda_;
  const int b = tid % B;  // nt is a multiple of B
  const int GL = B < 32 ? B : 32;  // lanes that share a bit word
  const unsigned gmask = GL == 32 ? 0xffffffffu : ((1u << GL) - 1u);

  for (int i = 0; i < count; ++i) {
    const int64_t t = t0 + i;
    int flag = 4;
    if (!plain) {
      // control
      if (tid < B) {
        Counters c;
        c.value = s_cnt[4 * tid] + (unsigned long long)(long long)s_step[3 * tid];
        c.a = s_cnt[4 * tid + 1] + (unsigned long long)(long long)s_step[3 * tid + 1];
        c.b = s_cnt[4 * tid + 2] + (unsigned long long)(long long)s_step[3 * tid + 2];
        c.commits = s_cnt[4 * tid + 3];
#pragma unroll
        for (int k = 0; k < 4; ++k) s_cnt[4 * tid + k] = 0ull;
#pragma unroll
        for (int k = 0; k < 3; ++k) s_step[3 * tid + k] = 0;
        int act, round;
        ctrl_decide(S, CTRL_MACHINE, tau0 + tid, g, ng, c, st[tid], act, round);
        st[tid].act = act;
        st[tid].round = round;
        s_act[tid] = act;
        s_rnd[tid] = round;
        atomicOr(&s_flag[i & 1],
                 ((act & ACT_APPLY_MASK) ? 1 : 0) | (round != RD_NONE ? 2 : 0) | ((act & ACT_STEP) ? 4 : 0));
      }
      if (tid == 0) {
        s_flag[(i + 1) & 1] = 0;
        s_nact = 0;
      }
      __syncthreads();
      flag = s_flag[i & 1];
      if (flag & 1) {
        // accept copies, resets and initialisations of the acting trajectories
        if (tid < B && (s_act[tid] & ACT_APPLY_MASK)) s_list[atomicAdd(&s_nact, 1)] = tid;
        __syncthreads();
        const int nact = s_nact;
        TX* Xc = X[t & 1];
        uint32_t* Zc = Z + (t & 1) * words;
        const uint32_t* Zp = Z + ((t + 1) & 1) * words;
        uint32_t *Zbest = Z + 2 * words, *Zwork = Z + 3 * words;
        for (int idx = tid; idx < nact * ng; idx += nt) {
          const int q = s_list[idx % nact], vl = idx / nact;
          const int act = s_act[q];
          bool base = get_bit(Zbest, vl, Bw, q);
          if (act & (ACT_ACC_ZX | ACT_ACC_WORK)) {
            const bool src = (act & ACT_ACC_ZX) ? get_bit(Zp, vl, Bw, q) : get_bit(Zwork, vl, Bw, q);
            if (src != base) set_bit_atomic(Zbest, vl, Bw, q, src);
            base = src;
          }
          if (act & (ACT_WORK_ZX | ACT_WORK_BEST))
            set_bit_atomic(Zwork, vl, Bw, q, (act & ACT_WORK_ZX) ? get_bit(Zp, vl, Bw, q) : base);
          if (act & (ACT_RESET | ACT_INIT)) {
            float x = (act & ACT_RESET)
                          ? reset_x(MIS, base, (uint32_t)ng, st[q].rkeys, st[q].rk, (uint32_t)vl)
                          : init_x(S.p, st[q].o, (uint32_t)vl, tau0 + q, rp[vl + 1] - rp[vl], S.g.dmax[g]);
            const TX h = from_f<TX>(x);
            Xc[vl * B + q] = h;
            V[vl * B + q] = from_f<TV>(0.0f);
            set_bit_atomic(Zc, vl, Bw, q, to_f(h) > thr);
          }
        }
        __syncthreads();
      }
    }
    if (flag & 4) {
      // the step: a thread owns (node, trajectory) pairs of trajectory b
      const TX* __restrict__ Xc = X[t & 1];
      TX* __restrict__ Xn = X[(t + 1) & 1];
      uint32_t* Zn = Z + ((t + 1) & 1) * words;
      const bool stepping = (s_act[b] & ACT_STEP) != 0;
      int c0 = 0, c1 = 0, c2 = 0;
      for (int base = tid & ~31; base < pairs; base += nt) {
        const int idx = base + lane;
        const bool in = idx < pairs;
        bool zn = false;
        const int vl = in ? idx / B : 0;
        if (in) {
          const int r0 = rp[vl], r1 = rp[vl + 1];
          float acc = 0.0f;
          int nb = 0, ws = weighted ? 0 : r1 - r0;
          if (!weighted) {
#pragma unroll 4
            for (int j = r0; j < r1; ++j) {
              const float f = to_f(Xc[col[j] * B + b]);
              acc = acc + f;
              nb += f > thr;
            }
          } else {
#pragma unroll 2
            for (int j = r0; j < r1; ++j) {
              const float f = to_f(Xc[col[j] * B + b]);
              const int w = wts[j];
              ws += w;
              acc = w >= 0 ? acc + f : acc - f;
              nb += f > thr ? w : 0;
            }
          }
          TX xo;
          TV vo;
          step_element<TX, TV>(a, MIS, thr, lo, Xc[idx], V[idx], acc, nb, ws, stepping, xo, vo, zn, c0, c1, c2);
          Xn[idx] = xo;
          V[idx] = vo;
        }
        const unsigned m = __ballot_sync(0xffffffffu, zn);
        if (in && (lane & (GL - 1)) == 0) Zn[vl * Bw + (b >> 5)] = (m >> (lane & ~(GL - 1))) & gmask;
      }
      if (plain && i + 1 < count) {
        // only the last step's evaluation is read
      } else {
        for (int o = B; o < 32; o <<= 1) {
          c0 += __shfl_xor_sync(0xffffffffu, c0, o);
          c1 += __shfl_xor_sync(0xffffffffu, c1, o);
          c2 += __shfl_xor_sync(0xffffffffu, c2, o);
        }
        if (stepping && lane < B) {
          if (c0) atomicAdd(&s_step[3 * b], c0);
          if (c1) atomicAdd(&s_step[3 * b + 1], c1);
          if (c2) atomicAdd(&s_step[3 * b + 2], c2);
        }
      }
    }
    if (flag & 2) {
      for (int pass = 0; pass < 3; ++pass) {
        disc_pass(D, item, pass, s_cnt);
        __syncthreads();
      }
    }
    __syncthreads();
  }

  for (int i = tid; i < pairs; i += nt) {
    static_cast<TX*>(S.X0)[poff + i] = X[0][i];
    static_cast<TX*>(S.X1)[poff + i] = X[1][i];
    static_cast<TV*>(S.V)[poff + i] = V[i];
  }
#pragma unroll
  for (int k = 0; k < 7; ++k)
    for (int i = tid; i < words; i += nt) gZ[k][woff + i] = Z[k * words + i];
  if (tid < B) {
    const int64_t tau = tau0 + tid;
    Counters c;
    c.value = (unsigned long long)(long long)s_step[3 * tid];
    c.a = (unsigned long long)(long long)s_step[3 * tid + 1];
    c.b = (unsigned long long)(long long)s_step[3 * tid + 2];
    c.commits = 0ull;
    if (plain) {
      plain[tau] = c;
    } else {
      c.value += s_cnt[4 * tid];
      c.a += s_cnt[4 * tid + 1];
      c.b += s_cnt[4 * tid + 2];
      c.commits = s_cnt[4 * tid + 3];
      S.cnt[tau] = c;
      S.st[tau] = st[tid];
      S.act[tau] = s_act[tid];
      S.rnd[tau] = s_rnd[tid];
      S.bestv[tau] = st[tid].best;
    }
  }
}

__global__ void k_tick_add(int64_t* tick, int64_t n) { *tick += n; }

cudaError_t launch_small(const SolverDev& S, int count, Counters* plain, int threads, size_t smem, cudaStream_t s) {
  auto run = [&](auto kern) -> cudaError_t {
    cudaError_t e = allow_smem(kern, kSmallSmemLimit);
    if (e != cudaSuccess) return e;
    kern<<<S.g.num_graphs, threads, smem, s>>>(S, count, plain);
    k_tick_add<<<1, 1, 0, s>>>(S.tick, (int64_t)count);
    return cudaGetLastError();
  };
  auto go = [&](auto tx, auto tv) -> cudaError_t {
    using TX = decltype(tx);
    using TV = decltype(tv);
    return S.p.problem == PROB_MIS ? run(k_small<TX, TV, true>) : run(k_small<TX, TV, false>);
  };
  const int xd = S.p.x_dtype, vd = S.p.v_dtype;
  if (xd == DT_F32) return go(float{}, float{});
  if (xd == DT_BF16 && vd == DT_BF16) return go(__nv_bfloat16{}, __nv_bfloat16{});
  if (xd == DT_BF16 && vd == DT_F32) return go(__nv_bfloat16{}, float{});
  if (xd == DT_F16 && vd == DT_F16) return go(__half{}, __half{});
  if (xd == DT_F16 && vd == DT_F32) return go(__half{}, float{});
  return cudaErrorInvalidValue;
}

}  // namespace mqo
