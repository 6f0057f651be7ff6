// mqo_disc_bits.cu -- the discrete passes of a tick (repair and local-search
// rounds, then the counts of the work set) for member graphs with bit matrices
// (mqo_step_dense.cuh).  Same rounds and results as k_disc and k_disc_graph:
// repair = Def. 2.1 feasibility + maximality; rounds of (1,2)-swaps (Def. 2.3),
// 1-flips (Def. 2.4) and 2-flips (Def. 2.5).
//
// Why: in a tick few trajectories are in a round (about 1 in 100 at steady
// state, more while descents end together), but the list kernels walk every
// node's neighbour list for all 32 trajectories of a word as soon as one of
// them is: 37 us a tick for 512 graphs of 750 nodes, 56 us (three launches) for
// 8 graphs of 1000 nodes with 128 trajectories.  Here the work follows the
// trajectories in a round: their sets are bit vectors over the nodes in the
// column order of the adjacency words, a row's count is popc(row & set), and
// a row is read once for kDbBatch trajectories.  Bound by the latency of the
// rows' words (L2) and of the block barriers.
//
// One CTA per (member graph, word of 32 trajectories), or a CTA takes several
// words of its graph where the graphs are many (disc_bits_ctas).
#include "mqo_dev.cuh"
#include "mqo_host.h"

namespace mqo {

namespace {

constexpr int kDbThreads = 512;
constexpr int kDbBatch = 4;    // trajectories processed together
constexpr int kDbWords = 64;   // words of a bit vector: member graphs of at most 2048 nodes
constexpr int32_t kNoOwner = 0x7fffffff;

// the column order of the adjacency words: element e of a word is bit perm(e)
__device__ __forceinline__ int perm(int e) { return (e >> 1) + 16 * (e & 1); }
__device__ __forceinline__ int unperm(int p) { return p < 16 ? 2 * p : 2 * (p - 16) + 1; }
// bits of the elements below e
__device__ __forceinline__ uint32_t below(int e) {
  return ((1u << ((e + 1) >> 1)) - 1u) | (((1u << (e >> 1)) - 1u) << 16);
}
__device__ __forceinline__ uint32_t natural(uint32_t x) {
  uint32_t t = (x ^ (x >> 8)) & 0x0000FF00u;
  x ^= t ^ (t << 8);
  t = (x ^ (x >> 4)) & 0x00F000F0u;
  x ^= t ^ (t << 4);
  t = (x ^ (x >> 2)) & 0x0C0C0C0Cu;
  x ^= t ^ (t << 2);
  t = (x ^ (x >> 1)) & 0x22222222u;
  x ^= t ^ (t << 1);
  return x;
}

struct BitRows {
  const uint32_t* bits;  // the member graph's words
  int nc;                // 128-column pieces per row
  __device__ __forceinline__ uint4 piece(int v, int c) const {
    return __ldg(reinterpret_cast<const uint4*>(bits) + ((v >> 7) * nc + c) * 128 + (v & 127));
  }
  __device__ __forceinline__ uint32_t word(int v, int w) const {
    return __ldg(bits + 4 * (((v >> 7) * nc + (w >> 2)) * 128 + (v & 127)) + (w & 3));
  }
};

// first element (natural order) of the warp's words: lane l holds words l and
// 32 + l in natural bit order; -1 if all are zero
__device__ __forceinline__ int warp_first(uint32_t a, uint32_t b) {
  unsigned m = __ballot_sync(0xffffffffu, a != 0u);
  if (m) {
    const int src = __ffs(m) - 1;
    return 32 * src + __ffs(__shfl_sync(0xffffffffu, a, src)) - 1;
  }
  m = __ballot_sync(0xffffffffu, b != 0u);
  if (m) {
    const int src = __ffs(m) - 1;
    return 1024 + 32 * src + __ffs(__shfl_sync(0xffffffffu, b, src)) - 1;
  }
  return -1;
}

}  // namespace

__global__ void __launch_bounds__(kDbThreads) k_disc_bits(SolverDev S, const uint4* __restrict__ bits,
                                                          const int64_t* __restrict__ bits_off) {
  extern __shared__ __align__(16) unsigned char smem[];
  __shared__ uint32_t vz[kDbBatch][kDbWords], va[kDbBatch][kDbWords], vf[kDbBatch][kDbWords], vp[kDbBatch][kDbWords];
  __shared__ int s_cnt[32][4];
  __shared__ int s_props[kDbBatch];
  const int parts = gridDim.x / S.g.num_graphs, g = blockIdx.x / parts;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kWarps = kDbThreads / 32;
  const int64_t t = *S.tick;
  if (S.any[1] != (int32_t)(t + 1)) return;
  if (S.gflag[S.g.num_graphs + g] != (int32_t)(t + 1)) return;
  const int B = S.B, Bw = S.Bw;
  const bool mis = S.p.problem == PROB_MIS;
  const int32_t off = S.g.node_off[g];
  const int n = S.g.node_off[g + 1] - off;
  const int words = (n + 31) >> 5;
  const BitRows rows{reinterpret_cast<const uint32_t*>(bits + bits_off[g]), (n + 127) >> 7};
  uint32_t* sW = reinterpret_cast<uint32_t*>(smem);
  uint32_t* sA = sW + n;
  uint32_t* sF = sA + n;
  int32_t* owner = reinterpret_cast<int32_t*>(sF + n);        // [kDbBatch][n]
  int32_t* gain = owner + kDbBatch * n;                       // [kDbBatch][n] (MaxCut)
  uint32_t* prop = reinterpret_cast<uint32_t*>(gain + (mis ? 0 : kDbBatch * n));  // [kDbBatch][n]: two ends
  uint16_t* propv = reinterpret_cast<uint16_t*>(prop + kDbBatch * n);             // [kDbBatch][n]: proposer
  for (int wk = blockIdx.x % parts; wk < Bw; wk += parts) {
    const int myround = S.rnd[(int64_t)g * B + wk * 32 + lane];
    unsigned active = __ballot_sync(0xffffffffu, myround != RD_NONE);
    if (!active) continue;
    for (int v = threadIdx.x; v < n; v += kDbThreads) {
      const int64_t i = (int64_t)(off + v) * Bw + wk;
      sW[v] = S.Zwork[i];
      sA[v] = S.Zaux[i];
      sF[v] = S.Zfree[i];
    }
    for (int i = threadIdx.x; i < 128; i += kDbThreads) s_cnt[i >> 2][i & 3] = 0;
    __syncthreads();

    while (active) {
      int b[kDbBatch], rd[kDbBatch];
      int nb = 0;
#pragma unroll
      for (int k = 0; k < kDbBatch; ++k) {
        b[k] = 0;
        rd[k] = RD_NONE;
        if (active) {
          b[k] = __ffs(active) - 1;
          rd[k] = __shfl_sync(0xffffffffu, myround, b[k]);
          active &= active - 1u;
          nb = k + 1;
        }
      }
      bool listed = false, rounds = false;
#pragma unroll
      for (int k = 0; k < kDbBatch; ++k) {
        listed |= rd[k] == RD_SWAP || rd[k] == RD_FLIP2;
        rounds |= rd[k] == RD_DROP || rd[k] == RD_COMPLETE || rd[k] == RD_FLIP1;
      }
      // the sets of the batch as bit vectors over the nodes
      for (int w = warp; w < kDbWords; w += kWarps) {
        const int v = 32 * w + unperm(lane);
        const bool in = v < n;
        const uint32_t xw = in ? sW[v] : 0u, xa = in ? sA[v] : 0u, xf = in ? sF[v] : 0u;
#pragma unroll
        for (int k = 0; k < kDbBatch; ++k) {
          const unsigned mz = __ballot_sync(0xffffffffu, (xw >> b[k]) & 1u);
          const unsigned ma = __ballot_sync(0xffffffffu, (xa >> b[k]) & 1u);
          const unsigned mf = __ballot_sync(0xffffffffu, (xf >> b[k]) & 1u);
          if (lane == 0) vz[k][w] = mz, va[k][w] = ma, vf[k][w] = mf, vp[k][w] = 0u;
        }
      }
      if (threadIdx.x < kDbBatch) s_props[threadIdx.x] = 0;
      if (listed)
        for (int v = threadIdx.x; v < n; v += kDbThreads)
#pragma unroll
          for (int k = 0; k < kDbBatch; ++k) {
            owner[k * n + v] = kNoOwner;
            if (rd[k] == RD_FLIP2) gain[k * n + v] = S.gain[(int64_t)(off + v) * B + wk * 32 + b[k]];
          }
      __syncthreads();

      // ---------------- pass A: decisions on the snapshot
      uint32_t change[(2048 + kDbThreads - 1) / kDbThreads];  // per own row: bit k = this row's bit changes
      if (rounds) {
#pragma unroll
        for (int q = 0; q < (2048 + kDbThreads - 1) / kDbThreads; ++q) change[q] = 0u;
#pragma unroll
        for (int q = 0; q < (2048 + kDbThreads - 1) / kDbThreads; ++q) {
          const int v = threadIdx.x + q * kDbThreads;
          if (v >= n) break;
          const int wv = v >> 5;
          const uint32_t pb = 1u << perm(v & 31), lt = below(v & 31);
          bool some[kDbBatch];  // some smaller neighbour in the round's set
#pragma unroll
          for (int k = 0; k < kDbBatch; ++k) some[k] = false;
          for (int c = 0; 4 * c <= wv; ++c) {
            const uint4 r4 = rows.piece(v, c);
            const uint32_t r[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              const int w = 4 * c + e;
              const uint32_t m = w < wv ? r[e] : (w == wv ? r[e] & lt : 0u);
#pragma unroll
              for (int k = 0; k < kDbBatch; ++k) {
                const uint32_t* src = rd[k] == RD_DROP ? vz[k] : rd[k] == RD_COMPLETE ? vf[k] : va[k];
                some[k] |= (m & src[w]) != 0u;
              }
            }
          }
#pragma unroll
          for (int k = 0; k < kDbBatch; ++k) {
            bool ch = false;
            if (rd[k] == RD_DROP) ch = (vz[k][wv] & pb) && some[k];
            else if (rd[k] == RD_COMPLETE) ch = (vf[k][wv] & pb) && !some[k];
            else if (rd[k] == RD_FLIP1) ch = (va[k][wv] & pb) && !some[k];
            change[q] |= (uint32_t)ch << k;
          }
        }
      }
#pragma unroll
      for (int k = 0; k < kDbBatch; ++k) {
        if (rd[k] == RD_SWAP) {
          // a warp per set node v: the first pair (in CSR order of N(v)) of
          // non-adjacent tight neighbours
          int task = 0;
          for (int w = 0; w < words; ++w) {
            uint32_t m = vz[k][w];
            while (m) {
              const int v = 32 * w + unperm(__ffs(m) - 1);
              m &= m - 1u;
              if (task++ % kWarps != warp) continue;
              uint32_t r0 = lane < words ? natural(rows.word(v, lane) & va[k][lane]) : 0u;
              uint32_t r1 = 32 + lane < words ? natural(rows.word(v, 32 + lane) & va[k][32 + lane]) : 0u;
              int fa, fb = -1;
              while ((fa = warp_first(r0, r1)) >= 0) {
                if ((fa >> 5) == lane) r0 &= r0 - 1u;
                if ((fa >> 5) == 32 + lane) r1 &= r1 - 1u;
                const uint32_t n0 = lane < words ? r0 & ~natural(rows.word(fa, lane)) : 0u;
                const uint32_t n1 = 32 + lane < words ? r1 & ~natural(rows.word(fa, 32 + lane)) : 0u;
                fb = warp_first(n0, n1);
                if (fb >= 0) break;
              }
              if (fb >= 0 && lane == 0) {
                owner[k * n + fa] = v;
                owner[k * n + fb] = v;
                atomicOr(&vp[k][fa >> 5], 1u << perm(fa & 31));
                atomicOr(&vp[k][fb >> 5], 1u << perm(fb & 31));
                const int i = atomicAdd(&s_props[k], 1);
                prop[k * n + i] = (uint32_t)fa | ((uint32_t)fb << 16);
                propv[k * n + i] = (uint16_t)v;
              }
            }
          }
        } else if (rd[k] == RD_FLIP2) {
          // node v proposes its first neighbour u > v on the other side with a
          // positive pair gain
          for (int v = threadIdx.x; v < n; v += kDbThreads) {
            const int wv = v >> 5;
            const bool zv = (vz[k][wv] >> perm(v & 31)) & 1u;
            const int ga = gain[k * n + v];
            int fu = -1;
            for (int c = wv >> 2; c < rows.nc && fu < 0; ++c) {
              const uint4 r4 = rows.piece(v, c);
              const uint32_t r[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const int w = 4 * c + e;
                if (w < wv || fu >= 0) continue;
                uint32_t m = r[e] & (zv ? ~vz[k][w] : vz[k][w]);
                if (w == wv) m &= ~(below(v & 31) | (1u << perm(v & 31)));
                m = natural(m);
                while (m) {
                  const int u = 32 * w + __ffs(m) - 1;
                  m &= m - 1u;
                  if (ga + gain[k * n + u] + 2 > 0) {
                    fu = u;
                    break;
                  }
                }
              }
            }
            if (fu >= 0) {
              atomicMin(&owner[k * n + v], v);
              atomicMin(&owner[k * n + fu], v);
              atomicOr(&vp[k][wv], 1u << perm(v & 31));
              atomicOr(&vp[k][fu >> 5], 1u << perm(fu & 31));
              const int i = atomicAdd(&s_props[k], 1);
              prop[k * n + i] = (uint32_t)v | ((uint32_t)fu << 16);
              propv[k * n + i] = (uint16_t)v;
            }
          }
        }
      }
      __syncthreads();

      // ---------------- pass B: commits
      if (rounds) {
#pragma unroll
        for (int q = 0; q < (2048 + kDbThreads - 1) / kDbThreads; ++q) {
          const int v = threadIdx.x + q * kDbThreads;
          if (v >= n) break;
#pragma unroll
          for (int k = 0; k < kDbBatch; ++k)
            if ((change[q] >> k) & 1u) {
              atomicXor(&vz[k][v >> 5], 1u << perm(v & 31));  // drops clear, completions set, flips toggle
              atomicAdd(&s_cnt[b[k]][3], 1);
            }
        }
      }
      if (listed) {
#pragma unroll
        for (int k = 0; k < kDbBatch; ++k) {
          const bool flip2 = rd[k] == RD_FLIP2;
          if (rd[k] != RD_SWAP && !flip2) continue;
          // a proposal commits if no neighbour of its two ends (other than the
          // ends) is claimed by a smaller proposer; a 2-flip also has to hold
          // both its claims
          for (int i = warp; i < s_props[k]; i += kWarps) {
            const int v = propv[k * n + i];
            const int e0 = (int)(prop[k * n + i] & 0xffffu), e1 = (int)(prop[k * n + i] >> 16);
            bool bad = flip2 && (owner[k * n + e0] != v || owner[k * n + e1] != v);
            for (int w = lane; w < words; w += 32) {
              uint32_t m = (rows.word(e0, w) | rows.word(e1, w)) & vp[k][w];
              while (m) {
                const int u = 32 * w + unperm(__ffs(m) - 1);
                m &= m - 1u;
                if (u != e0 && u != e1) bad |= owner[k * n + u] < v;
              }
            }
            if (!__any_sync(0xffffffffu, bad) && lane == 0) {
              if (!flip2) atomicXor(&vz[k][v >> 5], 1u << perm(v & 31));
              atomicXor(&vz[k][e0 >> 5], 1u << perm(e0 & 31));
              atomicXor(&vz[k][e1 >> 5], 1u << perm(e1 & 31));
              atomicAdd(&s_cnt[b[k]][3], 1);
            }
          }
        }
      }
      __syncthreads();

      // ---------------- pass C: counts of the (new) work sets
      int acc[kDbBatch][3];
#pragma unroll
      for (int k = 0; k < kDbBatch; ++k) acc[k][0] = acc[k][1] = acc[k][2] = 0;
      for (int v = threadIdx.x; v < n; v += kDbThreads) {
        int cnt[kDbBatch], deg = 0;
#pragma unroll
        for (int k = 0; k < kDbBatch; ++k) cnt[k] = 0;
#pragma unroll 4
        for (int c = 0; c < rows.nc; ++c) {
          const uint4 r4 = rows.piece(v, c);
          const uint32_t r[4] = {r4.x, r4.y, r4.z, r4.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            if (!mis) deg += __popc(r[e]);
#pragma unroll
            for (int k = 0; k < kDbBatch; ++k) cnt[k] += __popc(r[e] & vz[k][4 * c + e]);
          }
        }
        uint32_t xw = sW[v], xa = sA[v], xf = sF[v];
#pragma unroll
        for (int k = 0; k < kDbBatch; ++k) {
          if (k >= nb) break;
          const uint32_t bit = 1u << b[k];
          const bool z = (vz[k][v >> 5] >> perm(v & 31)) & 1u;
          bool aux, fr = false;
          if (mis) {
            const bool one = cnt[k] >= 1;
            acc[k][0] += z;
            acc[k][1] += z && one;
            fr = !z && !one;
            acc[k][2] += fr;
            aux = !z && cnt[k] == 1;  // tight: exactly one neighbour in the set
            xf = fr ? xf | bit : xf & ~bit;
          } else {
            const int as = 2 * cnt[k] - deg;
            acc[k][0] += z ? deg - cnt[k] : cnt[k];
            acc[k][1] += !(z ? as <= -1 : as >= 0);  // f_B rule (Thm 3.6), any objective
            const int gn = z ? as : -as;
            aux = gn > 0;
            acc[k][2] += aux;
            S.gain[(int64_t)(off + v) * B + wk * 32 + b[k]] = gn;
          }
          S.owner[(int64_t)(off + v) * B + wk * 32 + b[k]] = kNoOwner;  // as the list kernels leave it
          xw = z ? xw | bit : xw & ~bit;
          xa = aux ? xa | bit : xa & ~bit;
        }
        sW[v] = xw;
        sA[v] = xa;
        sF[v] = xf;
      }
#pragma unroll
      for (int k = 0; k < kDbBatch; ++k) {
        if (k >= nb) break;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
          const int sum = __reduce_add_sync(0xffffffffu, acc[k][i]);
          if (lane == 0 && sum) atomicAdd(&s_cnt[b[k]][i], sum);
        }
      }
      __syncthreads();
    }

    for (int v = threadIdx.x; v < n; v += kDbThreads) {
      const int64_t i = (int64_t)(off + v) * Bw + wk;
      S.Zwork[i] = sW[v];
      S.Zaux[i] = sA[v];
      S.Zfree[i] = sF[v];
    }
    if (threadIdx.x < 128) {
      const int tb = threadIdx.x >> 2, k = threadIdx.x & 3;
      const int val = s_cnt[tb][k];
      if (val) {
        Counters* c = S.cnt + ((int64_t)g * B + wk * 32 + tb) * S.R;  // replica 0
        unsigned long long* p = k == 0 ? &c->value : k == 1 ? &c->a : k == 2 ? &c->b : &c->commits;
        atomicAdd(p, (unsigned long long)(long long)val);
      }
    }
    __syncthreads();  // before the next word's sets
  }
}

// Exact evaluation of given bits (k_eval, mqo_tick.cu) for member graphs with
// bit matrices: one CTA per (member graph, word of 32 trajectories, part of the
// rows); the sets as bit vectors in shared memory, a thread per row, counts by
// popc (64 graphs of 750 nodes, degree 112: 204 us with a load per neighbour and
// trajectory, 36 us now).
__global__ void __launch_bounds__(256) k_eval_bits(SolverDev S, const uint4* __restrict__ bits,
                                                   const int64_t* __restrict__ bits_off, int parts,
                                                   const uint32_t* __restrict__ z, Counters* out) {
  __shared__ __align__(16) uint32_t s_z[32][kDbWords];
  __shared__ int s_cnt[32][3];
  const int part = blockIdx.x % parts;
  const int wk = (blockIdx.x / parts) % S.Bw, g = blockIdx.x / parts / S.Bw;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool mis = S.p.problem == PROB_MIS;
  const int32_t off = S.g.node_off[g];
  const int n = S.g.node_off[g + 1] - off;
  const int tiles = (n + 255) / 256;
  if (part >= tiles) return;
  const BitRows rows{reinterpret_cast<const uint32_t*>(bits + bits_off[g]), (n + 127) >> 7};
  if (threadIdx.x < 96) s_cnt[threadIdx.x / 3][threadIdx.x % 3] = 0;
  for (int w = warp; w < 4 * rows.nc; w += 8) {
    const int v = 32 * w + unperm(lane);
    uint32_t x = v < n ? z[(int64_t)(off + v) * S.Bw + wk] : 0u;
    for (int b = 0; b < 32; ++b) {
      const unsigned m = __ballot_sync(0xffffffffu, (x >> b) & 1u);
      if (lane == b) s_z[b][w] = m;
    }
  }
  __syncthreads();
  for (int tile = part; tile < tiles; tile += parts) {
    const int v = tile * 256 + threadIdx.x;
    const bool in = v < n;
    const uint32_t own = in ? z[(int64_t)(off + v) * S.Bw + wk] : 0u;
    int deg = 0;
    // eight trajectories at a time, so that their counts stay in registers
    for (int b0 = 0; b0 < 32; b0 += 8) {
      int cnt[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) cnt[k] = 0;
      for (int c = 0; in && c < rows.nc; ++c) {
        const uint4 r = rows.piece(v, c);
        if (b0 == 0) deg += __popc(r.x) + __popc(r.y) + __popc(r.z) + __popc(r.w);
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const uint4 m = *reinterpret_cast<const uint4*>(&s_z[b0 + k][4 * c]);
          cnt[k] += __popc(r.x & m.x) + __popc(r.y & m.y) + __popc(r.z & m.z) + __popc(r.w & m.w);
        }
      }
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const bool zv = (own >> (b0 + k)) & 1u;
        int a0, a1, a2;
        if (mis) {
          a0 = zv;
          a1 = zv ? cnt[k] : 0;
          a2 = !zv && cnt[k] == 0;
        } else {
          const int as = 2 * cnt[k] - deg;
          a0 = zv ? deg - cnt[k] : cnt[k];
          a1 = !(zv ? as <= -1 : as >= 0);
          a2 = (zv ? as : -as) > 0;
        }
        a0 = __reduce_add_sync(0xffffffffu, in ? a0 : 0);
        a1 = __reduce_add_sync(0xffffffffu, in ? a1 : 0);
        a2 = __reduce_add_sync(0xffffffffu, in ? a2 : 0);
        if (lane == 0) {
          if (a0) atomicAdd(&s_cnt[b0 + k][0], a0);
          if (a1) atomicAdd(&s_cnt[b0 + k][1], a1);
          if (a2) atomicAdd(&s_cnt[b0 + k][2], a2);
        }
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < 96) {
    const int b = threadIdx.x / 3, k = threadIdx.x % 3;
    const int val = s_cnt[b][k];
    if (val) {
      Counters* c = out + ((int64_t)g * S.B + wk * 32 + b) * S.R;
      atomicAdd(k == 0 ? &c->value : k == 1 ? &c->a : &c->b, (unsigned long long)val);
    }
  }
}

cudaError_t launch_eval_bits(const SolverDev& S, const uint4* bits, const int64_t* bits_off, int max_ng,
                             const uint32_t* z, Counters* out, cudaStream_t stream) {
  const int parts = (max_ng + 255) / 256;
  k_eval_bits<<<S.g.num_graphs * S.Bw * parts, 256, 0, stream>>>(S, bits, bits_off, parts, z, out);
  return cudaGetLastError();
}

size_t disc_bits_smem_bytes(int problem, int max_ng) {
  const size_t n = (size_t)max_ng;
  return n * (3 * 4 + kDbBatch * (4 + 4 + 2 + (problem == PROB_MIS ? 0 : 4))) + 16;
}

// a CTA per member graph and word of trajectories while there are SMs for
// them, else a CTA takes several words (one CTA fits on an SM, and a tick
// without rounds pays for the launch of each: 407 graphs, B = 128: 9.8 us with
// a CTA per word, 7.3 with one per graph)
int disc_bits_ctas(const SolverDev& S, int sms) {
  int parts = S.Bw;
  while (parts > 1 && S.g.num_graphs * parts > sms) parts /= 2;
  return S.g.num_graphs * parts;
}

cudaError_t launch_disc_bits(const SolverDev& S, const uint4* bits, const int64_t* bits_off, size_t smem,
                             int sms, cudaStream_t stream) {
  cudaError_t e = allow_smem(k_disc_bits, kDiscBitsSmemLimit);
  if (e != cudaSuccess) return e;
  k_disc_bits<<<disc_bits_ctas(S, sms), kDbThreads, smem, stream>>>(S, bits, bits_off);
  return cudaGetLastError();
}

}  // namespace mqo
