// mqo_machine.cuh -- device functions of the per-trajectory machine (Alg. 1 /
// Alg. 2) shared by the tick kernels (mqo_tick.cu) and the multi-tick kernel
// of small member graphs (mqo_small.cu): the control decision, the x of resets
// and initialisations, the (node, trajectory) pair frame and the discrete
// passes.
#pragma once

#include "mqo_dev.cuh"
#include "mqo_host.h"

namespace mqo {

// ---------------------------------------------------------------- control
__device__ __forceinline__ void reset_keys(const Params& p, int64_t tau, int32_t o, int32_t r, int32_t n_g,
                                           TrajState& st) {
  const U64x4 k = philox4x64_10(TAG_RESET, (uint64_t)o, (uint64_t)r, 0ULL, p.seed, (uint64_t)tau);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    st.rkeys[2 * i] = (uint32_t)(k.v[i] & 0xffffffffULL);
    st.rkeys[2 * i + 1] = (uint32_t)(k.v[i] >> 32);
  }
  st.rk = (int64_t)floor(p.rho * (double)n_g);
}

// What trajectory tau does in the next tick: folds the counters c of its last
// tick into st and decides the actions and the discrete round (the decisions
// of the oracle's control step).  Modes as CtrlMode; not for a forced reset.
__device__ __forceinline__ void ctrl_decide(const SolverDev& S, int mode, int64_t tau, int g, int32_t n_g,
                                            const Counters& c, TrajState& st, int& act, int& round) {
  const Params& p = S.p;
  const bool mis = p.problem == PROB_MIS;
  act = 0;
  round = RD_NONE;

  auto accept = [&](int bit, int64_t value, bool from_ls) {
    if (value > st.best) {
      credit_gain(st, value, from_ls);
      st.best = value;
      act |= bit;
      st.accepts += 1;
    }
  };

  // fold the previous tick's exact counters (summed and cleared by the
  // caller); in pool mode a trajectory that waited last tick keeps its
  // evaluation
  const bool pool = p.pool_k > 0 && mode == CTRL_MACHINE;
  if (!pool || (st.act & ACT_STEP) || st.round != RD_NONE) {
    const int64_t cv = (int64_t)c.value;
    st.ev_value = mis ? cv : cv / 2;
    st.ev_a = (int64_t)c.a;
    st.ev_b = (int64_t)c.b;
    st.last_commits = (int64_t)c.commits;
  }

  if (mode == CTRL_LS_BEGIN) {
    st.ls_done = 0;
    act = ACT_WORK_BEST;
    round = RD_COUNT;
    st.last_round = RD_COUNT;
  } else if (mode == CTRL_LS) {
    if (!st.ls_done) {
      bool done;
      if (mis) {
        if (st.ev_b > 0) { round = RD_COMPLETE; done = false; }
        else if (!(st.last_round == RD_SWAP && st.last_commits == 0)) { round = RD_SWAP; done = false; }
        else done = true;
      } else {
        if (st.ev_b > 0) { round = RD_FLIP1; done = false; }
        else if (!(st.last_round == RD_FLIP2 && st.last_commits == 0)) { round = RD_FLIP2; done = false; }
        else done = true;
      }
      if (done) {
        accept(ACT_ACC_WORK, st.ev_value, true);
        st.ls_done = 1;
        round = RD_NONE;
      }
      st.last_round = round;
    }
  } else if (pool) {
    // ----- pmQO (Alg. 3/4): the per-trajectory part of the graph's
    // decision of this tick (k_pool_ctrl) -----
    const PoolState ps = S.pool[g];
    const int b = (int)(tau - (int64_t)g * S.B);
    if (ps.best_src >= 0) {  // the graph's best set was replaced (steps 5, 12, 13)
      credit_gain(st, ps.best, ps.best_src >= S.K);
      st.best = ps.best;
      st.accepts += 1;
    }
    auto hold = [&](int bits, int64_t value) {
      act |= bits;
      st.held = value;
      st.phase = PH_WAIT;
    };
    if (st.phase == PH_WAIT) {
      if (ps.dec == DEC_NEXT) {  // steps 6-10 from pool member pbase[tau]
        st.r += 1;
        st.s = 0;
        st.phase = PH_DESCENT;
        reset_keys(p, tau, st.o, st.r, n_g, st);
        act |= ACT_RESET | ACT_POOL;
      } else if (ps.dec == DEC_LS) {  // step 13
        st.held = (int64_t)(-9223372036854775807LL - 1);
        if (mis ? b == 0 : b < ps.count) {
          st.phase = PH_LS;
          act |= mis ? ACT_WORK_BEST : (ACT_WORK_BEST | ACT_POOL);
          round = RD_COUNT;
        }
      } else if (ps.dec == DEC_OUTER) {  // step 2
        st.held = (int64_t)(-9223372036854775807LL - 1);
        st.o += 1;
        st.r = 0;
        st.s = 0;
        st.phase = PH_DESCENT;
        act |= ACT_INIT;
      }
    } else if (st.phase == PH_DESCENT) {
      if (st.s > 0) {
        const bool pass = mis ? (st.ev_a == 0 && st.ev_b == 0) : (st.ev_a == 0);
        if (pass) {
          st.descents += 1;
          hold(ACT_WORK_ZX, st.ev_value);
        } else if (st.s >= p.cap) {
          st.descents += 1;
          if (mis && p.repair) {
            st.phase = PH_REPAIR;
            act |= ACT_WORK_ZX;
            round = RD_COUNT;
          } else {
            // an unrepaired capped MIS point is not a candidate
            hold(ACT_WORK_ZX, mis ? (int64_t)(-9223372036854775807LL - 1) : st.ev_value);
          }
        }
      }
    } else if (st.phase == PH_REPAIR) {
      if (st.ev_a > 0) round = RD_DROP;
      else if (st.ev_b > 0) round = RD_COMPLETE;
      else hold(0, st.ev_value);
    } else if (st.phase == PH_LS) {
      bool done;
      if (mis) {
        if (st.ev_b > 0) { round = RD_COMPLETE; done = false; }
        else if (!(st.last_round == RD_SWAP && st.last_commits == 0)) { round = RD_SWAP; done = false; }
        else done = true;
      } else {
        if (st.ev_b > 0) { round = RD_FLIP1; done = false; }
        else if (!(st.last_round == RD_FLIP2 && st.last_commits == 0)) { round = RD_FLIP2; done = false; }
        else done = true;
      }
      if (done) {
        hold(0, st.ev_value);
        round = RD_NONE;
      }
    }
    if (st.phase == PH_DESCENT) {
      act |= ACT_STEP;
      st.s += 1;
      st.steps += 1;
      st.last_round = RD_NONE;
      round = RD_NONE;
    } else if (round != RD_NONE) {
      st.last_round = round;
    }
    st.ticks += 1;
  } else {
    // ----- the machine (same decisions as the oracle's control step) -----
    auto start_outer = [&]() {
      st.o += 1;
      st.r = 0;
      st.s = 0;
      st.phase = PH_DESCENT;
      act |= ACT_INIT;
    };
    auto after_accept = [&]() -> int {
      if (st.r < p.t_gs) {
        st.r += 1;
        st.s = 0;
        st.phase = PH_DESCENT;
        reset_keys(p, tau, st.o, st.r, n_g, st);
        act |= ACT_RESET;
        return RD_NONE;
      }
      if (p.local_search) {
        st.phase = PH_LS;
        act |= ACT_WORK_BEST;
        return RD_COUNT;
      }
      start_outer();
      return RD_NONE;
    };
    if (st.phase == PH_DESCENT) {
      if (st.s > 0) {
        const bool pass = mis ? (st.ev_a == 0 && st.ev_b == 0) : (st.ev_a == 0);
        if (pass) {
          st.descents += 1;
          accept(ACT_ACC_ZX, st.ev_value, false);
          round = after_accept();
        } else if (st.s >= p.cap) {
          st.descents += 1;
          if (mis) {
            if (p.repair) {
              st.phase = PH_REPAIR;
              act |= ACT_WORK_ZX;
              round = RD_COUNT;
            } else {
              round = after_accept();
            }
          } else {
            accept(ACT_ACC_ZX, st.ev_value, false);
            round = after_accept();
          }
        }
      }
    } else if (st.phase == PH_REPAIR) {
      if (st.ev_a > 0) round = RD_DROP;
      else if (st.ev_b > 0) round = RD_COMPLETE;
      else {
        accept(ACT_ACC_WORK, st.ev_value, false);
        round = after_accept();
      }
    } else if (st.phase == PH_LS) {
      bool done;
      if (mis) {
        if (st.ev_b > 0) { round = RD_COMPLETE; done = false; }
        else if (!(st.last_round == RD_SWAP && st.last_commits == 0)) { round = RD_SWAP; done = false; }
        else done = true;
      } else {
        if (st.ev_b > 0) { round = RD_FLIP1; done = false; }
        else if (!(st.last_round == RD_FLIP2 && st.last_commits == 0)) { round = RD_FLIP2; done = false; }
        else done = true;
      }
      if (done) {
        accept(ACT_ACC_WORK, st.ev_value, true);
        start_outer();
        round = RD_NONE;
      }
    }
    if (st.phase == PH_DESCENT) {
      act |= ACT_STEP;
      st.s += 1;
      st.steps += 1;
      st.last_round = RD_NONE;
      round = RD_NONE;
    } else {
      st.last_round = round;
    }
    st.ticks += 1;
  }
}

// x of a node after a reset: the base set with the nodes of R (the first rk of
// the keyed permutation) at 0
__device__ __forceinline__ float reset_x(bool mis, bool base, uint32_t n_g, const uint32_t* keys, int64_t rk,
                                         uint32_t vl) {
  const float x = base ? 1.0f : (mis ? 0.0f : -1.0f);
  // v in R sets x_v = 0: only needed where x_v is not 0 already (for
  // MIS the nodes of the base set, a few percent of the graph)
  if (x != 0.0f && (int64_t)feistel_sigma(n_g, keys, vl) < rk) return 0.0f;
  return x;
}

// x of a fresh initialisation (Alg. 1/2 step 2): node vl of degree d
__device__ __forceinline__ float init_x(const Params& p, int32_t outer, uint32_t vl, int64_t tau, int32_t d,
                                        int32_t dmax) {
  const bool mis = p.problem == PROB_MIS;
  const U64x4 r = philox4x64_10(TAG_INIT, (uint64_t)outer, (uint64_t)vl, 0ULL, p.seed, (uint64_t)tau);
  const float lo = mis ? 0.0f : -1.0f, hi = 1.0f;
  if (p.init_kind == 0) {
    const float u = unit24(r.v[0]);
    return lo + (hi - lo) * u;
  }
  const float q = dmax > 0 ? (float)d / (float)dmax : 0.0f;
  float base = 1.0f - q;
  if (!mis) base = 2.0f * base - 1.0f;
  float s = unit24(r.v[0]) + unit24(r.v[1]);
  s = s + unit24(r.v[2]);
  s = s + unit24(r.v[3]);
  s = s - 2.0f;
  float eps = s * 1.7320508075688772f;
  eps = p.sigma * eps;
  return clamp_box(base + eps, lo, hi);
}

// ------------------------------------------------------- pair-kernel frame
struct PairCtx {
  int g;
  int64_t v;
  int b;
  int64_t tau;
  bool in;
  int gl;          // lane within the word group
  int G;           // group size min(B, 32)
  unsigned gmask;  // lanes of the group
  int wk;          // word index of the group inside the node
};

// Walk the (node, trajectory) pairs of one item; warp w covers pair
// indices [v0*B + 32k, ...) so that each group holds one whole bit word.
// `body(ctx)` is called by all 32 lanes together.
template <typename Body>
__device__ __forceinline__ void item_pairs(const SolverDev& S, const Item& item, Body body) {
  const int B = S.B;
  const int lane = threadIdx.x & 31;
  const int G = B < 32 ? B : 32;
  const int gbase = lane & ~(G - 1);
  const unsigned gmask = G == 32 ? 0xffffffffu : (((1u << G) - 1u) << gbase);
  const int64_t lo = (int64_t)item.v0 * B, hi = (int64_t)item.v1 * B;
  for (int64_t base = lo + (threadIdx.x & ~31); base < hi; base += blockDim.x) {
    const int64_t idx = base + lane;
    PairCtx c;
    c.in = idx < hi;
    c.v = c.in ? idx / B : (int64_t)item.v0;
    c.b = (int)(idx % B);
    c.g = item.g;
    c.tau = (int64_t)item.g * B + c.b;
    c.gl = lane - gbase;
    c.G = G;
    c.gmask = gmask;
    c.wk = c.b >> 5;
    body(c);
  }
}

// OR over the neighbours u of v (only u < v if `less`) of word wk, computed
// by the lanes of a group together.
__device__ __forceinline__ uint32_t group_nb_or(const SolverDev& S, const uint32_t* words, const PairCtx& c,
                                                bool less) {
  const int32_t* rp = S.g.row_ptr;
  const int32_t* col = S.g.col;
  uint32_t r = 0u;
  for (int32_t j = rp[c.v] + c.gl; j < rp[c.v + 1]; j += c.G) {
    const int32_t u = col[j];
    if (less && u >= c.v) break;  // rows are sorted ascending
    r |= words[(int64_t)u * S.Bw + c.wk];
  }
  for (int o = 1; o < c.G; o <<= 1) r |= __shfl_xor_sync(c.gmask, r, o);
  return r;
}

__device__ __forceinline__ void set_bit_atomic(uint32_t* words, int64_t v, int Bw, int b, bool val) {
  uint32_t* wp = words + v * Bw + (b >> 5);
  const uint32_t bit = 1u << (b & 31);
  if (val) atomicOr(wp, bit);
  else atomicAnd(wp, ~bit);
}

// ---------------------------------------------------------------- discrete rounds
// One discrete pass over the pairs of an item: 0 = A (decide / propose),
// 1 = B (commit), 2 = C (count); adds into s_cnt[4 * trajectory + counter].
__device__ __forceinline__ void disc_pass(const SolverDev& S, const Item& item, int pass, unsigned long long* s_cnt) {
  const int B = S.B, Bw = S.Bw;
  const bool mis = S.p.problem == PROB_MIS;
  const int32_t* rp = S.g.row_ptr;
  const int32_t* col = S.g.col;
  const int8_t* wts = S.g.w;
  long long acc0 = 0, acc1 = 0, acc2 = 0, acc3 = 0;
  int my_b = (int)(threadIdx.x % B);
  item_pairs(S, item, [&](const PairCtx& c) {
    const int64_t v = c.v;
    const int b = c.b;
    const int round = c.in ? S.rnd[c.tau] : RD_NONE;
    const int64_t e = v * B + b;
    const int32_t rs = rp[v], re = rp[v + 1];
    const uint32_t bit = 1u << (b & 31);
    if (pass == 0) {
      // ---------------- pass A
      const bool zv = get_bit(S.Zwork, v, Bw, b);
      const bool need_drop = __any_sync(c.gmask, round == RD_DROP);
      const bool need_comp = __any_sync(c.gmask, round == RD_COMPLETE);
      const bool need_flip = __any_sync(c.gmask, round == RD_FLIP1);
      bool dropv = false, addv = false, flipv = false;
      if (need_drop) {
        const uint32_t o = group_nb_or(S, S.Zwork, c, true);
        dropv = round == RD_DROP && zv && (o & bit);
      }
      if (need_comp) {
        const uint32_t o = group_nb_or(S, S.Zfree, c, true);
        addv = round == RD_COMPLETE && get_bit(S.Zfree, v, Bw, b) && !(o & bit);
      }
      if (need_flip) {
        const uint32_t o = group_nb_or(S, S.Zaux, c, true);
        flipv = round == RD_FLIP1 && get_bit(S.Zaux, v, Bw, b) && !(o & bit);
      }
      update_word(S.Zdrop, v, Bw, b, B, dropv, round == RD_DROP);
      // complete sets bits, flip1 toggles: both are own-word updates
      update_word(S.Zwork, v, Bw, b, B, addv ? true : !zv, addv || flipv);
      acc3 += dropv + addv + flipv;
      if (round == RD_SWAP) {
        int32_t fa = -1, fb = -1;
        if (zv) {
          for (int32_t i = rs; i < re && fa < 0; ++i) {
            const int32_t a = col[i];
            if (!get_bit(S.Zaux, a, Bw, b)) continue;
            for (int32_t j = i + 1; j < re; ++j) {
              const int32_t cc = col[j];
              if (!get_bit(S.Zaux, cc, Bw, b)) continue;
              if (!sorted_contains(col, rp[a], rp[a + 1], cc)) { fa = a; fb = cc; break; }
            }
          }
        }
        S.pa[e] = fa;
        S.pb[e] = fb;
        if (fa >= 0) {
          S.owner[(int64_t)fa * B + b] = (int32_t)v;
          S.owner[(int64_t)fb * B + b] = (int32_t)v;
        }
      }
      if (round == RD_FLIP2) {
        int32_t fb = -1;
        const int32_t ga = S.gain[e];
        for (int32_t j = rs; j < re; ++j) {
          const int32_t u = col[j];
          if (u <= v) continue;
          if (get_bit(S.Zwork, u, Bw, b) == zv) continue;
          const int w = wts ? (int)wts[j] : 1;
          if (ga + S.gain[(int64_t)u * B + b] + 2 * w > 0) { fb = u; break; }
        }
        S.pb[e] = fb;
        if (fb >= 0) {
          atomicMin(&S.owner[e], (int32_t)v);
          atomicMin(&S.owner[(int64_t)fb * B + b], (int32_t)v);
        }
      }
    } else if (pass == 1) {
      // ---------------- pass B
      const bool dv = round == RD_DROP && get_bit(S.Zdrop, v, Bw, b);
      update_word_atomic(S.Zwork, v, Bw, b, B, false, dv);
      if (round == RD_SWAP) {
        const int32_t fa = S.pa[e];
        if (fa >= 0) {
          const int32_t fb = S.pb[e];
          bool ok = true;
          const int32_t ends[2] = {fa, fb};
          for (int k = 0; k < 2 && ok; ++k) {
            const int32_t x = ends[k];
            for (int32_t j = rp[x]; j < rp[x + 1]; ++j) {
              const int32_t o = S.owner[(int64_t)col[j] * B + b];
              if (o < (int32_t)v) { ok = false; break; }
            }
          }
          if (ok) {
            atomicAnd(&S.Zwork[v * Bw + (b >> 5)], ~bit);
            atomicOr(&S.Zwork[(int64_t)fa * Bw + (b >> 5)], bit);
            atomicOr(&S.Zwork[(int64_t)fb * Bw + (b >> 5)], bit);
            acc3 += 1;
          }
        }
      }
      if (round == RD_FLIP2) {
        const int32_t fb = S.pb[e];
        if (fb >= 0) {
          bool ok = S.owner[e] == (int32_t)v && S.owner[(int64_t)fb * B + b] == (int32_t)v;
          const int32_t ends[2] = {(int32_t)v, fb};
          for (int k = 0; k < 2 && ok; ++k) {
            const int32_t x = ends[k];
            for (int32_t j = rp[x]; j < rp[x + 1]; ++j) {
              const int32_t y = col[j];
              if (y == (int32_t)v || y == fb) continue;
              if (S.owner[(int64_t)y * B + b] < (int32_t)v) { ok = false; break; }
            }
          }
          if (ok) {
            atomicXor(&S.Zwork[v * Bw + (b >> 5)], bit);
            atomicXor(&S.Zwork[(int64_t)fb * Bw + (b >> 5)], bit);
            acc3 += 1;
          }
        }
      }
    } else {
      // ---------------- pass C: counts of the (new) work set
      const bool act = round != RD_NONE;
      const bool zv = get_bit(S.Zwork, v, Bw, b);
      bool aux = false, fr = false;
      if (act) S.owner[e] = 0x7fffffff;
      if (mis) {
        if (__any_sync(c.gmask, act)) {
          // once / twice: neighbours with the bit set at least once / twice
          uint32_t once = 0u, twice = 0u;
          for (int32_t j = rs + c.gl; j < re; j += c.G) {
            const uint32_t w = S.Zwork[(int64_t)col[j] * Bw + c.wk];
            twice |= once & w;
            once |= w;
          }
          for (int o = 1; o < c.G; o <<= 1) {
            const uint32_t o2 = __shfl_xor_sync(c.gmask, once, o);
            const uint32_t t2 = __shfl_xor_sync(c.gmask, twice, o);
            twice = twice | t2 | (once & o2);
            once |= o2;
          }
          if (act) {
            const bool one = (once & bit) != 0, two = (twice & bit) != 0;
            acc0 += zv;
            acc1 += zv && one;
            fr = !zv && !one;
            acc2 += fr;
            aux = !zv && one && !two;  // tight: exactly one neighbour in the set
          }
        }
      } else if (act) {
        int P = 0, W = 0;
        for (int32_t j = rs; j < re; ++j) {
          const int w = wts ? (int)wts[j] : 1;
          W += w;
          if (get_bit(S.Zwork, col[j], Bw, b)) P += w;
        }
        const int as = 2 * P - W;
        acc0 += zv ? (W - P) : P;
        const bool fixed = zv ? (as <= -1) : (as >= 0);  // f_B rule (Thm 3.6), any objective
        acc1 += !fixed;
        const int gn = zv ? as : -as;
        acc2 += gn > 0;
        S.gain[e] = gn;
        aux = gn > 0;
      }
      update_word(S.Zaux, v, Bw, b, B, aux, act);
      update_word(S.Zfree, v, Bw, b, B, fr, act && mis);
    }
  });
  if (acc0) atomicAdd(&s_cnt[4 * my_b + 0], (unsigned long long)acc0);
  if (acc1) atomicAdd(&s_cnt[4 * my_b + 1], (unsigned long long)acc1);
  if (acc2) atomicAdd(&s_cnt[4 * my_b + 2], (unsigned long long)acc2);
  if (acc3) atomicAdd(&s_cnt[4 * my_b + 3], (unsigned long long)acc3);
}

}  // namespace mqo
