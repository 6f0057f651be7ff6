// mqo_step_rows.cu -- the fused descent step with 16-bit x, for MIS and for
// MaxCut on f_B, reading neighbour rows straight from L2 (k_step_r).  The step
// itself (gradient, momentum, projection, rounding, exact evaluation) is the
// one of mqo_step.cuh.
//
// Why: while x stays in L2 the staged kernel is bound by issue, 140 lane
// instructions per (node, trajectory) pair of degree 3, most of them in the
// per-element tail.  Here a lane holds 8 trajectories in four words and works
// on words:
//  * a neighbour adds its four words to the sums with mixed-precision adds (one
//    rounding each, CSR order) and its four "in the set" masks to packed 16-bit
//    counts (MIS: to an OR);
//  * MaxCut: with Q the number of neighbours on the set's side (for a weight of
//    -1 the other side counts), As = 2 Q - d, so the fixed-point and gain tests
//    are one packed add and one logic operation per word;
//  * the cut needs only the set's own nodes: summed over a symmetric graph,
//    sum_v [z_v ? W_v - P_v : P_v] = 2 sum_{z_v = 1} (W_v - P_v).
// A row group of B / 8 lanes takes one row and gathers its neighbours' rows
// with 16-byte loads, three in flight.  Bound by the L2 path and its latency at
// 64 registers (32 warps per SM, one wave of CTAs).  Measured (step, degree 3,
// B = 128, MaxCut, BF16): n = 10^5 41 us against 79 of the staged kernel and 80
// of the global-memory one, FP32 V 48 against 103 and 83; n = 10^6 403 against
// 668; n = 10^5, degree 16: 92 against 210 and 185, MIS 85 against 182 and 185.
// Four or eight rows in flight take 43 and 61 us, 48 or 80 registers 49 and 55.
#include "mqo_step.cuh"
#include "mqo_x16.cuh"

namespace mqo {

namespace {

constexpr int kRowThreads = 256;
constexpr int kRowDepth = 3;    // neighbour rows in flight per lane
constexpr int kRowCols = 2048;  // staged column indices per CTA; longer lists are read from global memory

// (a, b) = (a, b) * (x, x) + (y, y), one rounding
__device__ __forceinline__ void fma2(float& a, float& b, float x, float y) {
  asm("{\n\t.reg .b64 p, q, r;\n\t"
      "mov.b64 p, {%0, %1};\n\t"
      "mov.b64 q, {%2, %2};\n\t"
      "mov.b64 r, {%3, %3};\n\t"
      "fma.rn.f32x2 p, p, q, r;\n\t"
      "mov.b64 {%0, %1}, p;\n\t}"
      : "+f"(a), "+f"(b)
      : "f"(x), "f"(y));
}

}  // namespace

// CTA c takes rows [c * per, (c + 1) * per) of the one member graph (per > 0),
// or part c % split of item c / split (per == 0); at most kItemMaxNodes rows
template <typename TX, typename TV, bool MIS, bool WEIGHTED>
__global__ void __launch_bounds__(kRowThreads, 4) k_step_r(StepArgs a, int per) {
  using X = X16<TX>;
  using T2 = typename X::T2;
  __shared__ unsigned long long s_cnt[3 * 128];
  __shared__ int32_t s_rp[kItemMaxNodes + 1];
  __shared__ int32_t s_col[kRowCols];
  __shared__ int8_t s_w[WEIGHTED ? kRowCols : 1];
  int g = 0, v0, v1, rep = blockIdx.x;
  if (per > 0) {
    v0 = blockIdx.x * per;
    v1 = min(a.g.n, v0 + per);
  } else {
    const int it = blockIdx.x / a.split;
    const Item item = a.g.items[it];
    g = item.g;
    rep = it;
    const int part = blockIdx.x - it * a.split;
    const int len = (item.v1 - item.v0 + a.split - 1) / a.split;
    v0 = item.v0 + part * len;
    v1 = min(item.v1, v0 + len);
  }
  const int64_t t = *a.tick;
  if (a.gflag_step && a.gflag_step[g] != (int32_t)(t + 1)) return;
  if (v0 >= v1) return;
  const int B = a.B, nrows = v1 - v0;
  const int32_t* __restrict__ rp = a.g.row_ptr;
  const int32_t* __restrict__ col = a.g.col;
  const int8_t* __restrict__ wts = a.g.w;
  for (int i = threadIdx.x; i < 3 * B; i += kRowThreads) s_cnt[i] = 0ull;
  const int32_t j0 = rp[v0], ncol = min(rp[v1] - j0, kRowCols);
  for (int i = threadIdx.x; i <= nrows; i += kRowThreads) s_rp[i] = rp[v0 + i] - j0;
  for (int i = threadIdx.x; i < ncol; i += kRowThreads) {
    s_col[i] = __ldcs(col + j0 + i);
    if constexpr (WEIGHTED) s_w[i] = wts[j0 + i];
  }
  __syncthreads();

  const int lpr = B / 8, rpw = 32 / lpr;
  const int lane = threadIdx.x & 31, sub = lane / lpr, l = lane - sub * lpr, b0 = l * 8, warp = threadIdx.x >> 5;
  const TX* __restrict__ Xc = static_cast<const TX*>((t & 1) ? a.X1 : a.X0) + b0;
  TX* __restrict__ Xn = static_cast<TX*>((t & 1) ? a.X0 : a.X1) + b0;
  uint32_t* __restrict__ Zn = (t & 1) ? a.ZX0 : a.ZX1;
  TV* __restrict__ V = static_cast<TV*>(a.V) + b0;
  uint32_t stepm = 0u;  // bit e: trajectory b0 + e steps
#pragma unroll
  for (int e = 0; e < 8; ++e)
    stepm |= (uint32_t)(a.act ? (a.act[(int64_t)g * B + b0 + e] & ACT_STEP) != 0 : true) << e;
  const bool all_step = __all_sync(0xffffffffu, stepm == 0xffu);
  const T2 thr2 = X::splat(MIS ? 0.5f : 0.0f), one2 = X::splat(1.0f), low2 = X::splat(MIS ? 0.0f : -1.0f);
  // packed 16-bit sums over the lane's rows.  MaxCut: of a set node's d -
  // (negative entries) and Q, of nodes not fixed and of nodes with a positive
  // gain; MIS: zd of nodes in the set, n1 of those in conflict, n2 of uncovered
  uint32_t zd[4], zq[4], n1[4], n2[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) zd[i] = zq[i] = n1[i] = n2[i] = 0u;

  for (int r0 = warp * rpw; r0 < nrows; r0 += (kRowThreads / 32) * rpw) {
    const int r = r0 + sub;
    const bool has = r < nrows;
    const int rs = has ? s_rp[r] : 0, len = has ? s_rp[r + 1] - rs : 0;
    const int longest = __reduce_max_sync(0xffffffffu, len);
    const int64_t base = (int64_t)(v0 + (has ? r : 0)) * B;
    const uint4 xq = *reinterpret_cast<const uint4*>(Xc + base);
    uint32_t xw[4] = {xq.x, xq.y, xq.z, xq.w}, vw[4];
    float vf[8];
    if constexpr (sizeof(TV) == 2) {
      const uint4 q = *reinterpret_cast<const uint4*>(V + base);
      vw[0] = q.x, vw[1] = q.y, vw[2] = q.z, vw[3] = q.w;
    } else {
      const float4 q0 = reinterpret_cast<const float4*>(V + base)[0], q1 = reinterpret_cast<const float4*>(V + base)[1];
      vf[0] = q0.x, vf[1] = q0.y, vf[2] = q0.z, vf[3] = q0.w, vf[4] = q1.x, vf[5] = q1.y, vf[6] = q1.z, vf[7] = q1.w;
    }
    float acc[8];
    uint32_t cq[4] = {0u, 0u, 0u, 0u};  // Q of the lane's pairs of trajectories; MIS: mask of a neighbour in the set
    int neg = 0;
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[e] = 0.0f;
    for (int k = 0; k < longest; k += kRowDepth) {
      uint4 p[kRowDepth];
      uint32_t sgn[kRowDepth];
#pragma unroll
      for (int q = 0; q < kRowDepth; ++q) {
        // past the row's end: zeros, which leave sums and counts as they are
        p[q] = make_uint4(0u, 0u, 0u, 0u);
        sgn[q] = 0u;
        if (k + q < len) {
          const int j = rs + k + q;
          const int32_t u = j < ncol ? s_col[j] : col[j0 + j];
          if constexpr (WEIGHTED) sgn[q] = (j < ncol ? s_w[j] : wts[j0 + j]) < 0 ? 0xffffffffu : 0u;
          p[q] = *reinterpret_cast<const uint4*>(Xc + (int64_t)u * B);
        }
      }
#pragma unroll
      for (int q = 0; q < kRowDepth; ++q) {
        const uint32_t w[4] = {p[q].x, p[q].y, p[q].z, p[q].w};
        if constexpr (WEIGHTED) neg += sgn[q] & 1u;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t m = __hgt2_mask(as2<T2>(w[i]), thr2) ^ sgn[q];
          if constexpr (MIS) cq[i] |= m;
          else cq[i] += m & 0x00010001u;
          X::add(acc[2 * i], acc[2 * i + 1], WEIGHTED ? w[i] ^ (sgn[q] & 0x80008000u) : w[i]);
        }
      }
    }
    // Q >= t as bit 15 of Q + (0x8000 - t): As >= 0 from t = ceil(d / 2), As > 0
    // from t = floor(d / 2) + 1
    const uint32_t ge0 = (uint32_t)(0x8000 - (len + 1) / 2) * 0x00010001u;
    const uint32_t gt0 = (uint32_t)(0x8000 - (len / 2 + 1)) * 0x00010001u;
    const uint32_t dn = has ? (uint32_t)(len - neg) * 0x00010001u : 0u;
    const uint32_t hb = has ? 0x00010001u : 0u;
    uint32_t zw = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t z = __hgt2_mask(as2<T2>(xw[i]), thr2);
      if constexpr (MIS) {
        zd[i] += z & hb;
        n1[i] += z & cq[i] & hb;
        n2[i] += ~(z | cq[i]) & hb;
      } else {
        const uint32_t g0 = cq[i] + ge0, g1 = cq[i] + gt0;
        zd[i] += z & dn;
        if (has) zq[i] += z & cq[i];
        n1[i] += (~(z ^ g0) >> 15) & hb;                     // set and As >= 0, or not set and As < 0
        n2[i] += (((z & g1) | (~z & ~g0)) >> 15) & hb;       // set and As > 0, or not set and As < 0
      }
      float x0, x1, u0, u1;
      X::unpack(xw[i], x0, x1);
      if constexpr (sizeof(TV) == 2) X::unpack(vw[i], u0, u1);
      else u0 = vf[2 * i], u1 = vf[2 * i + 1];
      float g0f = acc[2 * i], g1f = acc[2 * i + 1];
      if constexpr (MIS) {
        mul2(g0f, g1f, a.gamma, a.gamma);
        g0f = 1.0f - g0f;
        g1f = 1.0f - g1f;
      } else {
        // -lambda - 2 acc: doubling is exact, so one rounding either way
        fma2(g0f, g1f, -2.0f, -a.lambda_);
      }
      mul2(g0f, g1f, a.alpha, a.alpha);
      mul2(u0, u1, a.momentum, a.momentum);
      u0 = u0 + g0f;
      u1 = u1 + g1f;
      add_f32x2(x0, x1, u0, u1);
      T2 xr = as2<T2>(X::pack(x0, x1));
      xr = __hmin2_nan(__hmax2_nan(xr, low2), one2);
      uint32_t xn = *reinterpret_cast<const uint32_t*>(&xr);
      if (all_step) {
        if constexpr (sizeof(TV) == 2) vw[i] = X::pack(u0, u1);
        else vf[2 * i] = u0, vf[2 * i + 1] = u1;
      } else {
        const bool s0 = (stepm >> (2 * i)) & 1u, s1 = (stepm >> (2 * i + 1)) & 1u;
        const uint32_t km = (s0 ? 0u : 0xffffu) | (s1 ? 0u : 0xffff0000u);
        xn = (xn & ~km) | (xw[i] & km);
        if constexpr (sizeof(TV) == 2) {
          vw[i] = (X::pack(u0, u1) & ~km) | (vw[i] & km);
        } else {
          if (s0) vf[2 * i] = u0;
          if (s1) vf[2 * i + 1] = u1;
        }
      }
      xw[i] = xn;
      zw |= __hgt2_mask(as2<T2>(xn), thr2) & ((1u << (2 * i)) | (1u << (17 + 2 * i)));
    }
    uint32_t word = ((zw | (zw >> 16)) & 0xffu) << (b0 & 31);
    word |= __shfl_xor_sync(0xffffffffu, word, 1);
    word |= __shfl_xor_sync(0xffffffffu, word, 2);
    if (has) {
      *reinterpret_cast<uint4*>(Xn + base) = make_uint4(xw[0], xw[1], xw[2], xw[3]);
      if constexpr (sizeof(TV) == 2) {
        *reinterpret_cast<uint4*>(V + base) = make_uint4(vw[0], vw[1], vw[2], vw[3]);
      } else {
        reinterpret_cast<float4*>(V + base)[0] = make_float4(vf[0], vf[1], vf[2], vf[3]);
        reinterpret_cast<float4*>(V + base)[1] = make_float4(vf[4], vf[5], vf[6], vf[7]);
      }
      if ((l & 3) == 0) Zn[(int64_t)(v0 + r) * a.Bw + (b0 >> 5)] = word;
    }
  }
  int c0[8], c1[8], c2[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const int sh = 16 * (e & 1);
    c0[e] = (int)((zd[e >> 1] >> sh) & 0xffffu) - (int)((zq[e >> 1] >> sh) & 0xffffu);
    if constexpr (!MIS) c0[e] *= 2;
    c1[e] = (int)((n1[e >> 1] >> sh) & 0xffffu);
    c2[e] = (int)((n2[e >> 1] >> sh) & 0xffffu);
  }
  flush_step_counters<8>(a, s_cnt, g, rep, b0, lpr, c0, c1, c2, stepm);
}

// a row of x takes 4 to 16 lanes; the packed 16-bit sums hold a lane's share of
// kItemMaxNodes rows of at most 255 entries
bool step_rows_possible(int B, int x_dtype, int problem, int objective, int max_degree) {
  return (B == 32 || B == 64 || B == 128) && x_dtype != DT_F32 &&
         (problem == PROB_MIS || (objective == OBJ_FB && max_degree <= 255));
}

cudaError_t launch_step_rows(const StepArgs& a, int x_dtype, int v_dtype, int sms, cudaStream_t s) {
  StepArgs b = a;
  // one wave of four CTAs per SM where the rows allow it: one member graph's rows
  // are shared out, several graphs' items divided (8 and 16 CTAs per SM of fewer
  // rows: 48 and 57 us against 43, n = 10^5, degree 3, B = 128)
  const int target = 4 * sms;
  int per = 0, grid;
  if (a.g.num_graphs == 1) {
    per = (a.g.n + target - 1) / target;
    per = per < 16 ? 16 : (per > kItemMaxNodes ? kItemMaxNodes : per);
    grid = (a.g.n + per - 1) / per;
  } else {
    b.split = target / a.g.num_items;
    b.split = b.split < 1 ? 1 : (b.split > 8 ? 8 : b.split);
    grid = a.g.num_items * b.split;
  }
  auto go = [&](auto tx, auto tv) -> cudaError_t {
    using TX = decltype(tx);
    using TV = decltype(tv);
    if (a.problem == PROB_MIS) k_step_r<TX, TV, true, false><<<grid, kRowThreads, 0, s>>>(b, per);
    else if (a.g.w) k_step_r<TX, TV, false, true><<<grid, kRowThreads, 0, s>>>(b, per);
    else k_step_r<TX, TV, false, false><<<grid, kRowThreads, 0, s>>>(b, per);
    return cudaGetLastError();
  };
  if (x_dtype == DT_BF16 && v_dtype == DT_BF16) return go(__nv_bfloat16{}, __nv_bfloat16{});
  if (x_dtype == DT_BF16 && v_dtype == DT_F32) return go(__nv_bfloat16{}, float{});
  if (x_dtype == DT_F16 && v_dtype == DT_F16) return go(__half{}, __half{});
  if (x_dtype == DT_F16 && v_dtype == DT_F32) return go(__half{}, float{});
  return cudaErrorInvalidValue;
}

}  // namespace mqo
