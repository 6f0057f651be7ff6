// mqo_step_f32.cu -- the shared-memory step kernel with the sliced-ELL
// neighbour stream (the layout is described in mqo_step_smem.cuh) on x staged as
// float32: float32 x, and 16-bit x of fewer than 32 trajectories (widening is
// exact); MIS, and MaxCut without weights.  The step itself (gradient, momentum,
// projection, rounding, exact evaluation) is the one of mqo_step.cuh.
//
// Bound: the shared-memory reads of the neighbours' rows, 128 bytes per clock
// and SM.  The CSR form of k_step_s also takes a shuffle per neighbour and,
// for MIS, reads rounding words, both through the same path.  Here a lane holds
// four trajectories (one 16-byte read per neighbour), the neighbours' offsets come
// eight at a time from global memory (16 bits each: a vector's load takes four
// wavefronts of that path although eight lanes read the same 16 bytes), and the
// checker's counts come from the gathered values: MIS takes their maximum, MaxCut
// adds 1.0f for each positive one (exact up to 2^24).
// Measured (step, 512 graphs of about 750 nodes, degree 112, B = 32, MIS): 217 us
// against 308 of the CSR form with 8-byte lanes and 272 with 16-byte ones, and 248
// with four 32-bit offsets per vector (145 us are the reads' floor); 400 nodes,
// degree 8: 27 against 37 and 30.  Below 32 trajectories it replaces the staged
// and global-memory kernels: 345 graphs of 300 nodes, degree 150, B = 16: 78 us
// against 386 and 269 (BF16 79 against 233 and 209), B = 4: 39 against 126 and 196;
// 400 graphs, degree 6, B = 16: 26 against 34 and 44.
#include "mqo_step.cuh"

namespace mqo {

constexpr int kF32Threads = 512;  // two CTAs per SM

// LPR = B / 4 lanes per row, 32 / LPR rows per warp in lockstep
template <typename TX, typename TV, int LPR, bool MIS>
__global__ void __launch_bounds__(kF32Threads, 2)
    k_step_f(StepArgs a, const int4* __restrict__ ell, const int2* __restrict__ ell_pos) {
  extern __shared__ __align__(16) unsigned char smem[];
  constexpr int RPW = 32 / LPR, B = 4 * LPR, BW = (B + 31) / 32, PITCH = B * 4, PER = PITCH / 16;
  const int it = blockIdx.x;
  const Item item = a.g.items[it];
  const int g = item.g;
  const int64_t t = *a.tick;
  if (a.gflag_step && a.gflag_step[g] != (int32_t)(t + 1)) return;
  const int32_t off = a.g.node_off[g];
  const int32_t ng = a.g.node_off[g + 1] - off;
  const size_t xbytes = (size_t)(ng + 1) * PITCH;
  unsigned long long* s_cnt = reinterpret_cast<unsigned long long*>(smem + xbytes);
  // the item's rows in processing order: {node, group's first vector, its half vectors per row, degree}
  int4* s_rows = reinterpret_cast<int4*>(smem + xbytes + 3 * (size_t)B * 8);
  const int nrows = item.v1 - item.v0;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int nwarps = kF32Threads / 32;
  const TX* __restrict__ Xc = static_cast<const TX*>((t & 1) ? a.X1 : a.X0);
  TX* __restrict__ Xn = static_cast<TX*>((t & 1) ? a.X0 : a.X1);
  uint32_t* __restrict__ Zn = (t & 1) ? a.ZX0 : a.ZX1;
  TV* __restrict__ V = static_cast<TV*>(a.V);

  // stage the member graph's block of x and the zero row of the dummy neighbour
  {
    const TX* src = Xc + (int64_t)off * B;
    for (int i = threadIdx.x; i < ng * PER; i += kF32Threads) {
      if constexpr (sizeof(TX) == 4) {
        const uint32_t d = (uint32_t)__cvta_generic_to_shared(smem + 16 * i);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(d), "l"(src + 4 * (int64_t)i) : "memory");
      } else {
        const Pack<TX, 4> q = ld_pack<TX, 4>(src + 4 * (int64_t)i);
        *reinterpret_cast<float4*>(smem + 16 * i) = make_float4(to_f(q.e[0]), to_f(q.e[1]), to_f(q.e[2]), to_f(q.e[3]));
      }
    }
    if (threadIdx.x < PER) reinterpret_cast<int4*>(smem + (size_t)ng * PITCH)[threadIdx.x] = make_int4(0, 0, 0, 0);
    for (int i = threadIdx.x; i < 3 * B; i += kF32Threads) s_cnt[i] = 0ull;
    for (int i = threadIdx.x; i < nrows; i += kF32Threads) {
      const int v = a.g.order[item.v0 + i];
      const int2 ep = ell_pos[item.v0 + i];
      s_rows[i] = make_int4(v, ep.x, ep.y, a.g.row_ptr[v + 1] - a.g.row_ptr[v]);
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
  }
  __syncthreads();

  const int sub = lane / LPR, l = lane - sub * LPR, b0 = 4 * l;
  const float thr = MIS ? 0.5f : 0.0f, lo = MIS ? 0.0f : -1.0f;
  const unsigned char* sXl = smem + 16 * l;
  uint32_t stepm = 0u;  // bit e: trajectory b0 + e steps
#pragma unroll
  for (int e = 0; e < 4; ++e)
    stepm |= (uint32_t)(a.act ? (a.act[(int64_t)g * B + b0 + e] & ACT_STEP) != 0 : true) << e;
  // MIS: all three counts packed in cp (below 2^10 per lane); MaxCut: the last two
  int c0[4] = {0, 0, 0, 0};
  uint32_t cp[4] = {0u, 0u, 0u, 0u};
  // two entries of the dummy neighbour: offsets in units of 16 bytes
  const int dummy = ng * LPR * 0x00010001;
  const int4 none = make_int4(dummy, dummy, dummy, dummy);

  // a ring of two vectors (eight entries each) of a group: loaded during the
  // previous group's tail, refilled two vectors ahead once summed
  int4 e0 = none, e1 = none;
  auto first_vectors = [&](int i) {
    e0 = e1 = none;
    if (i < nrows) {
      const int4 r = s_rows[i];
      const int4* p = ell + r.y + sub;
      if (r.z > 0) e0 = __ldcs(p);
      if (r.z > 2) e1 = __ldcs(p + RPW);
    }
  };
  first_vectors(warp * RPW);
  for (int vb = warp * RPW; vb < nrows; vb += nwarps * RPW) {
    const bool has = vb + sub < nrows;
    const int4 grp = s_rows[vb];  // the group's vectors (same for its rows)
    const int4 row = s_rows[has ? vb + sub : vb];
    const int v = row.x;
    const int64_t base = (int64_t)v * B + b0;
    Pack<TV, 4> vv{};
    if (has) vv = ld_pack_stream<TV, 4>(V + base);
    float acc[4] = {0.f, 0.f, 0.f, 0.f};
    float nb[4] = {0.f, 0.f, 0.f, 0.f};  // MIS: maximum of the neighbours' x; MaxCut: their number in the set
    auto add = [&](int o) {
      const float4 f = *reinterpret_cast<const float4*>(sXl + o);
      add_f32x2(acc[0], acc[1], f.x, f.y);
      add_f32x2(acc[2], acc[3], f.z, f.w);
      if constexpr (MIS) {
        nb[0] = fmaxf(nb[0], f.x);
        nb[1] = fmaxf(nb[1], f.y);
        nb[2] = fmaxf(nb[2], f.z);
        nb[3] = fmaxf(nb[3], f.w);
      } else {
        add_f32x2(nb[0], nb[1], f.x > 0.f ? 1.f : 0.f, f.y > 0.f ? 1.f : 0.f);
        add_f32x2(nb[2], nb[3], f.z > 0.f ? 1.f : 0.f, f.w > 0.f ? 1.f : 0.f);
      }
    };
    auto add2 = [&](int w) {
      add((w & 0xffff) << 4);
      add((int)((uint32_t)w >> 16) << 4);
    };
    const int nhalf = grp.z;  // halves (four entries) of vectors
    const int4* ep = ell + grp.y + sub;
    int c = 0;
    for (; c + 4 <= nhalf; c += 4) {
      const int4 q0 = e0, q1 = e1;
      if (c + 4 < nhalf) e0 = __ldcs(ep + (c / 2 + 2) * RPW);
      add2(q0.x), add2(q0.y), add2(q0.z), add2(q0.w);
      if (c + 6 < nhalf) e1 = __ldcs(ep + (c / 2 + 3) * RPW);
      add2(q1.x), add2(q1.y), add2(q1.z), add2(q1.w);
    }
    if (c < nhalf) add2(e0.x), add2(e0.y);
    if (c + 1 < nhalf) add2(e0.z), add2(e0.w);
    if (c + 2 < nhalf) add2(e1.x), add2(e1.y);
    first_vectors(vb + nwarps * RPW);

    Pack<TX, 4> xv, xo;
    Pack<TV, 4> vo;
    if constexpr (sizeof(TX) == 4) xv = *reinterpret_cast<const Pack<TX, 4>*>(sXl + (size_t)(v - off) * PITCH);
    else xv = ld_pack<TX, 4>(Xc + base);
    unsigned zbits = 0u;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      bool zn;
      int d0 = 0, d1 = 0, d2 = 0;
      const int pos = MIS ? (int)(nb[e] > 0.5f) : (int)nb[e];
      step_element<TX, TV>(a, MIS, thr, lo, xv.e[e], vv.e[e], acc[e], pos, row.w, (stepm >> e) & 1u, xo.e[e], vo.e[e],
                           zn, d0, d1, d2);
      if (has) {
        if constexpr (MIS) {
          cp[e] += (uint32_t)d0 | ((uint32_t)d1 << 10) | ((uint32_t)d2 << 20);
        } else {
          c0[e] += d0;
          cp[e] += ((uint32_t)d1 << 10) | ((uint32_t)d2 << 20);
        }
      }
      zbits |= (unsigned)zn << e;
    }
    if (has) {
      st_pack<TX, 4>(Xn + base, xo);
      st_pack<TV, 4>(V + base, vo);
    }
    unsigned word = zbits << (b0 & 31);
#pragma unroll
    for (int o = 1; o < (LPR < 8 ? LPR : 8); o <<= 1) word |= __shfl_xor_sync(0xffffffffu, word, o);
    if (has && l % 8 == 0) Zn[(int64_t)v * BW + (b0 >> 5)] = word;
  }
  int c1[4], c2[4];
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if constexpr (MIS) c0[e] = (int)(cp[e] & 1023u);
    c1[e] = (int)((cp[e] >> 10) & 1023u);
    c2[e] = (int)(cp[e] >> 20);
  }
  flush_step_counters<4>(a, s_cnt, g, it, b0, LPR, c0, c1, c2, stepm);
}

// The stream: as k_ell_fill (mqo_step_ell.cu) with eight 16-bit entries per
// vector, offsets in units of 16 bytes (an x block is at most 110 KB); pos[..].y
// counts half vectors, and the second half of a group's last vector may be unused.
__global__ void k_ell_fill16(GraphDev g, int rpw, int lpr, const int2* __restrict__ pos, int4* __restrict__ ell) {
  const Item item = g.items[blockIdx.x];
  const int nrows = item.v1 - item.v0;
  const int32_t off = g.node_off[item.g];
  const int dummy = (g.node_off[item.g + 1] - off) * lpr;
  const int ngrp = (nrows + rpw - 1) / rpw;
  for (int i = threadIdx.x; i < ngrp * rpw; i += blockDim.x) {
    const int q = i / rpw, r = i - q * rpw;
    const int2 ep = pos[item.v0 + q * rpw];
    int rs = 0, re = 0;
    if (i < nrows) {
      const int v = g.order[item.v0 + i];
      rs = g.row_ptr[v];
      re = g.row_ptr[v + 1];
    }
    for (int c = 0; c < (ep.y + 1) / 2; ++c) {
      int e[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int j = rs + 8 * c + 2 * k;
        const int lo = j < re ? (g.col[j] - off) * lpr : dummy;
        const int hi = j + 1 < re ? (g.col[j + 1] - off) * lpr : dummy;
        e[k] = lo | (hi << 16);
      }
      ell[(int64_t)ep.x + (int64_t)c * rpw + r] = make_int4(e[0], e[1], e[2], e[3]);
    }
  }
}

cudaError_t launch_ell_fill16(const GraphDev& g, int rpw, int pitch, const int2* pos, int4* ell, cudaStream_t s) {
  if (g.num_items <= 0) return cudaSuccess;
  k_ell_fill16<<<g.num_items, 256, 0, s>>>(g, rpw, pitch / 16, pos, ell);
  return cudaGetLastError();
}

cudaError_t launch_smem_f32_ell(const StepArgs& a, size_t smem, bool mis, const int4* ell, const int2* ell_pos,
                                int grid, int x_dtype, int v_dtype, cudaStream_t s) {
  if (!mis && a.g.w != nullptr) return cudaErrorInvalidValue;  // the stream carries no weights
  auto run = [&](auto kern) -> cudaError_t {
    cudaError_t e = allow_smem(kern, kStepSmemLimit);
    if (e != cudaSuccess) return e;
    kern<<<grid, kF32Threads, smem, s>>>(a, ell, ell_pos);
    return cudaGetLastError();
  };
  auto go = [&](auto tx, auto tv) -> cudaError_t {
    using TX = decltype(tx);
    using TV = decltype(tv);
    if (a.B == 4) return mis ? run(k_step_f<TX, TV, 1, true>) : run(k_step_f<TX, TV, 1, false>);
    if (a.B == 8) return mis ? run(k_step_f<TX, TV, 2, true>) : run(k_step_f<TX, TV, 2, false>);
    if (a.B == 16) return mis ? run(k_step_f<TX, TV, 4, true>) : run(k_step_f<TX, TV, 4, false>);
    if constexpr (std::is_same<TX, float>::value) {
      if (a.B == 32) return mis ? run(k_step_f<TX, TV, 8, true>) : run(k_step_f<TX, TV, 8, false>);
      if (a.B == 64) return mis ? run(k_step_f<TX, TV, 16, true>) : run(k_step_f<TX, TV, 16, false>);
    }
    return cudaErrorInvalidValue;
  };
  if (x_dtype == DT_F32) return go(float{}, float{});
  if (x_dtype == DT_BF16 && v_dtype == DT_BF16) return go(__nv_bfloat16{}, __nv_bfloat16{});
  if (x_dtype == DT_BF16 && v_dtype == DT_F32) return go(__nv_bfloat16{}, float{});
  if (x_dtype == DT_F16 && v_dtype == DT_F16) return go(__half{}, __half{});
  if (x_dtype == DT_F16 && v_dtype == DT_F32) return go(__half{}, float{});
  return cudaErrorInvalidValue;
}

}  // namespace mqo
