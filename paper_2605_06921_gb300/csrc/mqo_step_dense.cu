// mqo_step_dense.cu -- the tensor-core step kernel of dense member graphs
// (k_step_t, mqo_step_dense.cuh) and the bit matrices it reads.
//
// One CTA per (member graph, group of 32 trajectories, part of the row
// tiles).  It stages the graph's x rows of its group once, as the B operand:
// row u (one k) holds 64 16-bit columns, x of the 32 trajectories and their
// companions w, 128 bytes in the 128-byte swizzle, N contiguous -- so staging
// is a copy of 16-byte pieces, no transpose.  A warpgroup then walks row
// tiles of 128: every thread expands 64 adjacency bits of its row per chunk
// into 32 registers of two 16-bit values (0 or 2.0 = 0x4000 in bfloat16 and
// float16 alike: one shift and one AND per two elements), writes them to
// TMEM (tcgen05.st) as the A operand, and one thread issues the MMAs
// (M 128, N 64, K 16) into a 64-column float32 accumulator.  Two A buffers
// per warpgroup and four warpgroups per SM keep expansion, MMA and epilogue
// of different tiles overlapped.  In the epilogue a thread owns one row and
// all 32 trajectories, so the per-trajectory counts come from bit words
// transposed across the warp instead of per-element counters.
#include "mqo_step_dense.cuh"
#include "mqo_x16.cuh"

namespace mqo {

namespace {

// ------------------------------------------------------------ bit matrices
// One warp per row of a tile: the row's words are assembled in shared memory
// and written once.  Word i of the row covers columns 32i .. 32i+31; column
// 2r of it is bit r, column 2r+1 bit 16 + r (the order the MMA kernel
// expands).  Rows past the graph's end are zero.
constexpr int kBitsMaxWords = 64;

__global__ void __launch_bounds__(256) k_dense_bits(GraphDev g, const int64_t* __restrict__ bits_off,
                                                    const int2* __restrict__ tiles, uint32_t* __restrict__ bits) {
  __shared__ uint32_t s_row[8][kBitsMaxWords];
  const int2 tl = tiles[blockIdx.x];  // {member graph, row tile}
  const int32_t off = g.node_off[tl.x];
  const int32_t ng = g.node_off[tl.x + 1] - off;
  const int nc = dense_tiles(ng);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t* out = bits + 4 * (bits_off[tl.x] + (int64_t)tl.y * nc * 128);
  for (int r = warp; r < 128; r += 8) {
    for (int i = lane; i < 4 * nc; i += 32) s_row[warp][i] = 0u;
    __syncwarp();
    const int v = tl.y * 128 + r;
    if (v < ng) {
      const int j1 = g.row_ptr[off + v + 1];
      for (int j = g.row_ptr[off + v] + lane; j < j1; j += 32) {
        const int u = g.col[j] - off;
        const int e = u & 31;
        atomicOr(&s_row[warp][u >> 5], 1u << ((e >> 1) + 16 * (e & 1)));
      }
    }
    __syncwarp();
    for (int i = lane; i < 4 * nc; i += 32) out[4 * ((int64_t)(i >> 2) * 128 + r) + (i & 3)] = s_row[warp][i];
    __syncwarp();
  }
}

// ------------------------------------------------------------ PTX helpers
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
// false if the phase has not ended after `polls` looks (looked at every 256;
// a wait is a few microseconds, kDensePolls looks about a second of running, in
// which time without the context on the GPU does not count)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, uint32_t polls) {
#pragma unroll 1
  for (uint32_t i = 0;; ++i) {
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\t"
                 "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(bar), "r"(parity)
                 : "memory");
    if (ok) return true;
    if ((i & 255u) == 255u) {
      if (i >= polls) return false;
      asm volatile("" ::: "memory");  // keeps the test out of the look's path
    }
  }
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void prefetch_l2_line(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}
// 64 adjacency bits (two words) as 32 pairs of 16-bit values: 0, or a power
// of two A_k that the staged rows make up for, A_k B_k = 2 x.
// float16: every bit goes to bit 14 of its half, 2.0, one shift and one AND
// per pair.  bfloat16 has the exponent range for more: bits 11 .. 14 of a half
// are 2^-111, 2^-95, 2^-63 and 2^1, so one shift serves four pairs and row k
// of B is x times 2^112, 2^96, 2^64 or 1 (shifts and ANDs run at half rate:
// 64 -> 40 instructions a chunk).
template <bool SCALED>
__device__ __forceinline__ void expand_bits(uint32_t w0, uint32_t w1, uint32_t (&r)[32]) {
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    if constexpr (SCALED) {
      const int q = (k + 1) & 3;  // the pair's bits go to bit 11 + q of the halves
      const uint32_t m = 0x08000800u << q;
      const int sh = 11 + q - k;  // 12, 8, 4, 0 or (k = 15) -4
      r[k] = (sh >= 0 ? w0 << (sh & 31) : w0 >> (-sh & 31)) & m;
      r[16 + k] = (sh >= 0 ? w1 << (sh & 31) : w1 >> (-sh & 31)) & m;
    } else {
      r[k] = (k < 15 ? w0 << (14 - k) : w0 >> 1) & 0x40004000u;
      r[16 + k] = (k < 15 ? w1 << (14 - k) : w1 >> 1) & 0x40004000u;
    }
  }
  // keeps the expansion where it is called (between a TMEM write and its wait)
#pragma unroll
  for (int k = 0; k < 32; k += 8)
    asm volatile(""
                 : "+r"(r[k]), "+r"(r[k + 1]), "+r"(r[k + 2]), "+r"(r[k + 3]), "+r"(r[k + 4]), "+r"(r[k + 5]),
                   "+r"(r[k + 6]), "+r"(r[k + 7]));
}
// exponent of the factor of B's row of bit e (0 .. 31) of a column word
__device__ __forceinline__ int row_exponent(int e) {
  const int q = ((e >> 1) + 1) & 3;
  return q == 0 ? 112 : q == 1 ? 96 : q == 2 ? 64 : 0;
}

// biased exponent of the inverse of that factor
__device__ __forceinline__ uint32_t row_inverse(int u) { return (16u << (((u >> 1) + 1) & 3)) - 1u; }

// 32 registers to 32 TMEM columns of the warp's 32 lanes (thread = lane)
__device__ __forceinline__ void tmem_st32(uint32_t addr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(addr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]),
      "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]),
      "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t addr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(addr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(uint32_t addr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(addr));
}
// waits for the loads of r and q; the operands keep their uses behind it
__device__ __forceinline__ void tmem_ld_wait(uint32_t (&r)[16], uint32_t (&q)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                 "+r"(r[8]), "+r"(r[9]), "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])::"memory");
  asm volatile(""
               : "+r"(q[0]), "+r"(q[1]), "+r"(q[2]), "+r"(q[3]), "+r"(q[4]), "+r"(q[5]), "+r"(q[6]), "+r"(q[7]),
                 "+r"(q[8]), "+r"(q[9]), "+r"(q[10]), "+r"(q[11]), "+r"(q[12]), "+r"(q[13]), "+r"(q[14]), "+r"(q[15])::"memory");
}

// true in one lane of a converged warp
__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n\t.reg .pred p;\n\t"
               "elect.sync _|p, 0xffffffff;\n\t"
               "selp.u32 %0, 1, 0, p;\n\t}"
               : "=r"(ok));
  return ok != 0;
}

// D[tmem] (+)= A[tmem] * B[smem]; acc = 0 overwrites D
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile("{\n\t.reg .pred p;\n\t"
               "setp.ne.b32 p, %4, 0;\n\t"
               "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d),
               "r"(a), "l"(bdesc), "r"(idesc), "r"(acc)
               : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// bit order of a trajectory word: trajectory 2i is bit i, 2i + 1 is bit 16 + i
__device__ __forceinline__ int traj_of_bit(int p) { return p < 16 ? 2 * p : 2 * (p - 16) + 1; }
__device__ __forceinline__ uint32_t to_natural(uint32_t x) {
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
// 32 x 32 bit transpose across the warp: bit i of lane j <-> bit j of lane i
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, int lane) {
#pragma unroll
  for (int s = 16; s >= 1; s >>= 1) {
    const uint32_t lo = s == 16 ? 0x0000ffffu : s == 8 ? 0x00ff00ffu : s == 4 ? 0x0f0f0f0fu : s == 2 ? 0x33333333u : 0x55555555u;
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, s);
    x = (lane & s) ? ((x & ~lo) | ((y >> s) & lo)) : ((x & lo) | ((y << s) & ~lo));
  }
  return x;
}

}  // namespace

// ------------------------------------------------------------ the step
template <typename TX, typename TV, bool MIS, int OBJ>
__global__ void __launch_bounds__(kDenseThreads + 32, 2) k_step_t(StepArgs a, DenseArgs d) {
  using X = X16<TX>;
  using T2 = typename X::T2;
  extern __shared__ unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t s_mbar[2][4];  // per warpgroup: A buffers 0 / 1 written, MMAs done with 0 / 1
  __shared__ uint32_t s_tmem;
  __shared__ uint32_t s_cnt[3][32];
  __shared__ uint16_t s_list[kDoubtful];  // doubtful pairs: node << 5 | trajectory bit
  __shared__ int s_listed;
  __shared__ int s_odd[8];                // per warp: small or irregular x staged
  const int part = blockIdx.x % d.parts;
  const int rest = blockIdx.x / d.parts;
  const int tg = rest % d.groups;
  const int g = rest / d.groups;
  const int B = a.B;
  const int64_t t = *a.tick;
  const int32_t flag = a.gflag_step ? a.gflag_step[g] : 0;
  const int32_t off = a.g.node_off[g], end = a.g.node_off[g + 1];
  const int64_t boff = d.bits_off[g];
  const int myact = a.act ? a.act[(int64_t)g * B + tg * kDenseGroup + traj_of_bit(threadIdx.x & 31)] : ACT_STEP;
  if (a.gflag_step && flag != (int32_t)(t + 1)) return;
  const int32_t ng = end - off;
  const int tiles = dense_tiles(ng);
  if (2 * part >= tiles) return;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // warp-uniform, for the compiler too
  const int wg = warp >> 2, wtid = tid & 127;
  unsigned char* sX = smem_raw + ((1024u - (smem_addr(smem_raw) & 1023u)) & 1023u);
  const TX* __restrict__ Xc = static_cast<const TX*>((t & 1) ? a.X1 : a.X0) + (int64_t)off * B + tg * kDenseGroup;
  TX* __restrict__ Xn = static_cast<TX*>((t & 1) ? a.X0 : a.X1) + (int64_t)off * B + tg * kDenseGroup;
  TV* __restrict__ V = static_cast<TV*>(a.V) + (int64_t)off * B + tg * kDenseGroup;
  uint32_t* __restrict__ Zn = ((t & 1) ? a.ZX0 : a.ZX1) + (int64_t)off * a.Bw + tg;

  if (warp == kIssuer) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)),
                 "r"(kDenseTmem)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  }
  if (tid == 32 * kIssuer) {
    for (int i = 0; i < 8; ++i) mbar_init(smem_addr(&s_mbar[i >> 2][i & 3]), (i & 2) ? 1 : 4);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (tid < 96) s_cnt[tid >> 5][tid & 31] = 0u;
  if (tid == 96) s_listed = 0;
  // the first tile's first adjacency words, on their way while x is staged
  const uint4* bits0 = d.bits + boff + wtid;
  const uint4 bfirst = __ldg(bits0 + (int64_t)(2 * part + (2 * part + wg < tiles && wg < 2 ? wg : 0)) * tiles * 128);
  // stage x and its companions: a lane takes a node's 64 bytes; the nodes of
  // a warp are in the bit order of the adjacency words, so that the
  // transposed "not zero" masks line up with them
  const float thr = MIS ? 0.5f : 0.0f;
  const int kpad = (ng + 15) & ~15;
  // behind the block a zero row, then the masks [32 columns][32 trajectories]
  uint32_t* s_nz = reinterpret_cast<uint32_t*>(sX + (size_t)kpad * 128 + 128);
  bool bad = false;  // some x is outside [-1, 1] or not a number (0 in the product)
  int marked = 0;    // small or irregular x
  {
    const T2 thr2 = X::splat(thr), t02 = X::splat(d.t0), one2 = X::splat(1.0f), zero2 = X::splat(0.0f);
    // the factor of this lane's rows of B (expand_bits), a power of two
    const int ex = X::kScaled ? row_exponent(traj_of_bit(lane)) : 0;
    const T2 scale2 = X::splat(__uint_as_float((uint32_t)(127 + ex) << 23));
    const uint32_t half = X::kHalf + ((uint32_t)ex << 7), half2 = half | (half << 16);
    uint32_t xl[16];  // the next node's x, one iteration ahead
    auto load = [&](int u) {
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint4 q = make_uint4(0u, 0u, 0u, 0u);
        if (u < ng) q = reinterpret_cast<const uint4*>(Xc + (int64_t)u * B)[c];
        xl[4 * c] = q.x, xl[4 * c + 1] = q.y, xl[4 * c + 2] = q.z, xl[4 * c + 3] = q.w;
      }
    };
    if (warp != kIssuer) load(warp * 32 + traj_of_bit(lane));
    for (int ub = warp * 32; ub < kpad && warp != kIssuer; ub += kDenseThreads) {
      const int u = ub + traj_of_bit(lane);
      uint32_t xs[16], w[16];
#pragma unroll
      for (int k = 0; k < 16; ++k) xs[k] = xl[k];
      load(u + kDenseThreads);
      uint32_t odd = 0u, nz = 0u;
#pragma unroll
      for (int k = 0; k < 16; ++k) {
        const T2 v = as2<T2>(xs[k]);
        w[k] = __hgt2_mask(v, thr2) & half2;  // 0.5 where x rounds into the set
        const T2 m = MIS ? v : __habs2(v);
        const uint32_t zero = __heq2_mask(m, zero2);
        odd |= ~((__hge2_mask(m, t02) & __hle2_mask(m, one2)) | zero);
        nz |= ~zero & ((1u << k) | (1u << (16 + k)));
      }
      if (odd) {
        // small, tiny, out of the box or not finite: mark the elements
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          uint32_t xn = xs[k], wn = w[k];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            float f0, f1;
            X::unpack((xs[k] >> (16 * h)) & 0xffffu, f0, f1);
            const float m = MIS ? f0 : fabsf(f0);
            const bool fine = (m >= d.t0 && m <= 1.0f) || m == 0.0f;
            const bool fin = fabsf(f0) <= 1.0f;
            if (!fine) {
              ++marked;
              const uint32_t mark = ((MIS && m >= d.t1 && m < d.t0) ? X::kTwo9 : X::kTwo13) + ((uint32_t)ex << 7);
              wn = (wn & ~(0xffffu << (16 * h))) | (mark << (16 * h));
            }
            if (!fin) {
              xn &= ~(0xffffu << (16 * h));
              bad = true;
            }
          }
          xs[k] = xn;
          w[k] = wn;
        }
      }
      if constexpr (X::kScaled) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const T2 v = __hmul2(as2<T2>(xs[k]), scale2);
          xs[k] = *reinterpret_cast<const uint32_t*>(&v);
        }
      }
      if (u < kpad) {
        unsigned char* row = sX + u * 128;
        const int sw = u & 7;
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          *reinterpret_cast<uint4*>(row + ((c ^ sw) << 4)) = make_uint4(xs[4 * c], xs[4 * c + 1], xs[4 * c + 2], xs[4 * c + 3]);
          *reinterpret_cast<uint4*>(row + (((c + 4) ^ sw) << 4)) = make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
        }
      }
      s_nz[ub + lane] = warp_transpose(nz, lane);
    }
  }
  marked = __reduce_add_sync(0xffffffffu, marked);
  if (warp != kIssuer && lane == 0) s_odd[warp] = marked;
  if (tid < 8) *reinterpret_cast<uint4*>(sX + (size_t)kpad * 128 + 16 * tid) = make_uint4(0u, 0u, 0u, 0u);
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  tc_fence_before();
  bad = __syncthreads_or(bad) != 0;
  tc_fence_after();
  // Where a tenth of the pairs would be doubtful (x spread over the whole box,
  // as after a uniform initialisation), or some x is irregular, every row is
  // summed in CSR order from a block staged as it is.
  marked = 0;
#pragma unroll
  for (int i = 0; i < 8; ++i) marked += s_odd[i];
  const bool heavy = bad || (float)marked * d.degree > 3.2f * (float)ng;
  if (heavy) {
    for (int i = tid; i < ng * 4; i += kDenseThreads + 32) {
      const int u = i >> 2, c = i & 3;
      *reinterpret_cast<uint4*>(sX + u * 128 + ((c ^ (u & 7)) << 4)) =
          *reinterpret_cast<const uint4*>(Xc + (int64_t)u * B + c * 8);
    }
    __syncthreads();
  }

  const uint32_t tmem0 = __shfl_sync(0xffffffffu, s_tmem, 0);
  const uint32_t tm = tmem0 + (uint32_t)wg * 128u;
  const uint32_t lsel = (uint32_t)(warp & 3) << 21;  // the warp's 32 TMEM lanes
  const uint32_t idesc = (1u << 4) | (X::kType << 7) | (X::kType << 10) | (1u << 16) | (8u << 17) | (8u << 24);
  // B operand: N contiguous (64 columns = one 128-byte swizzle atom), groups of 8 k 1024 bytes apart
  const uint64_t bdesc0 = (uint64_t)((smem_addr(sX) >> 4) & 0x3fffu) | ((uint64_t)64 << 16) | ((uint64_t)64 << 32) |
                          ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
  const uint32_t bar = smem_addr(&s_mbar[wg & 1][0]);  // + 8 * buffer; + 16 the MMAs-done pair
  const int nk16 = (ng + 15) >> 4, n64 = (ng + 63) >> 6;
  // the trajectories that step this tick (bit order of traj_of_bit)
  const uint32_t stepw = __ballot_sync(0xffffffffu, (myact & ACT_STEP) != 0);
  uint32_t n0 = 0u, n1 = 0u, n2 = 0u;  // counts of trajectory traj_of_bit(lane)
  uint32_t use[2] = {0u, 0u};          // chunks that went through each A buffer
  bool dead = d.polls == 0u;           // a wait ran out: no more waits; this block's results are void
  if (warp == kIssuer) {
    // Issues the MMAs of both warpgroups, chunk by chunk as they are written,
    // in a fixed order (few instructions: the warp shares its scheduler).  An
    // MMA instruction waits for the tensor pipe (32 cycles each at N = 64), so
    // a warp that also expands would hold its warpgroup up.
    if (!heavy && elect_one()) {
      const uint32_t full0 = smem_addr(&s_mbar[0][0]);
      const uint64_t bd0 = bdesc0;
      uint32_t ph = 0u;  // bit 2 w + buf: phase of the warpgroup's written barrier
      auto issue = [&](int w, int buf, int c, int nk) {
        const uint32_t full = full0 + 32u * w + 8u * buf;
        if (!dead && !mbar_wait(full, (ph >> (2 * w + buf)) & 1u, d.polls)) dead = true;
        if (dead) return;  // the warpgroups' waits for these MMAs run out too
        ph ^= 1u << (2 * w + buf);
        tc_fence_after();
        const uint32_t dd = tmem0 + 128u * w, ab = dd + 64u + 32u * buf;
        const uint64_t bd = bd0 + (uint64_t)(c * 512);
        mma_ts(dd, ab, bd, idesc, c != 0 ? 1u : 0u);
        if (nk > 1) mma_ts(dd, ab + 8u, bd + 128u, idesc, 1u);
        if (nk > 2) mma_ts(dd, ab + 16u, bd + 256u, idesc, 1u);
        if (nk > 3) mma_ts(dd, ab + 24u, bd + 384u, idesc, 1u);
        mma_commit(full + 16u);
      };
      for (int tile0 = 2 * part; tile0 < tiles; tile0 += 2 * d.parts) {
        const bool both = tile0 + 1 < tiles;
        for (int c = 0; c < n64; c += 2) {
          const int nk = nk16 - 4 * c;
          issue(0, 0, c, nk);
          if (both) issue(1, 0, c, nk);
          if (c + 1 < n64) {
            issue(0, 1, c + 1, nk - 4);
            if (both) issue(1, 1, c + 1, nk - 4);
          }
        }
      }
      // none is in flight when the block ends, also where a wait has run out
      for (int i = 0; i < 4; ++i)
        if (!mbar_wait(full0 + 16u + 32u * (i >> 1) + 8u * (i & 1), ((ph >> i) & 1u) ^ 1u, kDensePolls)) dead = true;
    }
    __syncwarp();
  }
  // produce: write a chunk's A values; the next chunk's bits are expanded
  // while the TMEM writes run.
  auto produce = [&](int buf, const uint32_t(&r)[32], auto next) {
    if (use[buf] > 0 && !dead && !mbar_wait(bar + 16u + 8u * buf, (use[buf] - 1) & 1u, d.polls)) dead = true;
    tmem_st32(tm + 64u + 32u * buf + lsel, r);
    next();
    tmem_st_wait();
    tc_fence_before();
    __syncwarp();
    if (lane == 0) mbar_arrive(bar + 8u * buf);
    ++use[buf];
  };
  // m doubtful pairs of the list, one per lane: their sum in CSR order, then
  // the step tail (the epilogue has left their x and V as they were)
  auto value = [&](int u, int b) -> float {
    const float f = to_f(*reinterpret_cast<const TX*>(sX + u * 128 + (((b >> 3) ^ (u & 7)) << 4) + (b & 7) * 2));
    return X::kScaled ? f * __uint_as_float(row_inverse(u) << 23) : f;
  };
  auto solve = [&](const uint16_t* list, int m) {
    __syncwarp();
    if (lane < m && list[lane] != 0xffffu) {
      const int e = list[lane];
      const int b = traj_of_bit(e & 31);
      const int v = e >> 5;
      const int dv = MIS ? 0 : a.g.row_ptr[off + v + 1] - a.g.row_ptr[off + v];
      const float lo = MIS ? 0.0f : -1.0f;
      // neighbours with x != 0 (the others leave the sum as it is), in
      // CSR order: ascending columns of the row's adjacency words
      const uint4* rp = d.bits + boff + (int64_t)(v >> 7) * tiles * 128 + (v & 127);
      const int words = (ng + 31) >> 5;
      float acc = 0.0f;
      int nb = 0;
      uint4 q4 = __ldg(rp);
      for (int w4 = 0; w4 < words; w4 += 4) {
        const uint4 cur = q4;
        if (w4 + 4 < words) q4 = __ldg(rp + (w4 / 4 + 1) * 128);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (w4 + k >= words) break;
          uint32_t m = (k == 0 ? cur.x : k == 1 ? cur.y : k == 2 ? cur.z : cur.w) & s_nz[32 * (w4 + k) + (e & 31)];
          if (m) m = to_natural(m);
          while (m) {
            // two neighbours at a time, so that their loads overlap
            const int u = 32 * (w4 + k) + __ffs(m) - 1;
            m &= m - 1u;
            const bool two = m != 0u;
            const int u2 = two ? 32 * (w4 + k) + __ffs(m) - 1 : u;
            m &= m - 1u;
            const float f = value(u, b), f2 = value(u2, b);
            acc = acc + f;
            nb += f > thr;
            if (two) {
              acc = acc + f2;
              nb += f2 > thr;
            }
          }
        }
      }
      if (MIS) nb = nb != 0;
      const int64_t q = (int64_t)v * B + b;
      TX xnew;
      TV vnew;
      bool zn;
      int k0 = 0, k1 = 0, k2 = 0;
      step_element<TX, TV, OBJ>(a, MIS, thr, lo, Xc[q], V[q], acc, nb, dv, true, xnew, vnew, zn, k0, k1, k2);
      Xn[q] = xnew;
      V[q] = vnew;
      uint32_t* zp = Zn + (int64_t)v * a.Bw;
      if (zn) atomicOr(zp, 1u << b);
      else atomicAnd(zp, ~(1u << b));
      if (k0) atomicAdd(&s_cnt[0][b], (uint32_t)k0);
      if (k1) atomicAdd(&s_cnt[1][b], (uint32_t)k1);
      if (k2) atomicAdd(&s_cnt[2][b], (uint32_t)k2);
    }
    __syncwarp();
  };
  // The sums and set counts of the warp's 32 rows of a tile in CSR order, 8 rows
  // at a time: four lanes per row, 8 trajectories (16 bytes) each; then to the
  // rows' lanes and into the accumulator columns.  Entries past a row's end
  // read the zero row behind the block (+0 leaves a sum as it is).  MIS wants
  // to know only whether some neighbour is in the set: a running signed max of
  // the 16-bit patterns, which order like the values in [0, 1].
  // An entry is kept as the byte offset of its row with the swizzle in bits
  // 4 .. 6 and, for scaled rows, the factor's index in bits 0 and 1.
  auto recompute = [&](int tile, auto scaled, auto counts) {
    constexpr bool kUnscale = decltype(scaled)::value;
    constexpr bool kMaxOnly = !decltype(counts)::value;
    const int sub = lane >> 2, l = lane & 3;
    const T2 thr2 = X::splat(thr);
    const uint32_t sbase = smem_addr(sX);
    for (int pass = 0; pass < 4; ++pass) {
      const int v = tile * 128 + (warp & 3) * 32 + pass * 8 + sub;
      const int j0 = v < ng ? a.g.row_ptr[off + v] : 0, j1 = v < ng ? a.g.row_ptr[off + v + 1] : 0;
      const int longest = __reduce_max_sync(0xffffffffu, j1 - j0);
      float acc[8];
      uint32_t cn[4] = {0u, 0u, 0u, 0u};
#pragma unroll
      for (int k = 0; k < 8; ++k) acc[k] = 0.0f;
      // entries 16 ahead of the sums; a lane holds every fourth
      uint32_t id[4], idn[4];
      auto entry = [&](int j) -> uint32_t {
        const int u = j < j1 ? a.g.col[j] - off : kpad;
        return (uint32_t)(u * 128 + ((u & 7) << 4) + (kUnscale ? ((u >> 1) + 1) & 3 : 0));
      };
#pragma unroll
      for (int i = 0; i < 4; ++i) id[i] = entry(j0 + 4 * i + l);
      for (int k = 0; k < longest; k += 16) {
#pragma unroll
        for (int i = 0; i < 4; ++i) idn[i] = entry(j0 + k + 16 + 4 * i + l);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          uint32_t q[4][4], inv[4];
#pragma unroll
          for (int r = 0; r < 4; ++r) {
            const uint32_t e = __shfl_sync(0xffffffffu, id[i], r, 4);
            asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
                         : "=r"(q[r][0]), "=r"(q[r][1]), "=r"(q[r][2]), "=r"(q[r][3])
                         : "r"(sbase + ((e ^ ((uint32_t)l << 4)) & ~15u)));
            inv[r] = (0x08000800u << (e & 3u)) - 0x00800080u;  // row_inverse in both halves
          }
#pragma unroll
          for (int r = 0; r < 4; ++r) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              uint32_t w = q[r][e];
              if constexpr (kUnscale) {
                const T2 y = __hmul2(as2<T2>(w), as2<T2>(inv[r]));
                w = *reinterpret_cast<const uint32_t*>(&y);
              }
              X::add(acc[2 * e], acc[2 * e + 1], w);
              if constexpr (kMaxOnly) cn[e] = __vmaxs2(cn[e], w);
              else cn[e] += __hgt2_mask(as2<T2>(w), thr2) & 0x00010001u;
            }
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) id[i] = idn[i];
      }
      if constexpr (kMaxOnly) {
#pragma unroll
        for (int e = 0; e < 4; ++e) cn[e] = __hgt2_mask(as2<T2>(cn[e]), thr2) & 0x00010001u;
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t s2[16], cw[16];
        tmem_ld16(tm + lsel + 16u * h, s2);
        tmem_ld16(tm + lsel + 32u + 16u * h, cw);
        tmem_ld_wait(s2, cw);
        const bool mine = (lane >> 3) == pass;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const int src = ((lane & 7) << 2) | (2 * h + (k >> 3));
          const float f = __shfl_sync(0xffffffffu, acc[k & 7], src);
          const uint32_t c = __shfl_sync(0xffffffffu, cn[(k & 7) >> 1], src);
          if (mine) {
            s2[k] = __float_as_uint(2.0f * f);
            cw[k] = __float_as_uint((float)((c >> (16 * (k & 1))) & 0xffffu));
          }
        }
        tmem_st16(tm + lsel + 16u * h, s2);
        tmem_st16(tm + lsel + 32u + 16u * h, cw);
        tmem_st_wait();
      }
    }
  };
  for (int tile = 2 * part + wg; warp != kIssuer && tile < tiles; tile += 2 * d.parts) {
    const int vl = tile * 128 + wtid;
    const bool has = vl < ng;
    const uint4* bp = bits0 + (int64_t)tile * tiles * 128;
    const int64_t rb = (int64_t)(has ? vl : 0) * B;
    prefetch_l2_line(V + rb);
    if (sizeof(TV) == 4) prefetch_l2_line(V + rb + 16);
    if (!heavy) {
      uint4 bw = tile == 2 * part + wg ? bfirst : __ldg(bp);
      // words two pieces ahead (four chunks: an L2 latency)
      uint4 b1 = n64 > 2 ? __ldg(bp + 128) : bw, b2 = bw;
      uint32_t ra[32], rc[32];
      expand_bits<X::kScaled>(bw.x, bw.y, ra);
      for (int c = 0; c < n64; c += 2) {
        if (c + 4 < n64) b2 = __ldg(bp + ((c >> 1) + 2) * 128);
        produce(0, ra, [&] { expand_bits<X::kScaled>(bw.z, bw.w, rc); });
        if (c + 1 < n64) produce(1, rc, [&] { expand_bits<X::kScaled>(b1.x, b1.y, ra); });
        bw = b1;
        b1 = b2;
      }
    }
    // this row's x and V of the 32 trajectories while the last MMAs run
    uint32_t xo[16];
    {
      const uint4* p = reinterpret_cast<const uint4*>(Xc + rb);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint4 q = p[k];
        xo[4 * k] = q.x, xo[4 * k + 1] = q.y, xo[4 * k + 2] = q.z, xo[4 * k + 3] = q.w;
      }
    }
    uint32_t vo[16];
    if constexpr (sizeof(TV) == 2) {
      const uint4* p = reinterpret_cast<const uint4*>(V + rb);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const uint4 q = p[k];
        vo[4 * k] = q.x, vo[4 * k + 1] = q.y, vo[4 * k + 2] = q.z, vo[4 * k + 3] = q.w;
      }
    }
    const int deg = MIS ? 0 : a.g.row_ptr[off + (has ? vl : 0) + 1] - a.g.row_ptr[off + (has ? vl : 0)];
    if (use[0] > 0 && !dead && !mbar_wait(bar + 16u, (use[0] - 1) & 1u, d.polls)) dead = true;
    if (use[1] > 0 && !dead && !mbar_wait(bar + 24u, (use[1] - 1) & 1u, d.polls)) dead = true;
    tc_fence_after();

    // Which pairs are doubtful?  Few go on the list; a warp with many sums its
    // 32 rows again from the staged block and puts the sums where the MMAs'
    // were.
    constexpr int kFew = MIS ? kDoubtfulMis : kDoubtfulCut;
    uint32_t doubt = 0u;
    if (heavy) {
      // (a NaN would hide others in the running max)
      if (MIS && !bad) recompute(tile, std::false_type{}, std::false_type{});
      else recompute(tile, std::false_type{}, std::true_type{});
    } else {
      bool odd = false;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t s2[16], cw[16];
        tmem_ld16(tm + lsel + 32u + 16u * h, cw);
        tmem_ld16(tm + lsel + 16u * h, s2);
        tmem_ld_wait(s2, cw);
        float wmax = 0.0f;
#pragma unroll
        for (int k = 0; k < 16; ++k) wmax = fmaxf(wmax, __uint_as_float(cw[k]));
        if (!__any_sync(0xffffffffu, wmax >= 1024.0f)) continue;
        odd = true;
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const float W = __uint_as_float(cw[k]);
          const bool db = MIS ? (W >= 16384.0f || (W >= 1024.0f && !(__uint_as_float(s2[k]) < d.s1x2))) : W >= 1024.0f;
          doubt |= (uint32_t)db << (8 * h + (k >> 1) + 16 * (k & 1));
          cw[k] = __float_as_uint((float)((int)W & 1023));
        }
        tmem_st16(tm + lsel + 32u + 16u * h, cw);
      }
      if (odd) {
        doubt &= has ? stepw : 0u;
        const int total = __reduce_add_sync(0xffffffffu, __popc(doubt));
        if (total > 0) {
          int base = 0;
          if (total <= kFew) {
            if (lane == 0) base = atomicAdd(&s_listed, total);
            base = __shfl_sync(0xffffffffu, base, 0);
          }
          if (total > kFew || base + total > kDoubtful) {
            if (total <= kFew)
              for (int i = base + lane; i < kDoubtful; i += 32) s_list[i] = 0xffffu;
            tmem_st_wait();
            recompute(tile, std::integral_constant<bool, X::kScaled>{}, std::integral_constant<bool, !MIS>{});
            doubt = 0u;
          } else {
            int at = __popc(doubt);
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
              const int y = __shfl_up_sync(0xffffffffu, at, o);
              if (lane >= o) at += y;
            }
            at += base - __popc(doubt);
            for (uint32_t m = doubt; m; m &= m - 1u) s_list[at++] = (uint16_t)(vl << 5 | (__ffs(m) - 1));
          }
        }
        tmem_st_wait();
      }
    }
    uint32_t zold = 0u, znew = 0u, f1 = 0u, f2 = 0u;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      uint32_t s2[16], cw[16];
      tmem_ld16(tm + lsel + 16u * h, s2);
      tmem_ld16(tm + lsel + 32u + 16u * h, cw);
      float vf[16];
      if constexpr (sizeof(TV) == 4) {
        const float4* p = reinterpret_cast<const float4*>(V + rb + 16 * h);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float4 q = p[k];
          vf[4 * k] = q.x, vf[4 * k + 1] = q.y, vf[4 * k + 2] = q.z, vf[4 * k + 3] = q.w;
        }
      }
      tmem_ld_wait(s2, cw);
      uint32_t cp[8];  // neighbours in the set
#pragma unroll
      for (int k = 0; k < 8; ++k) cp[k] = X::pack(__uint_as_float(cw[2 * k]), __uint_as_float(cw[2 * k + 1]));
      // pairs whose x and V stay as they are (for now): no step this tick, or doubtful
      const uint32_t keep = ~stepw | doubt;
      auto tail = [&](auto kept) {
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int i = 8 * h + k;
          const uint32_t pm = (1u << i) | (1u << (16 + i));
          float x0, x1;
          X::unpack(xo[i], x0, x1);
          float g0 = __uint_as_float(s2[2 * k]), g1 = __uint_as_float(s2[2 * k + 1]);
          const uint32_t zm = __hgt2_mask(as2<T2>(xo[i]), X::splat(thr));
          zold |= zm & pm;
          if constexpr (MIS) {
            // some neighbour in the set
            f1 |= __hgt2_mask(as2<T2>(cp[k]), X::splat(0.0f)) & pm;
            // grad = 1 - gamma * sum; g holds 2 * sum
            mul2(g0, g1, -0.5f * a.gamma, -0.5f * a.gamma);
            g0 = g0 + 1.0f;
            g1 = g1 + 1.0f;
          } else {
            const int p0 = (int)__uint_as_float(cw[2 * k]), p1 = (int)__uint_as_float(cw[2 * k + 1]);
            const int as0 = 2 * p0 - deg, as1 = 2 * p1 - deg;
            const bool z0 = (zm & 0xffffu) != 0u, z1 = (zm >> 16) != 0u;
            const bool fix0 = cut_fixed(OBJ >= 0 ? OBJ : a.objective, a.lambda_, z0, as0, deg);
            const bool fix1 = cut_fixed(OBJ >= 0 ? OBJ : a.objective, a.lambda_, z1, as1, deg);
            f1 |= (fix0 ? 0u : 1u << i) | (fix1 ? 0u : 1u << (16 + i));
            f2 |= ((z0 ? as0 : -as0) > 0 ? 1u << i : 0u) | ((z1 ? as1 : -as1) > 0 ? 1u << (16 + i) : 0u);
            // cut edges of the row, summed over the warp's rows per trajectory
            const bool q0 = has && !((doubt >> i) & 1u), q1 = has && !((doubt >> (16 + i)) & 1u);
            const uint32_t r0 = __reduce_add_sync(0xffffffffu, q0 ? (uint32_t)(z0 ? deg - p0 : p0) : 0u);
            const uint32_t r1 = __reduce_add_sync(0xffffffffu, q1 ? (uint32_t)(z1 ? deg - p1 : p1) : 0u);
            if (lane == i) n0 += r0;
            if (lane == 16 + i) n0 += r1;
            // the exact sum (a zero sum as +0)
            g0 = cut_grad(OBJ >= 0 ? OBJ : a.objective, a.lambda_, x0, 0.5f * g0 + 0.0f, deg);
            g1 = cut_grad(OBJ >= 0 ? OBJ : a.objective, a.lambda_, x1, 0.5f * g1 + 0.0f, deg);
          }
          float v0, v1;
          if constexpr (sizeof(TV) == 2) X::unpack(vo[i], v0, v1);
          else v0 = vf[2 * k], v1 = vf[2 * k + 1];
          mul2(v0, v1, a.momentum, a.momentum);
          mul2(g0, g1, a.alpha, a.alpha);
          v0 = v0 + g0;
          v1 = v1 + g1;
          add_f32x2(x0, x1, v0, v1);
          // the box after the storage rounding: its ends are representable and
          // rounding is monotone, so the order makes no difference
          T2 xr = as2<T2>(X::pack(x0, x1));
          xr = __hmin2_nan(__hmax2_nan(xr, X::splat(MIS ? 0.0f : -1.0f)), X::splat(1.0f));
          uint32_t xn = *reinterpret_cast<const uint32_t*>(&xr);
          uint32_t km = 0u;
          if constexpr (decltype(kept)::value) {
            km = ((keep >> i) & 0x00010001u) * 0xffffu;
            xn = (xn & ~km) | (xo[i] & km);
          }
          znew |= __hgt2_mask(as2<T2>(xn), X::splat(thr)) & pm;
          xo[i] = xn;
          if constexpr (sizeof(TV) == 2) {
            uint32_t vn = X::pack(v0, v1);
            if constexpr (decltype(kept)::value) vn = (vn & ~km) | (vo[i] & km);
            vo[i] = vn;
          } else if constexpr (decltype(kept)::value) {
            vf[2 * k] = (km & 1u) ? vf[2 * k] : v0;
            vf[2 * k + 1] = (km >> 16) ? vf[2 * k + 1] : v1;
          } else {
            vf[2 * k] = v0;
            vf[2 * k + 1] = v1;
          }
        }
      };
      if (__any_sync(0xffffffffu, keep != 0u)) tail(std::true_type{});
      else tail(std::false_type{});
      if (has) {
        uint4* px = reinterpret_cast<uint4*>(Xn + rb + 16 * h);
        px[0] = make_uint4(xo[8 * h], xo[8 * h + 1], xo[8 * h + 2], xo[8 * h + 3]);
        px[1] = make_uint4(xo[8 * h + 4], xo[8 * h + 5], xo[8 * h + 6], xo[8 * h + 7]);
        if constexpr (sizeof(TV) == 2) {
          uint4* pv = reinterpret_cast<uint4*>(V + rb + 16 * h);
          pv[0] = make_uint4(vo[8 * h], vo[8 * h + 1], vo[8 * h + 2], vo[8 * h + 3]);
          pv[1] = make_uint4(vo[8 * h + 4], vo[8 * h + 5], vo[8 * h + 6], vo[8 * h + 7]);
        } else {
          float4* pv = reinterpret_cast<float4*>(V + rb + 16 * h);
#pragma unroll
          for (int k = 0; k < 4; ++k) pv[k] = make_float4(vf[4 * k], vf[4 * k + 1], vf[4 * k + 2], vf[4 * k + 3]);
        }
      }
    }
    if (has) Zn[(int64_t)vl * a.Bw] = to_natural(znew);
    // counts over the tile's rows: rows of the warp -> bits of trajectory words
    const uint32_t in = has ? ~doubt : 0u;
    if constexpr (MIS) {
      n0 += __popc(warp_transpose(zold & in, lane));
      n1 += __popc(warp_transpose(zold & f1 & in, lane));
      n2 += __popc(warp_transpose(~zold & ~f1 & in, lane));
    } else {
      n1 += __popc(warp_transpose(f1 & in, lane));
      n2 += __popc(warp_transpose(f2 & in, lane));
    }
    tc_fence_before();  // this tile's TMEM loads before the next tile's MMAs
  }
  dead = __syncthreads_or(dead) != 0;
  for (int i = warp * 32; i < min(s_listed, kDoubtful) && !dead; i += kDenseThreads + 32)
    solve(s_list + i, min(32, min(s_listed, kDoubtful) - i));
  if (warp != kIssuer && !dead) {
    const int b = traj_of_bit(lane);
    if (n0) atomicAdd(&s_cnt[0][b], n0);
    if (n1) atomicAdd(&s_cnt[1][b], n1);
    if (n2) atomicAdd(&s_cnt[2][b], n2);
  }
  if (dead) *d.late = 1;
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == kIssuer)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(kDenseTmem));
  if (tid < 96) {
    const int k = tid >> 5, b = tid & 31;
    const uint32_t val = s_cnt[k][b];
    // stepw is uniform: bit of trajectory b
    const bool st = (stepw >> ((b >> 1) + 16 * (b & 1))) & 1u;
    if (val && st) {
      Counters* c = a.cnt + ((int64_t)g * B + tg * kDenseGroup + b) * a.R + part % a.R;
      unsigned long long* dst = k == 0 ? &c->value : (k == 1 ? &c->a : &c->b);
      atomicAdd(dst, (unsigned long long)val);
    }
  }
}

cudaError_t launch_dense_bits(const GraphDev& g, const int64_t* bits_off, const int2* tiles, int num_tiles,
                              uint4* bits, cudaStream_t s) {
  if (num_tiles <= 0) return cudaSuccess;
  k_dense_bits<<<num_tiles, 256, 0, s>>>(g, bits_off, tiles, reinterpret_cast<uint32_t*>(bits));
  return cudaGetLastError();
}

// dynamic shared memory of a CTA: the staged rows, their "not zero" masks, a
// kilobyte to align them,
// and never so little that a third CTA would share the SM (TMEM holds two)
size_t dense_smem_bytes(int max_ng) {
  const size_t need = 1024 + (size_t)((max_ng + 15) & ~15) * 128 + 128 + (size_t)((max_ng + 31) & ~31) * 4;
  return need < 80 * 1024 ? 80 * 1024 : need;
}

template <typename TX, typename TV>
static cudaError_t launch_t(const StepArgs& a, const DenseArgs& d, int grid, size_t smem, cudaStream_t s) {
  auto run = [&](auto kern) -> cudaError_t {
    cudaError_t e = allow_smem(kern, kDenseSmemLimit);
    if (e != cudaSuccess) return e;
    kern<<<grid, kDenseThreads + 32, smem, s>>>(a, d);
    return cudaGetLastError();
  };
  if (a.problem == PROB_MIS) return run(k_step_t<TX, TV, true, -1>);
  if (a.objective == OBJ_FB) return run(k_step_t<TX, TV, false, OBJ_FB>);
  return run(k_step_t<TX, TV, false, -1>);
}

cudaError_t launch_step_dense(const StepArgs& a, const DensePlan& p, int x_dtype, int v_dtype, cudaStream_t s) {
  DenseArgs d;
  d.bits = p.bits;
  d.bits_off = p.bits_off;
  d.groups = a.B / kDenseGroup;
  d.parts = p.parts;
  // exact sums: s + t + (significand bits) - 1 <= 24, with 2^s above the
  // largest degree; a sum of MIS below 2^(s-4) allows x 16 times smaller
  const int s0 = p.sum_bits;
  const int t = (x_dtype == DT_BF16 ? 17 : 14) - s0;
  d.t0 = ldexpf(1.0f, -t);
  d.t1 = ldexpf(1.0f, -t - 4);
  d.s1x2 = ldexpf(2.0f, s0 - 4);
  d.late = p.late;
  d.polls = p.polls;
  d.degree = (float)((double)a.g.nnz / (double)a.g.n);
  const int grid = a.g.num_graphs * d.groups * d.parts;
  if (x_dtype == DT_BF16 && v_dtype == DT_BF16) return launch_t<__nv_bfloat16, __nv_bfloat16>(a, d, grid, p.smem, s);
  if (x_dtype == DT_BF16 && v_dtype == DT_F32) return launch_t<__nv_bfloat16, float>(a, d, grid, p.smem, s);
  if (x_dtype == DT_F16 && v_dtype == DT_F16) return launch_t<__half, __half>(a, d, grid, p.smem, s);
  if (x_dtype == DT_F16 && v_dtype == DT_F32) return launch_t<__half, float>(a, d, grid, p.smem, s);
  return cudaErrorInvalidValue;
}

}  // namespace mqo
