// The layer-2 probe: from the queries, keys and values of one attention layer on the sequence
// [system, visual, prompt] (Sec. 3.1), the two things the compression reads: the visual rows of
// Z = Softmax(Q K^T / sqrt(d_k)) V (Eq. 3-1, 3-2; heads side by side), and the attention the
// probe rows pay to the visual tokens (the slice Eq. 3-7 averages).  The probability matrix is
// never written out in full.
//
// Both products run on the 5th-generation tensor cores (tcgen05.mma kind::f16, float32 accumulators in
// TMEM, operands staged by TMA with the 128-byte swizzle), 128 query rows at a time against blocks of
// keys, with an online softmax in the exp2 domain.  V is read as it lies: the contraction index is the
// row there.
// Every mbarrier wait is bounded; a wait that runs out records an error for the image and the
// CTA winds down (TMEM is still freed).
#include "tc_internal.cuh"
#include "tcgen05_util.cuh"

namespace tc {

namespace {

using namespace t5;

constexpr int QT = 128;          // query rows per CTA
constexpr int KB = 128;          // keys per block
constexpr int SB = 64;           // keys per softmax step of the rows of Z
constexpr int DH = 128;          // head dimension the kernel is built for
constexpr uint32_t ATOM = 128 * 128;        // bytes of one 128-row x 64-element swizzle atom
constexpr uint32_t TILE_B = 2 * ATOM;       // a 128 x 128 tile of 16-bit elements
constexpr uint32_t SMEM_Z = 6 * TILE_B + 1024;                      // two of Q, K and V each
constexpr uint32_t SMEM_P = 3 * TILE_B + 4 * 32 * 64 + 1024;        // Q, two of K, staging of the probabilities
constexpr uint32_t TMEM_COLS_Z = 512;                               // two of the scores and two of Z
constexpr uint32_t TMEM_COLS_P = 256;                               // two of the scores

// D float32, A and B float16 (bf = 0) or bfloat16 (bf = 1), both K-major, M = 128, N = n
__device__ __forceinline__ uint32_t idesc(int bf, int n = 128) {
  return (1u << 4) | (bf ? ((1u << 7) | (1u << 10)) : 0u) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void umma_16(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t id,
                                        uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(da), "l"(db), "r"(id), "r"(accum)
      : "memory");
}

// the eight tcgen05.mma of a product over dh of two swizzled 16-bit tiles
__device__ __forceinline__ void mma_tile(uint32_t tmem_d, uint32_t a_base, uint32_t b_base, uint32_t id) {
#pragma unroll
  for (int ks = 0; ks < 8; ++ks) {
    const uint32_t atom = (uint32_t)(ks >> 2) * ATOM;
    umma_16(tmem_d, umma_desc(a_base + atom) + (uint64_t)(2 * (ks & 3)),
            umma_desc(b_base + atom) + (uint64_t)(2 * (ks & 3)), id, ks > 0 ? 1u : 0u);
  }
}

// Descriptor of a tile whose rows of 128 bytes run along the operand's N, 128-byte swizzle: eight rows
// (K) are 1024 bytes, the next 64 columns of N one atom further.
__device__ __forceinline__ uint64_t umma_desc_mn(uint32_t smem_addr) {
  return umma_desc(smem_addr) | ((uint64_t)(ATOM >> 4) << 16);
}
// D (+)= P V for 64 keys, with P (16-bit pairs, a row per lane) in TMEM and V stored [K][N]: 16 rows of V per tcgen05.mma
__device__ __forceinline__ void mma_tile_pv(uint32_t tmem_d, uint32_t tmem_p, uint32_t v_base, uint32_t id, bool accum) {
#pragma unroll
  for (int ks = 0; ks < SB / 16; ++ks)
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "setp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
        ::"r"(tmem_d), "r"(tmem_p + (uint32_t)(8 * ks)), "l"(umma_desc_mn(v_base + (uint32_t)ks * 2048u)), "r"(id | (1u << 16)),
        "r"((accum || ks > 0) ? 1u : 0u)
        : "memory");
}

__device__ __forceinline__ void tmem_ld32_issue(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
        "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// 2^x on the special-function unit (relative error 2^-22: far inside the 16-bit outputs)
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

template <typename T>
__device__ __forceinline__ uint32_t pack2(float a, float b);
template <>
__device__ __forceinline__ uint32_t pack2<__half>(float a, float b) {
  __half2 h = __floats2half2_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}
template <>
__device__ __forceinline__ uint32_t pack2<__nv_bfloat16>(float a, float b) {
  __nv_bfloat162 h = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t*>(&h);
}

struct ProbeArgs {
  int L, n_sys, n_vis, H;
  int row0;          // sequence position of the first query row this launch covers
  int n_rows;        // number of query rows
  float scale2;      // log2(e) / sqrt(dh)
  int bf;
};

constexpr int Z_TMA = 8, Z_MMA = 9, Z_THREADS = 352;   // (a warp that issues products per query tile)
constexpr int P_TMA = 4, P_MMA = 5, P_THREADS = 192;
constexpr float MAX_SLACK = 8.f;

// Visual query rows -> rows of Z (out [B][n_vis][H * dh]).  Two neighbouring query tiles per CTA: one
// tile's softmax runs while the tensor core works for the other, and both read the same key and value
// tiles, in steps of 64 keys:
//   - warp 8 (one lane): TMA, two key and value tiles (128 keys) ahead;
//   - warps 9 and 10: a query tile each, per step Z += P V and the scores of a later step.  P is read
//     from TMEM, where it lies over the scores that it came from; the two score buffers of a tile
//     alternate, so that the next scores are there when a step of the softmax ends;
//   - warps 0-3 and 4-7: the softmax of a tile, a thread per row, all scores of a step in registers.
//     Z stays in TMEM.  The maximum that the exponents refer to is moved (and Z and the row sum
//     rescaled) only when a row's own has grown by more than 2^8 over it: Z = P V / sum is the same
//     whatever the reference, and float16 holds 2^8 with the same relative precision as 1.
// TMEM is full with 2 x 2 x 64 columns of scores and 2 x 128 of Z.
// What bounds it: the chain of a step, 1 070 cycles of softmax (512 of them exponentials at the unit's
// rate), which the other tile's overlaps, and issuing its products with their waits, 1 400 cycles.
// Measured, 16 prompts of 675 tokens, 32 heads: 220 us (one tile per CTA, P through shared memory, V
// transposed beforehand) -> 126.
template <typename T>
__global__ void __launch_bounds__(Z_THREADS, 1) probe_z_kernel(
    const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK,
    const __grid_constant__ CUtensorMap mapV, ProbeArgs pa, T* __restrict__ out,
    int32_t* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_q[2], bar_k[2], bar_kfree[2], bar_v[2], bar_vfree[2];   // (the last four by stage)
  __shared__ __align__(8) uint64_t bar_s[2][2], bar_p[2][2], bar_pv[2][2];   // by query tile and buffer: scores ready; P written; P V done
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.y, b = blockIdx.z, bh = b * pa.H + h;
  const int tile0 = 2 * (int)(gridDim.x - 1 - blockIdx.x);           // the longest rows first
  const int end = pa.row0 + pa.n_rows;                               // past the last query row
  auto q0_of = [&](int t) { return pa.row0 + (tile0 + t) * QT; };
  auto last_of = [&](int t) { return min(end, q0_of(t) + QT) - 1; };
  const int nt = q0_of(1) < end ? 2 : 1;                             // tiles that have rows
  auto steps_of = [&](int t) { return t < nt ? last_of(t) / SB + 1 : 0; };   // causal
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  auto sQ = [&](int t) { return smem_base + (uint32_t)t * TILE_B; };
  auto sK = [&](int s) { return smem_base + (uint32_t)(2 + s) * TILE_B; };
  auto sV = [&](int s) { return smem_base + (uint32_t)(4 + s) * TILE_B; };
  const uint32_t id_s = idesc(pa.bf, SB), id_o = idesc(pa.bf);

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&bar_q[i]), 1);
      mbar_init(smem_u32(&bar_k[i]), 1);
      mbar_init(smem_u32(&bar_kfree[i]), (uint32_t)nt);
      mbar_init(smem_u32(&bar_v[i]), 1);
      mbar_init(smem_u32(&bar_vfree[i]), (uint32_t)nt);
      for (int u = 0; u < 2; ++u) {
        mbar_init(smem_u32(&bar_s[i][u]), 1);
        mbar_init(smem_u32(&bar_p[i][u]), 4);
        mbar_init(smem_u32(&bar_pv[i][u]), 1);
      }
    }
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == Z_MMA) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(TMEM_COLS_Z)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  auto tmem_s = [&](int t, int i) { return s_tmem + (uint32_t)t * 128u + ((uint32_t)i & 1u) * 64u; };
  auto tmem_o = [&](int t) { return s_tmem + 256u + (uint32_t)t * 128u; };
  auto sphase = [](int i) { return ((uint32_t)i >> 1) & 1u; };

  if (warp == Z_TMA) {
    if (lane == 0) {
      bool ok = true;
      auto load = [&](const CUtensorMap* map, uint32_t dst, int row, uint64_t* bar) {
        mbar_expect_tx(smem_u32(bar), TILE_B);
        tma_load_3d(dst, map, 0, row, bh, smem_u32(bar));
        tma_load_3d(dst + ATOM, map, 64, row, bh, smem_u32(bar));
      };
      load(&mapQ, sQ(0), q0_of(0), &bar_q[0]);
      // (a stage is free when every tile is done with it: both walk all key tiles but the last, which
      // no other follows in its stage)
      for (int it = 0; 2 * it < steps_of(nt - 1) && ok; ++it) {
        const int s = it & 1;
        if (it >= 2 && !mbar_wait(smem_u32(&bar_kfree[s]), sphase(it - 2))) { ok = false; break; }
        load(&mapK, sK(s), it * KB, &bar_k[s]);
        if (it == 0 && nt > 1) load(&mapQ, sQ(1), q0_of(1), &bar_q[1]);
        if (it >= 2 && !mbar_wait(smem_u32(&bar_vfree[s]), sphase(it - 2))) { ok = false; break; }
        load(&mapV, sV(s), it * KB, &bar_v[s]);
      }
      if (!ok) s_fail = 1;
    }
  } else if (warp >= Z_MMA) {
    // A step's few waits and commits take as long to issue as its products: a warp per tile.
    const int t = warp - Z_MMA, n = steps_of(t);
    // scores of step i, over the buffer of step i - 2
    auto scores = [&](int i) {
      const int s = (i >> 1) & 1;
      if (i == 0 && !mbar_wait(smem_u32(&bar_q[t]), 0)) return false;
      if ((i & 1) == 0 && !mbar_wait(smem_u32(&bar_k[s]), sphase(i >> 1))) return false;
      if (i >= 2 && !mbar_wait(smem_u32(&bar_pv[t][i & 1]), sphase(i - 2))) return false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (elect_one()) {
        mma_tile(tmem_s(t, i), sQ(t), sK(s) + ((uint32_t)i & 1u) * (SB * 128u), id_s);
        umma_commit(smem_u32(&bar_s[t][i & 1]));
        if ((i & 1) || i == n - 1) umma_commit(smem_u32(&bar_kfree[s]));
      }
      __syncwarp();
      return true;
    };
    auto weigh = [&](int i) {   // Z += P V of step i
      const int s = (i >> 1) & 1;
      if ((i & 1) == 0 && !mbar_wait(smem_u32(&bar_v[s]), sphase(i >> 1))) return false;
      if (!mbar_wait(smem_u32(&bar_p[t][i & 1]), sphase(i))) return false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (elect_one()) {
        mma_tile_pv(tmem_o(t), tmem_s(t, i), sV(s) + ((uint32_t)i & 1u) * (SB * 128u), id_o, i > 0);
        umma_commit(smem_u32(&bar_pv[t][i & 1]));
        if ((i & 1) || i == n - 1) umma_commit(smem_u32(&bar_vfree[s]));
      }
      __syncwarp();
      return true;
    };
    bool ok = n < 1 || (scores(0) && (n < 2 || scores(1)));
    for (int i = 0; i < n && ok; ++i) ok = weigh(i) && (i + 2 >= n || scores(i + 2));
    if (!ok && lane == 0) s_fail = 1;
  } else {
    const int t = warp >> 2, row = (warp & 3) * 32 + lane;
    const int qpos = q0_of(t) + row, q_last = last_of(t), n = steps_of(t);
    const uint32_t lanes = (uint32_t)((warp & 3) * 32) << 16, to = tmem_o(t) + lanes;
    // (a warp without rows in use only keeps the barriers going)
    const bool work = q0_of(t) + (warp & 3) * 32 <= q_last;
    float m = -INFINITY, l = 0.f;
    bool ok = true;
    for (int i = 0; i < n; ++i) {
      if (ok && !mbar_wait(smem_u32(&bar_s[t][i & 1]), sphase(i))) ok = false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (work) {
        const uint32_t ts = tmem_s(t, i) + lanes;
        float x[SB];
        {
          uint32_t* r = reinterpret_cast<uint32_t*>(x);
#pragma unroll
          for (int c = 0; c < SB / 32; ++c) tmem_ld32_issue(ts + (uint32_t)(c * 32), r + c * 32);
          tmem_wait_ld();
        }
        const int jmax = qpos - i * SB;   // columns 0 .. jmax are visible (a row in use is no later than the last key)
        if (!__all_sync(0xffffffffu, jmax >= SB - 1)) {   // (only on the diagonal)
#pragma unroll
          for (int j = 0; j < SB; ++j) x[j] = j <= jmax ? x[j] : -INFINITY;
        }
        float bm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int j = 0; j < SB; j += 8)
#pragma unroll
          for (int u = 0; u < 4; ++u) bm[u] = fmaxf(fmaxf(bm[u], x[j + u]), x[j + 4 + u]);
        const float own = fmaxf(fmaxf(bm[0], bm[1]), fmaxf(bm[2], bm[3])) * pa.scale2;
        if (__any_sync(0xffffffffu, own > m + MAX_SLACK)) {
          const float m_new = fmaxf(m, own), alpha = m_new == -INFINITY ? 1.f : ex2(m - m_new);
          m = m_new;
          l *= alpha;
          if (i > 0) {
            if (ok && !mbar_wait(smem_u32(&bar_pv[t][(i - 1) & 1]), sphase(i - 1))) ok = false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
            for (int c = 0; c < DH / 32; ++c) {
              uint32_t r[32];
              tmem_ld32_issue(to + (uint32_t)(c * 32), r);
              tmem_wait_ld();
#pragma unroll
              for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) * alpha);
              tmem_st16(to + (uint32_t)(c * 32), r);
              tmem_st16(to + (uint32_t)(c * 32 + 16), r + 16);
            }
          }
        }
        const float mm = m == -INFINITY ? 0.f : m;
        float ls[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int c = 0; c < SB / 32; ++c) {
          uint32_t r[16];
#pragma unroll
          for (int j = 0; j < 32; j += 2) {
            const float e0 = ex2(fmaf(x[c * 32 + j], pa.scale2, -mm)), e1 = ex2(fmaf(x[c * 32 + j + 1], pa.scale2, -mm));
            ls[j & 2] += e0;
            ls[(j & 2) + 1] += e1;
            r[j / 2] = pack2<T>(e0, e1);
          }
          tmem_st16(ts + (uint32_t)(c * 16), r);
        }
        l += (ls[0] + ls[1]) + (ls[2] + ls[3]);
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar_p[t][i & 1])) : "memory");
    }
    if (n > 0) {
      // (by buffer, since a thread that has the last scores knows of the product three steps back, not two)
      if (ok && !mbar_wait(smem_u32(&bar_pv[t][(n - 1) & 1]), sphase(n - 1))) ok = false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (!ok) s_fail = 1;
      // The rows leave through the tile's query tile (its last scores are formed): a thread owns a row,
      // so stores from its registers would put each lane of a store into a sector of its own; from
      // there a warp writes a row per store.  16-byte chunk c of row r lies at c ^ (r & 7).
      uint8_t* stg = smem_gen + (uint32_t)t * TILE_B + (uint32_t)((warp & 3) * 32) * 256u;
      if (work) {
        const float inv_l = l > 0.f ? 1.0f / l : 0.f;
#pragma unroll
        for (int c = 0; c < DH / 32; ++c) {
          uint32_t r[32];
          tmem_ld32_issue(to + (uint32_t)(c * 32), r);
          tmem_wait_ld();
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            auto z = [&](int j) { return __uint_as_float(r[q * 8 + j]) * inv_l; };
            uint4 v;
            v.x = pack2<T>(z(0), z(1));
            v.y = pack2<T>(z(2), z(3));
            v.z = pack2<T>(z(4), z(5));
            v.w = pack2<T>(z(6), z(7));
            *reinterpret_cast<uint4*>(stg + (uint32_t)lane * 256u + (((uint32_t)(c * 4 + q) ^ ((uint32_t)lane & 7u)) << 4)) = v;
          }
        }
        __syncwarp();
        if (s_fail == 0) {   // its own 32 rows
          const int q0w = q0_of(t) + (warp & 3) * 32, n_out = min(32, q_last + 1 - q0w);
          // row q0w + i - n_sys of O, columns h * dh ..: 256 bytes, 8 per lane
          uint2* dst = reinterpret_cast<uint2*>(out + (((size_t)b * pa.n_vis + (q0w - pa.n_sys)) * pa.H + h) * DH) + lane;
#pragma unroll 8
          for (int i = 0; i < n_out; ++i)
            dst[(size_t)i * pa.H * (DH / 4)] = *reinterpret_cast<const uint2*>(
                stg + (uint32_t)i * 256u + ((((uint32_t)lane >> 1) ^ ((uint32_t)i & 7u)) << 4) + ((uint32_t)lane & 1u) * 8u);
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && s_fail != 0 && status != nullptr) atomicMax(&status[b], (int)TC_ERR_CUDA);
  if (warp == Z_MMA) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(TMEM_COLS_Z) : "memory");
  }
}

// Probe rows -> probabilities of the visual columns (out [B][H][n_rows][n_vis]), 128 rows per CTA, in
// two passes over the keys: row maxima and sums of all of them, then the normalised probabilities of
// the blocks with visual columns.  Warp 4 (one lane) loads, two key tiles ahead; warp 5 forms scores, one
// block ahead; warps 0-3: a thread per row.  Prompts are short, so most tiles hold few rows and what
// bounds a CTA is the chain of a block (load, product, exponentials): two CTAs share an SM.
// Measured, 64 rows against 675 keys, 512 heads: 95 us (one CTA per SM, scores read twice) -> 74.
template <typename T>
__global__ void __launch_bounds__(P_THREADS, 2) probe_rows_kernel(
    const __grid_constant__ CUtensorMap mapQ, const __grid_constant__ CUtensorMap mapK, ProbeArgs pa,
    T* __restrict__ out, int32_t* __restrict__ status) {
  extern __shared__ uint8_t smem_raw[];
  __shared__ __align__(8) uint64_t bar_q, bar_k[2], bar_kfree[2], bar_s[2], bar_sfree[2];
  __shared__ uint32_t s_tmem;
  __shared__ int s_fail;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.y, b = blockIdx.z, bh = b * pa.H + h;
  const int q0 = pa.row0 + (int)blockIdx.x * QT;             // position of this tile's first row
  const int q_last = min(pa.row0 + pa.n_rows, q0 + QT) - 1;  // ... and of its last row in use
  const int nkb = q_last / KB + 1;                           // causal: keys up to the last row's position
  const uint32_t smem_base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  uint8_t* smem_gen = smem_raw + (smem_base - smem_u32(smem_raw));
  const uint32_t sQ = smem_base;
  auto sK = [&](int i) { return smem_base + (uint32_t)(1 + (i & 1)) * TILE_B; };
  const uint32_t id = idesc(pa.bf);

  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&bar_q), 1);
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&bar_k[i]), 1);
      mbar_init(smem_u32(&bar_kfree[i]), 1);
      mbar_init(smem_u32(&bar_s[i]), 1);
      mbar_init(smem_u32(&bar_sfree[i]), 4);
    }
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == P_MMA) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&s_tmem)), "r"(TMEM_COLS_P)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  auto tmem_s = [&](int i) { return s_tmem + (uint32_t)(i & 1) * 128u; };
  auto phase = [](int i) { return ((uint32_t)i >> 1) & 1u; };

  // key blocks in the order they are walked
  const int vb0 = pa.n_sys / KB, vb1 = min(nkb - 1, (pa.n_sys + pa.n_vis - 1) / KB);
  const int n_iter = nkb + max(0, vb1 - vb0 + 1);
  auto block_of = [&](int it) { return it < nkb ? it : vb0 + (it - nkb); };

  if (warp == P_TMA) {
    if (lane == 0) {
      mbar_expect_tx(smem_u32(&bar_q), TILE_B);
      tma_load_3d(sQ, &mapQ, 0, q0, bh, smem_u32(&bar_q));
      tma_load_3d(sQ + ATOM, &mapQ, 64, q0, bh, smem_u32(&bar_q));
      for (int it = 0; it < n_iter; ++it) {
        if (it >= 2 && !mbar_wait(smem_u32(&bar_kfree[it & 1]), phase(it - 2))) {
          s_fail = 1;
          break;
        }
        const uint32_t full = smem_u32(&bar_k[it & 1]);
        mbar_expect_tx(full, TILE_B);
        tma_load_3d(sK(it), &mapK, 0, block_of(it) * KB, bh, full);
        tma_load_3d(sK(it) + ATOM, &mapK, 64, block_of(it) * KB, bh, full);
      }
    }
  } else if (warp == P_MMA) {
    bool ok = mbar_wait(smem_u32(&bar_q), 0);
    for (int it = 0; it < n_iter && ok; ++it) {
      ok = mbar_wait(smem_u32(&bar_k[it & 1]), phase(it)) &&
           (it < 2 || mbar_wait(smem_u32(&bar_sfree[it & 1]), phase(it - 2)));
      if (!ok) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (elect_one()) {
        mma_tile(tmem_s(it), sQ, sK(it), id);
        umma_commit(smem_u32(&bar_s[it & 1]));
        umma_commit(smem_u32(&bar_kfree[it & 1]));
      }
      __syncwarp();
    }
    if (!ok && lane == 0) s_fail = 1;
  } else {
    const int row = warp * 32 + lane, qpos = q0 + row;
    const bool work = q0 + warp * 32 <= q_last;   // some row of the warp is in use
    uint8_t* stg = smem_gen + 3 * TILE_B + (uint32_t)warp * (32u * 64u);   // 32 rows x 32 columns
    float m = -INFINITY, l = 0.f, inv_l = 0.f;
    bool ok = true;
    for (int it = 0; it < n_iter; ++it) {
      if (ok && !mbar_wait(smem_u32(&bar_s[it & 1]), phase(it))) ok = false;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      float x[KB];
      if (work) {
        uint32_t* r = reinterpret_cast<uint32_t*>(x);
#pragma unroll
        for (int c = 0; c < KB / 32; ++c)
          tmem_ld32_issue(tmem_s(it) + ((uint32_t)(warp * 32) << 16) + (uint32_t)(c * 32), r + c * 32);
        tmem_wait_ld();
      }
      // this score accumulator may be overwritten
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&bar_sfree[it & 1])) : "memory");
      if (!work) continue;
      const int kb = block_of(it), jmax = qpos - kb * KB;   // columns 0 .. jmax are visible
      if (!__all_sync(0xffffffffu, jmax >= KB - 1)) {       // (only blocks on the diagonal)
#pragma unroll
        for (int j = 0; j < KB; ++j) x[j] = j <= jmax ? x[j] : -INFINITY;
      }
      if (it < nkb) {
        float bm[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY}, ls[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
        for (int j = 0; j < KB; ++j) bm[j & 3] = fmaxf(bm[j & 3], x[j]);
        const float m_new = fmaxf(m, fmaxf(fmaxf(bm[0], bm[1]), fmaxf(bm[2], bm[3])) * pa.scale2);
        if (m_new != -INFINITY) {
          l *= ex2(m - m_new);
          m = m_new;
#pragma unroll
          for (int j = 0; j < KB; ++j) ls[j & 3] += ex2(fmaf(x[j], pa.scale2, -m));
          l += (ls[0] + ls[1]) + (ls[2] + ls[3]);
        }
        if (it == nkb - 1) inv_l = l > 0.f ? 1.0f / l : 0.f;
        continue;
      }
      // Normalised probabilities, 32 columns at a time through a staging tile of the warp's, from which
      // rows leave in runs of 32 neighbouring elements per store (a thread owns a row, so stores from
      // its registers would put every lane into a sector of its own).  16-byte chunk q of row r lies
      // at q ^ (r / 2 & 3).
      const float mm = m == -INFINITY ? 0.f : m;
      const int x0 = kb * KB - pa.n_sys;   // visual index of the block's first column
#pragma unroll
      for (int c = 0; c < KB / 32; ++c) {
        if (x0 + c * 32 + 31 < 0 || x0 + c * 32 >= pa.n_vis) continue;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          auto p = [&](int j) { return ex2(fmaf(x[c * 32 + q * 8 + j], pa.scale2, -mm)) * inv_l; };
          uint4 v;
          v.x = pack2<T>(p(0), p(1));
          v.y = pack2<T>(p(2), p(3));
          v.z = pack2<T>(p(4), p(5));
          v.w = pack2<T>(p(6), p(7));
          *reinterpret_cast<uint4*>(stg + (uint32_t)lane * 64u + ((uint32_t)(q ^ ((lane >> 1) & 3)) << 4)) = v;
        }
        __syncwarp();
        const int xv = x0 + c * 32 + lane;
        const int n_out = min(32, q_last + 1 - q0 - warp * 32);
        if (xv >= 0 && xv < pa.n_vis) {
          T* dst = out + ((size_t)bh * pa.n_rows + (q0 - pa.row0) + warp * 32) * pa.n_vis + xv;
#pragma unroll 8
          for (int rr = 0; rr < n_out; ++rr) {
            *dst = *reinterpret_cast<const T*>(stg + (uint32_t)rr * 64u + ((uint32_t)((lane >> 3) ^ ((rr >> 1) & 3)) << 4) +
                                               ((uint32_t)lane & 7u) * 2u);
            dst += pa.n_vis;
          }
        }
        __syncwarp();
      }
    }
    if (!ok) s_fail = 1;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (threadIdx.x == 0 && s_fail != 0 && status != nullptr) atomicMax(&status[b], (int)TC_ERR_CUDA);
  if (warp == P_MMA) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(s_tmem), "r"(TMEM_COLS_P) : "memory");
  }
}

// [inner, rows, BH] 16-bit tensor, box 64 x 128 x 1, 128-byte swizzle, zero fill
bool encode16(CUtensorMap* map, const void* base, int inner, int rows, int bh, int bf) {
  encode_fn enc = get_encode();
  if (enc == nullptr) return false;
  const cuuint64_t dims[3] = {(cuuint64_t)inner, (cuuint64_t)rows, (cuuint64_t)bh};
  const cuuint64_t strides[2] = {(cuuint64_t)inner * 2, (cuuint64_t)rows * inner * 2};
  const cuuint32_t box[3] = {64, 128, 1};
  const cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, bf ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3,
             const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <typename T>
tc_status run_probe(int B, int H, int L, int n_sys, int n_vis, int probe_start, int n_probe,
                    const void* Q, const void* K, const void* V, void* O, void* A,
                    int32_t* status, cudaStream_t st, int bf) {
  CUtensorMap mq, mk, mv;
  if (!encode16(&mq, Q, DH, L, B * H, bf) || !encode16(&mk, K, DH, L, B * H, bf)) return TC_ERR_CUDA;
  if (O != nullptr && !encode16(&mv, V, DH, L, B * H, bf)) return TC_ERR_CUDA;
  if (cudaFuncSetAttribute((const void*)probe_z_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)SMEM_Z) != cudaSuccess ||
      cudaFuncSetAttribute((const void*)probe_rows_kernel<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)SMEM_P) != cudaSuccess)
    return TC_ERR_CUDA;
  ProbeArgs pa;
  pa.L = L; pa.n_sys = n_sys; pa.n_vis = n_vis; pa.H = H;
  pa.scale2 = 1.4426950408889634f / sqrtf((float)DH);
  pa.bf = bf;
  if (O != nullptr) {
    Scope scope_(KC_GRAM, st);
    pa.row0 = n_sys; pa.n_rows = n_vis;
    dim3 grid((n_vis + 2 * QT - 1) / (2 * QT), H, B);
    probe_z_kernel<T><<<grid, Z_THREADS, SMEM_Z, st>>>(mq, mk, mv, pa, (T*)O, status);
    note_launch();
  }
  if (A != nullptr && n_probe > 0) {
    Scope scope_(KC_ATTN, st);
    // columns a probe row may not see (keys after it) are not all visited: they read as zero
    if (probe_start < n_sys + n_vis - 1 &&
        cudaMemsetAsync(A, 0, (size_t)B * H * n_probe * n_vis * sizeof(T), st) != cudaSuccess) return TC_ERR_CUDA;
    pa.row0 = probe_start; pa.n_rows = n_probe;
    dim3 grid((n_probe + QT - 1) / QT, H, B);
    probe_rows_kernel<T><<<grid, P_THREADS, SMEM_P, st>>>(mq, mk, pa, (T*)A, status);
    note_launch();
  }
  return TC_OK;
}

}  // namespace

size_t probe_workspace_bytes(int B, int H, int L, int dh) {
  (void)B; (void)H; (void)L; (void)dh;
  return 256;   // (nothing is kept there)
}

tc_status launch_probe(int B, int H, int dh, int L, int n_sys, int n_vis, int probe_start, int n_probe,
                       const void* Q, const void* K, const void* V, void* O, void* A, void* ws,
                       int32_t* status, cudaStream_t st, int bf) {
  if (dh != DH) return TC_ERR_UNSUPPORTED;
  if (bf)
    return run_probe<__nv_bfloat16>(B, H, L, n_sys, n_vis, probe_start, n_probe, Q, K, V, O, A, status, st, 1);
  return run_probe<__half>(B, H, L, n_sys, n_vis, probe_start, n_probe, Q, K, V, O, A, status, st, 0);
}

}  // namespace tc
