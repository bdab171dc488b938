// Inverse Cholesky factor of a symmetric matrix S (+ shift), order up to 192, one block per matrix:
// RinvT = L^{-1} with L L^T = S + shift_rel max_i S_ii I, so that Y RinvT^T has (nearly) orthonormal
// columns when S = Y^T Y: one pass of Cholesky-QR behind Eq. 3-5.  The shift keeps the factorisation
// alive when S is numerically singular; a later pass with a smaller one removes its effect.
//
// Elimination of S next to the identity: step j subtracts multiples of row j from the rows below, in S
// (columns right of j) and in what was the identity (columns left of j), which takes the place of the
// columns of S that are finished.  A row is scaled by the root of its pivot at the end.
// What bounds it is the chain of n steps.  So 16 rows are taken at a time (a panel), and the chain runs
// in one warp: it factors the panel's diagonal block (a lane per column, two steps at a time, 200 cycles),
// then a thread per column eliminates the panel's rows among themselves.  Eight other warps meanwhile
// subtract the panel before from the rows below it, which they hold in registers (all columns of a row in
// one warp: a multiplier costs a cycle of shared memory per warp that reads it); the next panel's rows
// come first and are handed over.
// Measured, 16 matrices: order 144 and 160, 53 and 62 us with the matrix in shared memory, 39 and 47 us
// with all warps in step and two rows per barrier, 25 and 28 us here.  The first panels are bound by the
// subtraction (5 000 cycles, 3 000 of them multiply-adds), the last ones by the chain (4 600).
#include "pair_math.cuh"
#include "tc_internal.cuh"

#include <type_traits>

namespace tc {

namespace {

constexpr int UW = 8;    // warps that hold the matrix
constexpr int WARPS = 16;  // and those of the panels (two warpgroups each)
constexpr int PB = 16;   // rows of a panel
// registers of a thread where the matrix fills them (three column groups); together the 512 x 128 of the launch
constexpr int REGS_MATRIX = 176, REGS_PANEL = 80;
static_assert(REGS_MATRIX * UW + REGS_PANEL * (WARPS - UW) <= 128 * WARPS, "registers of a block");
constexpr int XT_ROW = PB + 4;   // padded: a quarter warp's 16-byte accesses meet no bank twice

struct CholArgs {
  float* S;          // [batch][..][ldS], order n; see `first`
  size_t sS;
  int ldS, n;
  float* R;          // [batch][..][ldR] out
  size_t sR;
  int ldR;
  float shift_rel;
  // A diagonal block of a larger matrix: the first one takes the shift from the whole diagonal (n_rest
  // more entries), adds it there, and leaves the largest entry in `largest` for the others; every
  // block is replaced by the identity, which the products of the other blocks start from.
  bool blocked, first;
  int n_rest;
  float* largest;    // [batch], sL apart
  size_t sL;
  int32_t* status;
};

// NP: 64-column groups, P: panels (n = 16 P <= 64 NP).
template <int NP, int P>
__global__ void __launch_bounds__(WARPS * 32, 1) chol_inv_kernel(const CholArgs ca) {
  constexpr int NC = 64 * NP, PW = 2 * NP, THREADS = (UW + PW) * 32, n = PB * P;
  constexpr int RW = 2 * P;                    // rows of a warp: 16 q + 2 w, + 1 of panel q
  extern __shared__ __align__(16) uint8_t chol_smem[];
  typedef float Rows[PB][NC];
  typedef float Cols[NC][XT_ROW];
  Rows& raw = *reinterpret_cast<Rows*>(chol_smem);   // rows of the next panel as the warps hand them over
  Rows* xs = reinterpret_cast<Rows*>(chol_smem) + 1;   // [2]: rows of a panel, eliminated among themselves
  Cols* xt = reinterpret_cast<Cols*>(xs + 2);          // [2]: the same by columns, times -1 / pivot: multipliers of the rows below
  __shared__ __align__(16) float db[PB][PB], lt[PB][PB];
  __shared__ float s_ninv[PB], s_rs[PB];
  __shared__ float s_red[WARPS];
  __shared__ int s_bad;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.x;
  float* S = ca.S + (size_t)b * ca.sS;
  pdl_wait();
  float md = 0.f;
  for (int i = threadIdx.x; i < n + ca.n_rest; i += WARPS * 32) md = fmaxf(md, S[(size_t)i * (ca.ldS + 1)]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
  if (lane == 0) s_red[warp] = md;
  if (threadIdx.x == 0) s_bad = 0;

  if (warp < UW) {
    if constexpr (NP == 3) asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(REGS_MATRIX));
    const int w = warp;
    auto row_of = [&](int i) { return PB * (i >> 1) + 2 * w + (i & 1); };
    f2 B[RW][NP];
#pragma unroll
    for (int i = 0; i < RW; ++i)
#pragma unroll
      for (int g = 0; g < NP; ++g) {
        const int c = 2 * lane + 64 * g;
        B[i][g] = c < n ? *reinterpret_cast<const f2*>(S + (size_t)row_of(i) * ca.ldS + c) : 0ull;
      }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < WARPS; ++v) md = fmaxf(md, s_red[v]);
    if (ca.blocked && !ca.first) md = ca.largest[(size_t)b * ca.sL];
    const float shift = ca.first ? ca.shift_rel * md : 0.f;
#pragma unroll
    for (int i = 0; i < RW; ++i)
#pragma unroll
      for (int g = 0; g < NP; ++g) {
        const int r = row_of(i), c = 2 * lane + 64 * g;
        float2 t = upk(B[i][g]);
        if (c == r) t.x += shift;
        if (c + 1 == r) t.y += shift;
        B[i][g] = pk(t.x, t.y);
      }
    auto hand_over = [&](auto qc) {   // rows of panel q
      constexpr int q = decltype(qc)::value;
#pragma unroll
      for (int u = 0; u < 2; ++u)
#pragma unroll
        for (int g = 0; g < NP; ++g) *reinterpret_cast<f2*>(&raw[2 * w + u][2 * lane + 64 * g]) = B[2 * q + u][g];
      asm volatile("bar.arrive 1, %0;" ::"n"(THREADS) : "memory");
    };
    // rows i0 .. i1 - 1 -= multipliers times the rows of panel p
    auto subtract = [&](auto pc, auto ac, auto bc) {
      constexpr int p = decltype(pc)::value, i0 = decltype(ac)::value, i1 = decltype(bc)::value;
      constexpr int buf = p & 1;
      // the panel's columns of the rows below start over as columns of the inverse
      const bool zero = ((2 * lane + 64 * (p / 4)) >> 4) == p;
#pragma unroll
      for (int i = i0; i < i1; ++i) B[i][p / 4] = zero ? 0ull : B[i][p / 4];
#pragma unroll(i1 - i0 <= 2 ? 4 : P <= 10 ? 2 : 1)   // (as far as the registers go)
      for (int m = 0; m < PB; m += 2) {
        f2 x[2][NP];
#pragma unroll
        for (int u = 0; u < 2; ++u)
#pragma unroll
          for (int g = 0; g < NP; ++g) x[u][g] = *reinterpret_cast<const f2*>(&xs[buf][m + u][2 * lane + 64 * g]);
#pragma unroll
        for (int i = i0; i < i1; ++i) {
          const float2 l = *reinterpret_cast<const float2*>(&xt[buf][row_of(i)][m]);
          const f2 l0 = pk(l.x, l.x), l1 = pk(l.y, l.y);
#pragma unroll
          for (int g = 0; g < NP; ++g) B[i][g] = fma2(l1, x[1][g], fma2(l0, x[0][g], B[i][g]));
        }
      }
    };
    hand_over(std::integral_constant<int, 0>{});
    auto panel = [&](auto pc) {
      constexpr int p = decltype(pc)::value;
      if constexpr (p + 1 < P) {
        asm volatile("bar.sync 3, %0;" ::"n"(THREADS) : "memory");   // panel p is there
        subtract(pc, std::integral_constant<int, 2 * p + 2>{}, std::integral_constant<int, 2 * p + 4>{});
        hand_over(std::integral_constant<int, p + 1>{});
        if constexpr (p + 2 < P) {
          subtract(pc, std::integral_constant<int, 2 * p + 4>{}, std::integral_constant<int, RW>{});
        }
      }
    };
    panel(std::integral_constant<int, 0>{});
    panel(std::integral_constant<int, 1>{});
    panel(std::integral_constant<int, 2>{});
    panel(std::integral_constant<int, 3>{});
    panel(std::integral_constant<int, 4>{});
    panel(std::integral_constant<int, 5>{});
    panel(std::integral_constant<int, 6>{});
    panel(std::integral_constant<int, 7>{});
    panel(std::integral_constant<int, 8>{});
    panel(std::integral_constant<int, 9>{});
    panel(std::integral_constant<int, 10>{});
    return;
  }

  // ---- the panels ----
  if constexpr (NP == 3) asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(REGS_PANEL));
  __syncthreads();
#pragma unroll
  for (int v = 0; v < WARPS; ++v) md = fmaxf(md, s_red[v]);
  if (ca.blocked && !ca.first) md = ca.largest[(size_t)b * ca.sL];
  // A direction of S under the rounding level of its entries can leave any pivot: one below 2.5e-7 of
  // the largest entry is raised to that.  Only a pivot that is negative by far more than rounding (or
  // no number) says that S is not what it should be.
  const float floor_p = 2.5e-7f * fmaxf(md, 1e-30f);
  const float bad_p = -1e-5f * md;
  const int c = threadIdx.x - UW * 32;
  if (c >= NC) return;
  float* R = ca.R + (size_t)b * ca.sR;
  bool bad = false;
#pragma unroll 1
  for (int q = 0; q < P; ++q) {
    const int j0 = PB * q, buf = q & 1;
    asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");   // its rows have been handed over
    float x[PB];
    if (warp == UW) {
      const int cl = lane & (PB - 1);
      float own_p = 1.f, own_inv = 1.f;
#pragma unroll
      for (int i = 0; i < PB; ++i) x[i] = raw[i][j0 + cl];
#pragma unroll
      for (int m = 0; m < PB; m += 2) {   // two steps: rows m and m + 1, the second with the first one applied
        db[m][cl] = x[m];
        db[m + 1][cl] = x[m + 1];
        const float piv = __shfl_sync(0xffffffffu, x[m], m), off = __shfl_sync(0xffffffffu, x[m + 1], m);
        const float piv1 = __shfl_sync(0xffffffffu, x[m + 1], m + 1);
        __syncwarp();
        const float pa = fmaxf(piv, floor_p), ia = rcp_newton(pa), g = -off * ia, ta = x[m] * ia;
        const float qb = fmaf(g, off, piv1), pb = fmaxf(qb, floor_p), ib = rcp_newton(pb);
        const float tb = fmaf(g, x[m], x[m + 1]) * ib;
        bad |= !(piv > bad_p) | !(qb > bad_p);
        lt[m][cl] = ta;
        lt[m + 1][cl] = tb;
        if (cl == m) {
          own_p = pa;
          own_inv = ia;
        }
        if (cl == m + 1) {
          own_p = pb;
          own_inv = ib;
        }
        auto next = [&](int i, float r0, float r1) { x[i] = fmaf(-fmaf(g, r0, r1), tb, fmaf(-r0, ta, x[i])); };
#pragma unroll
        for (int i4 = (m + 2) & ~3; i4 < PB; i4 += 4) {
          const float4 r0 = *reinterpret_cast<const float4*>(&db[m][i4]), r1 = *reinterpret_cast<const float4*>(&db[m + 1][i4]);
          if (i4 > m + 1) {
            next(i4, r0.x, r1.x);
            next(i4 + 1, r0.y, r1.y);
          }
          next(i4 + 2, r0.z, r1.z);
          next(i4 + 3, r0.w, r1.w);
        }
      }
      s_ninv[cl] = -own_inv;
      s_rs[cl] = rsqrtf(own_p);
    }
    const bool mine = (c >> 4) == q;   // a column of the panel starts over as one of the identity
#pragma unroll
    for (int i = 0; i < PB; ++i) x[i] = mine ? (c == j0 + i ? 1.f : 0.f) : raw[i][c];
    asm volatile("bar.sync 2, %0;" ::"n"(PW * 32) : "memory");   // the block's factor is there
#pragma unroll
    for (int m = 0; m < PB - 1; ++m) {
#pragma unroll
      for (int i4 = (m + 1) & ~3; i4 < PB; i4 += 4) {
        const float4 l = *reinterpret_cast<const float4*>(&lt[m][i4]);
        if (i4 > m) x[i4] = fmaf(-l.x, x[m], x[i4]);
        if (i4 + 1 > m) x[i4 + 1] = fmaf(-l.y, x[m], x[i4 + 1]);
        if (i4 + 2 > m) x[i4 + 2] = fmaf(-l.z, x[m], x[i4 + 2]);
        if (i4 + 3 > m) x[i4 + 3] = fmaf(-l.w, x[m], x[i4 + 3]);
      }
    }
#pragma unroll
    for (int i = 0; i < PB; ++i) xs[buf][i][c] = x[i];
#pragma unroll
    for (int i = 0; i < PB; i += 4)
      *reinterpret_cast<float4*>(&xt[buf][c][i]) = make_float4(x[i] * s_ninv[i], x[i + 1] * s_ninv[i + 1],
                                                               x[i + 2] * s_ninv[i + 2], x[i + 3] * s_ninv[i + 3]);
    if (q + 1 < P) asm volatile("bar.arrive 3, %0;" ::"n"(THREADS) : "memory");
    if (c < n) {
#pragma unroll
      for (int i = 0; i < PB; ++i) R[(size_t)(j0 + i) * ca.ldR + c] = c <= j0 + i ? x[i] * s_rs[i] : 0.f;
    }
  }
  if (bad) atomicMax(&ca.status[b], (int)TC_ERR_BREAKDOWN);
  if (ca.blocked) {
    for (int i = warp - UW; i < n; i += PW)
      for (int k = lane; k < n; k += 32) S[(size_t)i * ca.ldS + k] = (k == i) ? 1.f : 0.f;
    if (ca.first) {
      if (c == 0) ca.largest[(size_t)b * ca.sL] = md;
      for (int i = n + c; i < n + ca.n_rest; i += PW * 32) S[(size_t)i * (ca.ldS + 1)] += ca.shift_rel * md;
    }
  }
  pdl_trigger();
}

template <int NP, int P>
tc_status run(const CholArgs& ca, int batch, cudaStream_t st) {
  constexpr int smem = (3 * PB + 2 * XT_ROW) * 64 * NP * 4;
  auto kernel = chol_inv_kernel<NP, P>;
  if (NP == 3) {   // the split of the registers counts on what the launch brings
    static const int regs = [&] {
      cudaFuncAttributes a;
      return cudaFuncGetAttributes(&a, (const void*)kernel) == cudaSuccess ? a.numRegs : 0;
    }();
    if (regs != 128) return TC_ERR_CUDA;
    if (cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess) return TC_ERR_CUDA;
  }
  static_assert(NP == 3 || smem <= 48 * 1024, "shared memory without opting in");
  if (launch_pdl(kernel, dim3(batch), dim3(WARPS * 32), smem, st, 0, ca) != cudaSuccess) return TC_ERR_CUDA;
  note_launch();
  return TC_OK;
}

tc_status launch_block(const CholArgs& ca, int batch, cudaStream_t st) {
  switch (ca.n / PB) {
    case 1: return run<1, 1>(ca, batch, st);
    case 2: return run<1, 2>(ca, batch, st);
    case 3: return run<1, 3>(ca, batch, st);
    case 4: return run<1, 4>(ca, batch, st);
    case 5: return run<2, 5>(ca, batch, st);
    case 6: return run<2, 6>(ca, batch, st);
    case 7: return run<2, 7>(ca, batch, st);
    case 8: return run<2, 8>(ca, batch, st);
    case 9: return run<3, 9>(ca, batch, st);
    case 10: return run<3, 10>(ca, batch, st);
    case 11: return run<3, 11>(ca, batch, st);
    case 12: return run<3, 12>(ca, batch, st);
    default: return TC_ERR_UNSUPPORTED;
  }
}

}  // namespace

// Orders above CHOL_BLOCK_MAX go block by block (equal blocks, multiples of 16, up to 160: the widest
// tile of the product kernel that keeps the cross terms apart).  Left of the block
// column J that is eliminated, S holds the transposed columns of the inverse so far (from the identity
// on), right of it what is left of S:
//   P = S[:, J] L_JJ^{-T}              (block row J of the inverse, transposed, in the rows left of J)
//   S[:, r] -= P P[r]^T                for the columns r right of J (rows J start from zero)
static int chol_block(int k) {
  const int nb = (k + 159) / 160;
  return ((k + nb - 1) / nb + 15) / 16 * 16;
}
size_t chol_panel_floats(int k) { return k <= CHOL_BLOCK_MAX ? 0 : (size_t)k * chol_block(k) + 4; }

tc_status launch_chol_inv(float* S, float* RinvT, float* panel, int k, int batch, int of_batch, float shift_rel,
                          int32_t* status, cudaStream_t st) {
  if (k < 1 || (k & 15)) return TC_ERR_UNSUPPORTED;
  const size_t sK = (size_t)k * k;
  CholArgs ca;
  ca.sS = ca.sR = sK; ca.ldS = ca.ldR = k; ca.status = status; ca.shift_rel = shift_rel;
  if (k <= CHOL_BLOCK_MAX) {
    Scope scope_(KC_CHOL, st);
    ca.S = S; ca.R = RinvT; ca.n = k;
    ca.blocked = false; ca.first = true; ca.n_rest = 0; ca.largest = nullptr; ca.sL = 0;
    return launch_block(ca, batch, st);
  }
  const int nb = chol_block(k);
  const size_t sP = chol_panel_floats(k);
  if (cudaMemsetAsync(RinvT, 0, (size_t)batch * sK * sizeof(float), st) != cudaSuccess) return TC_ERR_CUDA;
  for (int j0 = 0; j0 < k; j0 += nb) {
    const int w = k - j0 < nb ? k - j0 : nb, j1 = j0 + w;
    {
      Scope scope_(KC_CHOL, st);
      ca.S = S + (size_t)j0 * (k + 1); ca.R = RinvT + (size_t)j0 * (k + 1); ca.n = w;
      ca.blocked = true; ca.first = j0 == 0; ca.n_rest = j0 == 0 ? k - w : 0;
      ca.largest = panel + (size_t)k * nb; ca.sL = sP;
      const tc_status e = launch_block(ca, batch, st);
      if (e != TC_OK) return e;
    }
    if (j0 == 0 && j1 == k) break;
    F32x3Result rp;
    rp.C = panel; rp.ld = w; rp.stride = sP;
    rp.CT = RinvT + (size_t)j0 * k; rp.ldT = k; rp.strideT = sK; rp.rows_t = j0;
    tc_status e = launch_gemm_f32x3({S + j0, k, sK}, {RinvT + (size_t)j0 * (k + 1), k, sK}, k, w, w, batch, of_batch, rp, status,
                                    st, KC_CHOL);
    if (e != TC_OK) return e;
    if (j1 < k) {
      F32x3Result rs;
      rs.C = S + j1; rs.ld = k; rs.stride = sK;
      rs.CT = nullptr; rs.ldT = 0; rs.strideT = 0;
      rs.subtract = true; rs.zero_from = j0; rs.zero_to = j1;
      e = launch_gemm_f32x3({panel, w, sP}, {panel + (size_t)j1 * w, w, sP}, k, k - j1, w, batch, of_batch, rs, status, st, KC_CHOL);
      if (e != TC_OK) return e;
    }
  }
  return TC_OK;
}

// ------------------------------------------------------------------------------------------
// The same for a wide basis (float32 multiply-adds only): every entry of the factor and of the inverse
// is the chain of multiply-adds that the textbook loops give, in their order, whatever the tiling.
//   chol_f32_prepare   adds the shift, keeps the largest diagonal entry
//   chol_f32_panel     32 rows of the factor: every block factors the diagonal block for itself (one
//                      warp), then a thread per column substitutes
//   chol_f32_update    S[r][c] -= sum_m F[m][r] F[m][c] over those 32 rows, 64 x 64 tiles
//   chol_f32_inverse   a warp per four columns of the inverse, back substitution
// What bounds the first three is 2 k / 32 dependent launches of about 4 us, the last one a chain of k
// steps of 400 to 900 cycles.  Measured at k = 736, four matrices: 62 ms (one block per matrix, out of
// L2) -> 1.0 ms, half of it the inverse.
// ------------------------------------------------------------------------------------------
namespace {

constexpr int WB = 32;  // rows per step

__global__ void __launch_bounds__(256) chol_f32_prepare(float* __restrict__ S, float* __restrict__ F, int k,
                                                       float shift_rel) {
  __shared__ float s_red[8];
  pdl_wait();
  pdl_trigger();
  float* Sb = S + (size_t)blockIdx.x * k * k;
  float md = 0.f;
  for (int i = threadIdx.x; i < k; i += 256) md = fmaxf(md, Sb[(size_t)i * (k + 1)]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = md;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) md = fmaxf(md, s_red[w]);
  const float shift = shift_rel * md;
  for (int i = threadIdx.x; i < k; i += 256) Sb[(size_t)i * (k + 1)] += shift;
  if (threadIdx.x == 0) F[(size_t)blockIdx.x * k * k + (size_t)(k - 1) * k] = md;  // (below the diagonal: free)
}

// grid (column tiles of 128, batch), block 128
__global__ void __launch_bounds__(128) chol_f32_panel(const float* __restrict__ S, float* __restrict__ F, int k, int j0,
                                                     int32_t* __restrict__ status) {
  __shared__ float D[WB][WB + 1];
  __shared__ float s_inv[WB];
  const int tid = threadIdx.x, lane = tid & 31, b = blockIdx.y;
  const int w = min(WB, k - j0);
  pdl_wait();
  pdl_trigger();
  const float* Sb = S + (size_t)b * k * k;
  float* Fb = F + (size_t)b * k * k;
  for (int e = tid; e < WB * WB; e += 128) {
    const int r = e >> 5, c = e & 31;
    D[r][c] = (r < w && c < w && c >= r) ? Sb[(size_t)(j0 + r) * k + j0 + c] : 0.f;
  }
  const int c = j0 + w + blockIdx.x * 128 + tid;
  float x[WB];
#pragma unroll
  for (int i = 0; i < WB; ++i) x[i] = (i < w && c < k) ? Sb[(size_t)(j0 + i) * k + c] : 0.f;
  __syncthreads();
  if (tid < 32) {
    const float md = Fb[(size_t)(k - 1) * k];
    float col[WB];  // lane = column of the block
#pragma unroll
    for (int r = 0; r < WB; ++r) col[r] = D[r][lane];
    __syncwarp();
    bool bad = false;
#pragma unroll
    for (int j = 0; j < WB; ++j) {
      if (j < w) {
        float p = __shfl_sync(0xffffffffu, col[j], j);
        if (!(p > 0.f)) {
          p = fmaxf(md, 1e-30f) * 1e-12f;
          bad = true;
        }
        const float dj = sqrtf(p), inv = 1.0f / dj;
        col[j] = (lane == j) ? dj : col[j] * inv;
        if (lane == 0) s_inv[j] = inv;
        // row j of the factor goes through shared memory: broadcast reads pipeline, shuffles do not
        D[j][lane] = col[j];
        __syncwarp();
#pragma unroll
        for (int r = j + 1; r < WB; ++r) {
          const float f = D[j][r];
          if (lane >= r) col[r] = fmaf(-f, col[j], col[r]);
        }
      }
    }
    if (blockIdx.x == 0) {
#pragma unroll
      for (int r = 0; r < WB; ++r)
        if (r <= lane && lane < w) Fb[(size_t)(j0 + r) * k + j0 + lane] = col[r];
      if (bad && lane == 0) atomicMax(&status[b], (int)TC_ERR_BREAKDOWN);
    }
  }
  __syncthreads();
  if (c >= k) return;
#pragma unroll
  for (int m = 0; m < WB; ++m) {
    if (m < w) {
      x[m] *= s_inv[m];
      Fb[(size_t)(j0 + m) * k + c] = x[m];
#pragma unroll
      for (int j = m + 1; j < WB; ++j) x[j] = fmaf(-D[m][j], x[m], x[j]);
    }
  }
}

// grid (tiles of 64 x 64 on or above the diagonal of what is left, batch), block 256, 4 x 4 per thread
__global__ void __launch_bounds__(256) chol_f32_update(float* __restrict__ S, const float* __restrict__ F, int k, int j0,
                                                      int j1) {
  __shared__ __align__(16) float fr[WB][64], fc[WB][64];
  int t = blockIdx.x, tj = 0;  // t -> (ti <= tj): t = tj (tj + 1) / 2 + ti
  while ((tj + 1) * (tj + 2) / 2 <= t) ++tj;
  pdl_wait();
  pdl_trigger();
  const int ti = t - tj * (tj + 1) / 2;
  const int r0 = j1 + ti * 64, c0 = j1 + tj * 64, tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  float* Sb = S + (size_t)blockIdx.y * k * k;
  const float* Fb = F + (size_t)blockIdx.y * k * k;
  for (int e = tid; e < WB * 64; e += 256) {
    const int m = e >> 6, i = e & 63;
    fr[m][i] = (r0 + i < k) ? Fb[(size_t)(j0 + m) * k + r0 + i] : 0.f;
    fc[m][i] = (c0 + i < k) ? Fb[(size_t)(j0 + m) * k + c0 + i] : 0.f;
  }
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = r0 + 4 * ty + i, c = c0 + 4 * tx + j;
      acc[i][j] = (r < k && c < k && c >= r) ? Sb[(size_t)r * k + c] : 0.f;
    }
  __syncthreads();
#pragma unroll 8
  for (int m = 0; m < j1 - j0; ++m) {
    const float4 a4 = *reinterpret_cast<const float4*>(&fr[m][4 * ty]), b4 = *reinterpret_cast<const float4*>(&fc[m][4 * tx]);
    const float a[4] = {a4.x, a4.y, a4.z, a4.w}, bb[4] = {b4.x, b4.y, b4.z, b4.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(-a[i], bb[j], acc[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int r = r0 + 4 * ty + i, c = c0 + 4 * tx + j;
      if (r < k && c < k && c >= r) Sb[(size_t)r * k + c] = acc[i][j];
    }
}

// XT[c][m] = (R^{-1})[m][c], zero for m > c.  grid (ceil(k / 16), batch), block 128: a warp per four
// columns c, c - 1, ..., the long columns first.  A row of the factor is read once for the four, two
// steps ahead; the steps come in phases of 128 whose code has no test that would keep the reads and
// multiply-adds of a step from overlapping.
template <int T>  // k <= 32 T
__global__ void __launch_bounds__(128) chol_f32_inverse(const float* __restrict__ F, float* __restrict__ XT, int k) {
  extern __shared__ float xs[];  // [4 warps][4 columns][k]
  constexpr int Q = T / 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.y;
  const int c0 = k - 1 - 4 * (blockIdx.x * 4 + warp);
  pdl_wait();
  pdl_trigger();
  if (c0 < 0) return;
  const float* R = F + (size_t)b * k * k;
  float* x = xs + (size_t)warp * 4 * k;
  float rv[2][T], dv[2];
  // NQ: groups of 128 entries that a row holds in the current phase
  auto fetch = [&](int i, int buf, auto nq) {  // entries i + 1 + lane + 32 t <= c0 of row i, and its diagonal
    if (i < 0) return;
    const float* row = R + (size_t)i * k + i + 1 + lane;
    const int left = c0 - i - 1 - lane;  // >= 32 t: entry t exists
#pragma unroll
    for (int t = 0; t < 4 * decltype(nq)::value; ++t) rv[buf][t] = (left >= 32 * t) ? __ldg(row + 32 * t) : 0.f;
    dv[buf] = __ldg(R + (size_t)i * k + i);
  };
  auto step = [&](int i, int buf, auto nq) {
    if (i < 0) return;
    constexpr int NT = 4 * decltype(nq)::value;
    const int left = c0 - i - 1 - lane;
    float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
    for (int t = 0; t < NT; ++t) {
      const float* xt = x + i + 1 + lane + 32 * t;
#pragma unroll
      for (int col = 0; col < 4; ++col)
        if (left - col >= 32 * t) s[col] = fmaf(rv[buf][t], xt[col * k], s[col]);
    }
    const float d = dv[buf];
    // (the next phase begins within two steps: it may need a group more)
    fetch(i - 2, buf, std::integral_constant<int, (NT / 4 < Q) ? NT / 4 + 1 : Q>{});
    // the four sums over the lanes, pairwise in the order of a butterfly: lanes 8 col .. get column col
    {
      const bool up = (lane & 16) != 0;
      const float a0 = (up ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, up ? s[0] : s[2], 16);
      const float a1 = (up ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, up ? s[1] : s[3], 16);
      const bool up8 = (lane & 8) != 0;
      float a = (up8 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, up8 ? a0 : a1, 8);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
      const int col = lane >> 3, c = c0 - col;
      if ((lane & 7) == 0 && i <= c) x[col * k + i] = (i == c ? 1.0f : -a) / d;
    }
    __syncwarp();
  };
  fetch(c0, 0, std::integral_constant<int, 1>{});
  fetch(c0 - 1, 1, std::integral_constant<int, 1>{});
  // steps j = c0 - i in phases of 128
  auto phase = [&](auto nq) {
    constexpr int NQ = decltype(nq)::value;
    if constexpr (NQ <= Q) {
      for (int j = 128 * (NQ - 1); j < 128 * NQ && j <= c0; j += 2) {
        step(c0 - j, 0, nq);
        step(c0 - j - 1, 1, nq);
      }
    }
  };
  phase(std::integral_constant<int, 1>{});
  phase(std::integral_constant<int, 2>{});
  phase(std::integral_constant<int, 3>{});
  phase(std::integral_constant<int, 4>{});
  phase(std::integral_constant<int, 5>{});
  phase(std::integral_constant<int, 6>{});
  phase(std::integral_constant<int, 7>{});
  phase(std::integral_constant<int, 8>{});
  for (int col = 0; col < 4 && c0 - col >= 0; ++col) {
    const int c = c0 - col;
    float* out = XT + ((size_t)b * k + c) * k;
    for (int m = lane; m < k; m += 32) out[m] = (m <= c) ? x[col * k + m] : 0.f;
  }
}

}  // namespace

void launch_chol_inv_f32(float* S, float* RinvT, float* F, int k, int batch, float shift_rel, int32_t* status,
                         cudaStream_t st) {
  Scope scope_(KC_CHOL, st);
  launch_pdl(chol_f32_prepare, dim3(batch), dim3(256), 0, st, 0, S, F, k, shift_rel);
  note_launch();
  for (int j0 = 0; j0 < k; j0 += WB) {
    const int j1 = j0 + WB < k ? j0 + WB : k, left = k - j1;
    launch_pdl(chol_f32_panel, dim3(left > 0 ? (left + 127) / 128 : 1, batch), dim3(128), 0, st, 0, S, F, k, j0, status);
    note_launch();
    if (left > 0) {
      const int nt = (left + 63) / 64;
      launch_pdl(chol_f32_update, dim3(nt * (nt + 1) / 2, batch), dim3(256), 0, st, 0, S, F, k, j0, j1);
      note_launch();
    }
  }
  const size_t smem = (size_t)16 * k * sizeof(float);
  const dim3 grid((k + 15) / 16, batch);
  auto inverse = [&](auto kernel) {
    cudaFuncSetAttribute((const void*)kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_pdl(kernel, grid, dim3(128), smem, st, 0, F, RinvT, k);
  };
  if (k <= 512) inverse(chol_f32_inverse<16>);
  else if (k <= 768) inverse(chol_f32_inverse<24>);
  else inverse(chol_f32_inverse<32>);
  note_launch();
}

}  // namespace tc
