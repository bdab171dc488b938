// Inverse Cholesky factor of a symmetric matrix S (+ shift), order up to 192, one block per matrix:
// RinvT = L^{-1} with L L^T = S + shift_rel max_i S_ii I, so that Y RinvT^T has (nearly) orthonormal
// columns when S = Y^T Y: one pass of Cholesky-QR behind Eq. 3-5.  The shift keeps the factorisation
// alive when S is numerically singular; a later pass with a smaller one removes its effect.
//
// Elimination of S next to the identity: step j subtracts multiples of row j from the rows below, in S
// (columns right of j) and in what was the identity (columns left of j), which takes the place of the
// columns of S that are finished.  A row is scaled by the root of its pivot at the end.
// What bounds it is the latency of a step, in a chain of n: the matrix lives in registers (rows dealt
// cyclically over eight warps, two neighbouring columns of each 64 per lane), two steps at a time
// exchange their two rows through shared memory, behind one barrier, and the warp that owns the next
// two rows updates and publishes them before it goes on with its other rows.
// The steps come in phases of 32: the code of a phase covers, without any test, the rows that are not
// finished when it begins.
// Measured, 16 matrices: order 144 and 160, 53 and 62 us with the matrix in shared memory and blocks of
// 16 columns -> 39 and 47 us here; a pair of steps takes 1000 cycles at order 160, of which the
// multiply-adds are 240.
#include "pair_math.cuh"
#include "tc_internal.cuh"

#include <type_traits>

namespace tc {

namespace {

constexpr int CW = 8;  // warps

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

// NP: 64-column groups, RW: rows per warp (n <= 8 RW).  Rows go to the warps in pairs: row 16 i' + 2 w + u
// is row 2 i' + u of warp w.
template <int NP, int RW>
__global__ void __launch_bounds__(CW * 32, 1) chol_inv_reg_kernel(const CholArgs ca) {
  constexpr int NC = 64 * NP;
  constexpr int NPH = (RW + 3) / 4;                       // phases of 32 columns = 4 rows of a warp
  __shared__ __align__(16) float rowp[2][2][NC];          // rows j, j + 1 as the others subtract them
  __shared__ __align__(16) float rowr[2][2][CW][(RW + 3) & ~3];  // their entries below the pivots, by owner of the row of that number
  __shared__ float2 s_piv[2];
  __shared__ float s_pv[NC];                              // pivots
  __shared__ float s_red[CW];
  __shared__ int s_bad;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, b = blockIdx.x;
  const int n = ca.n;
  float* S = ca.S + (size_t)b * ca.sS;
  pdl_wait();
  auto row_of = [&](int i) { return 16 * (i >> 1) + 2 * warp + (i & 1); };

  f2 B[RW][NP];
#pragma unroll
  for (int i = 0; i < RW; ++i)
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int r = row_of(i), c = 2 * lane + 64 * p;
      B[i][p] = (r < n && c < n) ? *reinterpret_cast<const f2*>(S + (size_t)r * ca.ldS + c) : 0ull;
    }
  float md = 0.f;
  for (int i = threadIdx.x; i < n + ca.n_rest; i += CW * 32) md = fmaxf(md, S[(size_t)i * (ca.ldS + 1)]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
  if (lane == 0) s_red[warp] = md;
  if (threadIdx.x == 0) s_bad = 0;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < CW; ++w) md = fmaxf(md, s_red[w]);
  if (ca.blocked && !ca.first) md = ca.largest[(size_t)b * ca.sL];
  const float shift = ca.first ? ca.shift_rel * md : 0.f;
  // A direction of S under the rounding level of its entries can leave any pivot: one below 2.5e-7 of
  // the largest entry is raised to that.  Only a pivot that is negative by far more than rounding (or
  // no number) says that S is not what it should be.
  const float floor_p = 2.5e-7f * fmaxf(md, 1e-30f);
  const float bad_p = -1e-5f * md;
#pragma unroll
  for (int i = 0; i < RW; ++i)
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int r = row_of(i), c = 2 * lane + 64 * p;
      float2 t = upk(B[i][p]);
      if (c == r) t.x += shift;
      if (c + 1 == r) t.y += shift;
      B[i][p] = pk(t.x, t.y);
    }
  if (ca.blocked) {
#pragma unroll
    for (int i = 0; i < RW; ++i) {
      const int r = row_of(i);
      for (int c = lane; c < n && r < n; c += 32) S[(size_t)r * ca.ldS + c] = (c == r) ? 1.f : 0.f;
    }
    if (ca.first) {
      if (threadIdx.x == 0) ca.largest[(size_t)b * ca.sL] = md;
      for (int i = n + threadIdx.x; i < n + ca.n_rest; i += CW * 32) S[(size_t)i * (ca.ldS + 1)] += shift;
    }
  }

  // rows j, j + 1 (j even) by their owner; their register indices lie in [I, I + 6).  Row j + 1 is
  // published with step j applied to it (the owner's registers get that like everyone's, later).
  auto publish = [&](int j, auto ic) {
    constexpr int I = decltype(ic)::value;
    if (((j >> 1) & (CW - 1)) == warp && j < n) {
      f2 ra[NP], rb[NP];
      const uint32_t at = 1u << (2 * (j >> 4)), atp = 1u << (j >> 6);
      f2 ap = 0ull, bp = 0ull;  // columns j, j + 1 of both
#pragma unroll
      for (int i = I; i < I + 6 && i + 1 < RW; i += 2)
        if ((at >> i) & 1u) {
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            ra[p] = B[i][p];
            rb[p] = B[i + 1][p];
            if ((atp >> p) & 1u) {
              ap = ra[p];
              bp = rb[p];
            }
          }
        }
      const int src = (j & 63) >> 1;
      const float2 a2 = upk(ap), b2 = upk(bp);
      const float pj = __shfl_sync(0xffffffffu, a2.x, src), sj = __shfl_sync(0xffffffffu, a2.y, src);
      const float qj = __shfl_sync(0xffffffffu, b2.y, src);
      const float m = -sj * rcp_newton(fmaxf(pj, floor_p));
      const f2 m2 = pk(m, m);
#pragma unroll
      for (int p = 0; p < NP; ++p) {
        const int c = 2 * lane + 64 * p;
        const float2 x = upk(ra[p]), y = upk(fma2(m2, ra[p], rb[p]));
        const bool here = c == j, right = c > j;
        *reinterpret_cast<float2*>(&rowp[(j >> 1) & 1][0][c]) = make_float2(here ? 1.f : x.x, here ? 0.f : x.y);
        *reinterpret_cast<float2*>(&rowp[(j >> 1) & 1][1][c]) = make_float2(here ? m : y.x, here ? 1.f : y.y);
        if (c < 8 * RW) {
          const int w = (c >> 1) & (CW - 1), i = 2 * (c >> 4);
          *reinterpret_cast<float2*>(&rowr[(j >> 1) & 1][0][w][i]) = make_float2(right ? x.x : 0.f, here || right ? x.y : 0.f);
          *reinterpret_cast<float2*>(&rowr[(j >> 1) & 1][1][w][i]) = make_float2(right ? y.x : 0.f, right ? y.y : 0.f);
        }
      }
      if (lane == 0) s_piv[(j >> 1) & 1] = make_float2(pj, fmaf(m, sj, qj));
    }
  };
  publish(0, std::integral_constant<int, 0>{});
  int j = 0;
  auto phase = [&](auto fc) {
    constexpr int F = decltype(fc)::value, I0 = 4 * F, PJ = F / 2;
    if constexpr (F < NPH) {
      for (; j < n && j < 32 * (F + 1); j += 2) {
        __syncthreads();  // rows j, j + 1 are there, and everyone has read the two before
        const int buf = (j >> 1) & 1;
        const float2 piv = s_piv[buf];
        const float pa = fmaxf(piv.x, floor_p), pb = fmaxf(piv.y, floor_p);
        const float ma = -rcp_newton(pa), mb = -rcp_newton(pb);
        f2 xa[NP], xb[NP];
#pragma unroll
        for (int p = 0; p < NP; ++p) {
          xa[p] = *reinterpret_cast<const f2*>(&rowp[buf][0][2 * lane + 64 * p]);
          xb[p] = *reinterpret_cast<const f2*>(&rowp[buf][1][2 * lane + 64 * p]);
        }
        // columns j, j + 1 of the rows below start over as columns of the inverse
        const f2 keep = (2 * lane + 64 * PJ == j) ? 0ull : pk(1.f, 1.f);
        auto update = [&](int i, float la, float lb) {
          const float ua = la * ma, ub = lb * mb;
          const f2 ua2 = pk(ua, ua), ub2 = pk(ub, ub);
#pragma unroll
          for (int p = 0; p < NP; ++p)
            B[i][p] = fma2(ub2, xb[p], fma2(ua2, xa[p], p == PJ ? mul2(keep, B[i][p]) : B[i][p]));
        };
        auto update2 = [&](int i) {  // rows i, i + 1
          const float2 la = *reinterpret_cast<const float2*>(&rowr[buf][0][warp][i]);
          const float2 lb = *reinterpret_cast<const float2*>(&rowr[buf][1][warp][i]);
          update(i, la.x, lb.x);
          update(i + 1, la.y, lb.y);
        };
#pragma unroll
        for (int i = I0; i < I0 + 6 && i < RW; i += 2) update2(i);
        publish(j + 2, std::integral_constant<int, I0>{});
#pragma unroll
        for (int i = I0 + 6; i < RW; i += 2) update2(i);
        if (threadIdx.x == 32 * (CW - 1)) {
          s_pv[j] = pa;
          s_pv[j + 1] = pb;
          if (!(piv.x > bad_p) || !(piv.y > bad_p)) s_bad = 1;
        }
      }
    }
  };
  phase(std::integral_constant<int, 0>{});
  phase(std::integral_constant<int, 1>{});
  phase(std::integral_constant<int, 2>{});
  phase(std::integral_constant<int, 3>{});
  phase(std::integral_constant<int, 4>{});
  phase(std::integral_constant<int, 5>{});
  __syncthreads();
  pdl_trigger();
  if (threadIdx.x == 0 && s_bad) atomicMax(&ca.status[b], (int)TC_ERR_BREAKDOWN);
  float* R = ca.R + (size_t)b * ca.sR;
#pragma unroll
  for (int i = 0; i < RW; ++i) {
    const int r = row_of(i);
    if (r >= n) continue;
    const float rs = rsqrtf(s_pv[r]);
#pragma unroll
    for (int p = 0; p < NP; ++p) {
      const int c = 2 * lane + 64 * p;
      const float2 t = upk(B[i][p]);
      if (c < n)
        *reinterpret_cast<float2*>(R + (size_t)r * ca.ldR + c) =
            make_float2(c < r ? t.x * rs : (c == r ? rs : 0.f), c + 1 < r ? t.y * rs : (c + 1 == r ? rs : 0.f));
    }
  }
}

template <int NP, int RW>
void run(const CholArgs& ca, int batch, cudaStream_t st) {
  launch_pdl(chol_inv_reg_kernel<NP, RW>, dim3(batch), dim3(CW * 32), 0, st, 0, ca);
  note_launch();
}

void launch_block(const CholArgs& ca, int batch, cudaStream_t st) {
  if (ca.n <= 64) run<1, 8>(ca, batch, st);
  else if (ca.n <= 96) run<2, 12>(ca, batch, st);
  else if (ca.n <= 128) run<2, 16>(ca, batch, st);
  else if (ca.n <= 144) run<3, 18>(ca, batch, st);
  else if (ca.n <= 160) run<3, 20>(ca, batch, st);
  else run<3, 24>(ca, batch, st);
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
    launch_block(ca, batch, st);
    return TC_OK;
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
      launch_block(ca, batch, st);
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
