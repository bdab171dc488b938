// Dense linear algebra behind Eq. 3-5 / 3-6: the eigen-decomposition of the Gram matrix
// G = O O^T = U Sigma^2 U^T, which yields the singular values and the rows of U Sigma that the
// information contribution score sums.
//
// Two routes, chosen by rank_cap:
//   full      the Gram matrix itself: reduction to tridiagonal form (eig_tridiag.cu), or one-sided
//             Jacobi (columns of W = G J are orthogonalised; the accumulated rotations J are the
//             eigenvectors, the column norms the eigenvalues) where eigenvectors under the rounding
//             level are wanted, see use_tridiag.
//   subspace  when the caller bounds the numerical rank by k < N: a k-dimensional dominant
//             subspace is built (sign sketch of O, one multiplication by G, Cholesky-QR
//             orthonormalisation), G is projected onto it (Rayleigh-Ritz) and only the k x k
//             projection is decomposed.
#include <cooperative_groups.h>

#include "tc_internal.cuh"

#include <utility>

namespace tc {

// ==========================================================================================
// Batched float32 GEMM on the plain ALUs:  C[m][n] = sum_k opA[m][k] * opB[k][n].
//   opA[m][k] = TRA ? A[k * lda + m] : A[m * lda + k]
//   opB[k][n] = TRB ? B[n * ldb + k] : B[k * ldb + n]
// 64 x 64 tile per block, 16-deep slices, 4 x 4 outputs per thread.  blockIdx.z = batch.
// ==========================================================================================
__device__ inline float ld_f32(const float* p) { return __ldg(p); }
__device__ inline float ld_f32(const __half* p) { return __half2float(__ldg(p)); }
__device__ inline float ld_f32(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// flags for structured products
constexpr int GEMM_SYM = 1;       // C is symmetric (A^T A): tiles below the diagonal are mirrored
constexpr int GEMM_B_UPPER = 2;   // opB[k][n] = 0 for k > n: the K loop stops at the tile's edge

template <typename TA, typename TB, bool TRA, bool TRB, int RM, int CN>
__global__ void __launch_bounds__(256) gemm_kernel(const TA* __restrict__ A,
                                                  const TB* __restrict__ B, float* __restrict__ C,
                                                  int M, int N, int K, int lda, int ldb, int ldc,
                                                  size_t sA, size_t sB, size_t sC, int flags) {
  // (64 RM) x (16 CN) tile per block, 16-deep slices, (4 RM) x CN outputs per thread.  The next
  // slice is fetched into registers while the current one is multiplied out of shared memory.
  // CN = 4 gives 64-column tiles, CN = 3 gives 48-column tiles (for widths like 144 = 3 * 48).
  constexpr int BM = 64 * RM, BN = 16 * CN, BK = 16;
  constexpr int LA = BM * BK / 256, LB = BN * BK / 256;
  __shared__ __align__(16) float As[BK][BM + 4];
  __shared__ __align__(16) float Bs[BK][BN + 4];
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  pdl_wait();
  pdl_trigger();
  if ((flags & GEMM_SYM) && n0 + BN <= m0) return;  // strictly below the diagonal
  A += (size_t)blockIdx.z * sA;
  B += (size_t)blockIdx.z * sB;
  C += (size_t)blockIdx.z * sC;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int Kend = (flags & GEMM_B_UPPER) ? min(K, n0 + BN) : K;
  float acc[4 * RM][CN];
#pragma unroll
  for (int i = 0; i < 4 * RM; ++i)
#pragma unroll
    for (int j = 0; j < CN; ++j) acc[i][j] = 0.f;
  // Slices are fetched as 16-byte vectors along the contiguous direction of each operand when
  // every address involved is 16-byte aligned (float32 operands, leading dimensions, sizes and
  // batch strides multiples of four); otherwise element by element.
  constexpr bool F32 = (sizeof(TA) == 4) && (sizeof(TB) == 4);
  const bool vec = F32 && ((lda | ldb | M | N | K) & 3) == 0 && ((sA | sB) & 3) == 0 &&
                   ((((uintptr_t)A) | ((uintptr_t)B)) & 15) == 0;
  constexpr int VA = LA / 4, VB = (LB + 3) / 4;  // vectors per thread (B: some threads idle)
  float ra[LA], rb[VB * 4];

  auto fetch = [&](int k0) {
    if (vec) {
#pragma unroll
      for (int i = 0; i < VA; ++i) {
        const int e = tid + i * 256;  // vector index inside the A slice
        int m, k;
        if (TRA) {  // stored [k][m]: vectors run along m
          m = (e % (BM / 4)) * 4;
          k = e / (BM / 4);
        } else {  // stored [m][k]: vectors run along k
          k = (e & 3) * 4;
          m = e >> 2;
        }
        const int gm = m0 + m, gk = k0 + k;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (gm < M && gk < Kend)
          v = __ldg(reinterpret_cast<const float4*>(
              TRA ? (const float*)A + (size_t)gk * lda + gm : (const float*)A + (size_t)gm * lda + gk));
        ra[4 * i] = v.x; ra[4 * i + 1] = v.y; ra[4 * i + 2] = v.z; ra[4 * i + 3] = v.w;
      }
#pragma unroll
      for (int i = 0; i < VB; ++i) {
        const int e = tid + i * 256;
        float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
        if (e < BN * BK / 4) {
          int n, k;
          if (TRB) {  // stored [n][k]: vectors run along k
            k = (e & 3) * 4;
            n = e >> 2;
          } else {  // stored [k][n]: vectors run along n
            n = (e % (BN / 4)) * 4;
            k = e / (BN / 4);
          }
          const int gn = n0 + n, gk = k0 + k;
          if (gn < N && gk < Kend)
            v = __ldg(reinterpret_cast<const float4*>(
                TRB ? (const float*)B + (size_t)gn * ldb + gk : (const float*)B + (size_t)gk * ldb + gn));
        }
        rb[4 * i] = v.x; rb[4 * i + 1] = v.y; rb[4 * i + 2] = v.z; rb[4 * i + 3] = v.w;
      }
      return;
    }
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      const int e = tid + i * 256;
      int m, k;
      if (TRA) {
        m = e % BM;
        k = e / BM;
      } else {
        k = e & 15;
        m = e >> 4;
      }
      const int gm = m0 + m, gk = k0 + k;
      float v = 0.f;
      if (gm < M && gk < Kend) v = TRA ? ld_f32(A + (size_t)gk * lda + gm) : ld_f32(A + (size_t)gm * lda + gk);
      ra[i] = v;
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
      const int e = tid + i * 256;
      int n, k;
      if (TRB) {
        k = e & 15;
        n = e >> 4;
      } else {
        n = e % BN;
        k = e / BN;
      }
      const int gn = n0 + n, gk = k0 + k;
      float v = 0.f;
      if (gn < N && gk < Kend) v = TRB ? ld_f32(B + (size_t)gn * ldb + gk) : ld_f32(B + (size_t)gk * ldb + gn);
      rb[i] = v;
    }
  };
  auto stash = [&]() {
    if (vec) {
#pragma unroll
      for (int i = 0; i < VA; ++i) {
        const int e = tid + i * 256;
        if (TRA) {
          const int m = (e % (BM / 4)) * 4, k = e / (BM / 4);
          *reinterpret_cast<float4*>(&As[k][m]) = make_float4(ra[4 * i], ra[4 * i + 1], ra[4 * i + 2], ra[4 * i + 3]);
        } else {
          const int k = (e & 3) * 4, m = e >> 2;
#pragma unroll
          for (int u = 0; u < 4; ++u) As[k + u][m] = ra[4 * i + u];
        }
      }
#pragma unroll
      for (int i = 0; i < VB; ++i) {
        const int e = tid + i * 256;
        if (e < BN * BK / 4) {
          if (TRB) {
            const int k = (e & 3) * 4, n = e >> 2;
#pragma unroll
            for (int u = 0; u < 4; ++u) Bs[k + u][n] = rb[4 * i + u];
          } else {
            const int n = (e % (BN / 4)) * 4, k = e / (BN / 4);
            *reinterpret_cast<float4*>(&Bs[k][n]) = make_float4(rb[4 * i], rb[4 * i + 1], rb[4 * i + 2], rb[4 * i + 3]);
          }
        }
      }
      return;
    }
#pragma unroll
    for (int i = 0; i < LA; ++i) {
      const int e = tid + i * 256;
      if (TRA) As[e / BM][e % BM] = ra[i];
      else As[e & 15][e >> 4] = ra[i];
    }
#pragma unroll
    for (int i = 0; i < LB; ++i) {
      const int e = tid + i * 256;
      if (TRB) Bs[e & 15][e >> 4] = rb[i];
      else Bs[e / BN][e % BN] = rb[i];
    }
  };

  fetch(0);
  for (int k0 = 0; k0 < Kend; k0 += BK) {
    stash();
    __syncthreads();
    if (k0 + BK < Kend) fetch(k0 + BK);
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float4 av[RM];
#pragma unroll
      for (int g = 0; g < RM; ++g) av[g] = *reinterpret_cast<const float4*>(&As[kk][g * 64 + ty * 4]);
      float bb[CN];
      if (CN == 4) {
        const float4 bv = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
        bb[0] = bv.x; bb[1] = bv.y; bb[2] = bv.z; bb[CN - 1] = bv.w;
      } else {
#pragma unroll
        for (int j = 0; j < CN; ++j) bb[j] = Bs[kk][tx * CN + j];
      }
#pragma unroll
      for (int g = 0; g < RM; ++g) {
        const float a[4] = {av[g].x, av[g].y, av[g].z, av[g].w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < CN; ++j) acc[g * 4 + i][j] = fmaf(a[i], bb[j], acc[g * 4 + i][j]);
      }
    }
    __syncthreads();
  }
  // symmetric output: a tile writes its entries on or above the diagonal and their mirror
  // images, so each pair is produced exactly once and C is symmetric bit for bit
  const bool sym = (flags & GEMM_SYM) != 0;
#pragma unroll
  for (int g = 0; g < RM; ++g)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int gm = m0 + g * 64 + ty * 4 + i;
      if (gm >= M) continue;
#pragma unroll
      for (int j = 0; j < CN; ++j) {
        const int gn = n0 + tx * CN + j;
        if (gn < N && (!sym || gn >= gm)) {
          C[(size_t)gm * ldc + gn] = acc[g * 4 + i][j];
          if (sym && gn > gm) C[(size_t)gn * ldc + gm] = acc[g * 4 + i][j];
        }
      }
    }
}

template <typename TA, typename TB, bool TRA, bool TRB, int RM, int CN>
static void gemm_launch(const TA* A, const TB* B, float* C, int M, int N, int K, int lda, int ldb,
                        int ldc, size_t sA, size_t sB, size_t sC, int batch, cudaStream_t st,
                        int flags) {
  dim3 grid((N + 16 * CN - 1) / (16 * CN), (M + 64 * RM - 1) / (64 * RM), batch);
  { launch_pdl(gemm_kernel<TA, TB, TRA, TRB, RM, CN>, grid, dim3(256), 0, st, 0, A, B, C, M, N, K, lda, ldb, ldc, sA, sB, sC, flags); note_launch(); }
}

template <typename TA, typename TB, bool TRA, bool TRB>
static void gemm(const TA* A, const TB* B, float* C, int M, int N, int K, int lda, int ldb,
                 int ldc, size_t sA, size_t sB, size_t sC, int batch, cudaStream_t st,
                 int cls = KC_GEMM, int flags = 0) {
  Scope scope_(cls, st);
  // column tiles of 48 when they pad the width less than tiles of 64 (e.g. 144 = 3 * 48)
  const bool narrow = ((N + 47) / 48) * 48 < ((N + 63) / 64) * 64;
  if (M >= 256 && !(flags & GEMM_SYM)) {
    if (narrow) gemm_launch<TA, TB, TRA, TRB, 2, 3>(A, B, C, M, N, K, lda, ldb, ldc, sA, sB, sC, batch, st, flags);
    else gemm_launch<TA, TB, TRA, TRB, 2, 4>(A, B, C, M, N, K, lda, ldb, ldc, sA, sB, sC, batch, st, flags);
  } else {
    if (narrow) gemm_launch<TA, TB, TRA, TRB, 1, 3>(A, B, C, M, N, K, lda, ldb, ldc, sA, sB, sC, batch, st, flags);
    else gemm_launch<TA, TB, TRA, TRB, 1, 4>(A, B, C, M, N, K, lda, ldb, ldc, sA, sB, sC, batch, st, flags);
  }
}

// G = O O^T for float32 inputs.
tc_status launch_gram_simt(const Dims& D, const void* O, float* G, int ldg, cudaStream_t st) {
  const size_t sO = (size_t)D.N * D.d, sG = (size_t)D.N * ldg;
  gemm<float, float, false, true>((const float*)O, (const float*)O, G, D.N, D.N, D.d, D.d, D.d, ldg, sO, sO, sG,
                                  D.B, st, KC_GRAM);
  return TC_OK;
}

// ==========================================================================================
// Sign sketch of O:  Y[x][j] = sum over columns c == j (mod k) of s(c) O[x][c],  s(c) = +-1
// from a fixed integer hash.  grid (N, B), block k.  It only has to capture the dominant
// column space of O; the steps after it correct it against G itself.
// ==========================================================================================
__device__ inline float hash_sign(uint32_t c) {
  uint32_t h = c * 2654435761u;
  h ^= h >> 15;
  h *= 2246822519u;
  h ^= h >> 13;
  return (h & 1u) ? 1.f : -1.f;
}

template <typename T>
__global__ void sketch_kernel(const T* __restrict__ O, float* __restrict__ Y, int N, int d, int k) {
  const int x = blockIdx.x, b = blockIdx.y, j = threadIdx.x;
  pdl_wait();
  pdl_trigger();
  if (j >= k) return;
  const T* row = O + ((size_t)b * N + x) * d;
  float acc = 0.f;
  for (int c = j; c < d; c += k) acc += hash_sign((uint32_t)c) * ld_f32(row + c);
  Y[((size_t)b * N + x) * k + j] = acc;
}

// The same sketch with 16-byte loads, for k a multiple of the vector length L (8 halves or 4
// floats): columns are taken in groups of L, group g goes to bucket group g mod (k / L), column
// i of the group to bucket i of that bucket group.  block (k / L, rows), grid (N / rows, B).
template <typename T, int L>
__global__ void sketch_vec_kernel(const T* __restrict__ O, float* __restrict__ Y, int N, int d, int k) {
  extern __shared__ float sgn[];  // [d]
  const int kg = blockDim.x, tx = threadIdx.x, ty = threadIdx.y;
  const int b = blockIdx.y, x = blockIdx.x * blockDim.y + ty;
  for (int c = ty * kg + tx; c < d; c += kg * blockDim.y) sgn[c] = hash_sign((uint32_t)c);
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  if (x >= N) return;
  const uint4* row = reinterpret_cast<const uint4*>(O + ((size_t)b * N + x) * d);
  const int ng = d / L;
  float acc[L];
#pragma unroll
  for (int i = 0; i < L; ++i) acc[i] = 0.f;
  int g = tx;
  for (; g + 7 * kg < ng; g += 8 * kg) {  // eight 16-byte loads in flight per thread
    uint4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) v[u] = __ldg(row + g + u * kg);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const T* e = reinterpret_cast<const T*>(&v[u]);
      const float* sg = sgn + (size_t)(g + u * kg) * L;
#pragma unroll
      for (int i = 0; i < L; ++i) acc[i] = fmaf(sg[i], (float)e[i], acc[i]);
    }
  }
  for (; g < ng; g += kg) {
    const uint4 v = __ldg(row + g);
    const T* e = reinterpret_cast<const T*>(&v);
    const float* sg = sgn + (size_t)g * L;
#pragma unroll
    for (int i = 0; i < L; ++i) acc[i] = fmaf(sg[i], (float)e[i], acc[i]);
  }
  float* out = Y + ((size_t)b * N + x) * k + tx * L;
#pragma unroll
  for (int i = 0; i < L; ++i) out[i] = acc[i];
}

// ==========================================================================================
// One-sided Jacobi eigen-solver for a symmetric positive semi-definite n x n matrix.
// One block (16 warps) per image.  W (column-major) starts as the matrix, J as the identity;
// each pair step rotates columns p, q of both so that the W columns become orthogonal.  At
// convergence  W = Z Theta  and  J = Z  (eigenvectors), column norms = eigenvalues.
// Pairs follow a round-robin tournament: n/2 disjoint pairs per round, one warp per pair,
// a block barrier between rounds.  R = elements of a column each lane keeps in registers.
// ==========================================================================================
constexpr int JACOBI_CL_THREADS = 640;

// AHEAD: the columns of J are loaded with those of W, not after the decision to rotate (out of L2 the
// second wait would double a round).
template <int R, bool AHEAD>
__device__ inline int jacobi_pair(float* __restrict__ W, float* __restrict__ J, int n, int p,
                                  int q, int lane, float tol, float floor2,
                                  float count_floor2) {
  float wp[R], wq[R];
  float a = 0.f, bq = 0.f, g = 0.f;
  float* Wp = W + (size_t)p * n;
  float* Wq = W + (size_t)q * n;
  float* Jp = J + (size_t)p * n;
  float* Jq = J + (size_t)q * n;
  float jpv[AHEAD ? R : 1], jqv[AHEAD ? R : 1];
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int r = lane + 32 * i;
    wp[i] = (r < n) ? Wp[r] : 0.f;
    wq[i] = (r < n) ? Wq[r] : 0.f;
    if constexpr (AHEAD) {
      jpv[i] = (r < n) ? Jp[r] : 0.f;
      jqv[i] = (r < n) ? Jq[r] : 0.f;
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    a = fmaf(wp[i], wp[i], a);
    bq = fmaf(wq[i], wq[i], bq);
    g = fmaf(wp[i], wq[i], g);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    bq += __shfl_xor_sync(0xffffffffu, bq, o);
    g += __shfl_xor_sync(0xffffffffu, g, o);
  }
  const float nn = sqrtf(a) * sqrtf(bq);
  if (!(fabsf(g) > tol * nn) || !(fmaxf(a, bq) > floor2)) return 0;
  const float zeta = (bq - a) / (2.0f * g);
  const float t = copysignf(1.0f, zeta) / (fabsf(zeta) + sqrtf(fmaf(zeta, zeta, 1.0f)));
  const float c = rsqrtf(fmaf(t, t, 1.0f));
  const float s = c * t;
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int r = lane + 32 * i;
    if (r < n) {
      Wp[r] = c * wp[i] - s * wq[i];
      Wq[r] = fmaf(s, wp[i], c * wq[i]);
    }
  }
#pragma unroll
  for (int i = 0; i < R; ++i) {
    const int r = lane + 32 * i;
    if (r < n) {
      const float jp = AHEAD ? jpv[AHEAD ? i : 0] : Jp[r], jq = AHEAD ? jqv[AHEAD ? i : 0] : Jq[r];
      Jp[r] = c * jp - s * jq;
      Jq[r] = fmaf(s, jp, c * jq);
    }
  }
  // a rotation between two columns that both lie under the rank cut-off does not delay
  // convergence: neither column enters Eq. 3-6
  return fmaxf(a, bq) > count_floor2 ? 1 : 0;
}

// CL == 1: a block per image with both matrices in shared memory.  Else a cluster of CL blocks, the
// matrices in L2, the pairs of a round dealt over all its warps: every pair's arithmetic is the same
// whoever does it.  What bounds it is a round's latency, m rounds to a sweep.
template <int R, int CL>
__global__ void __launch_bounds__(CL == 1 ? 1024 : JACOBI_CL_THREADS) jacobi_kernel(const float* __restrict__ Hin, int ldh,
                                                    float* __restrict__ Wg, float* __restrict__ ZTg,
                                                    float* __restrict__ theta, int n,
                                                    int max_sweeps, float tol,
                                                    int32_t* __restrict__ status, float floor_rel,
                                                    float count_rel) {
  extern __shared__ float sm[];
  __shared__ int s_rot;
  __shared__ float s_red[32];
  const int rank = CL == 1 ? 0 : (int)(blockIdx.x % CL), nt = blockDim.x, warps = nt / 32;
  const int b = blockIdx.x / CL, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int gwarp = warp * CL + rank, gwarps = warps * CL;   // (neighbouring pairs on different SMs)
  auto everyone = [] {
    if constexpr (CL == 1) {
      __syncthreads();
    } else {
      __syncwarp();
      asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
      asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    }
  };
  const size_t nn = (size_t)n * n;
  const float* Hb = Hin + b * (size_t)n * ldh;
  float* W = CL == 1 ? sm : Wg + b * nn;
  float* J = CL == 1 ? sm + nn : ZTg + b * nn;

  // W = (H + H^T) / 2 (column-major == row-major for a symmetric matrix), J = I
  float md = 0.f;
  for (size_t e = (size_t)rank * nt + tid; e < nn; e += (size_t)CL * nt) {
    const int p = (int)(e / n), i = (int)(e % n);
    const float v = 0.5f * (Hb[(size_t)p * ldh + i] + Hb[(size_t)i * ldh + p]);
    W[e] = v;
    J[e] = (p == i) ? 1.f : 0.f;
  }
  for (int i = tid; i < n; i += nt) md = fmaxf(md, fabsf(0.5f * (Hb[(size_t)i * ldh + i] + Hb[(size_t)i * ldh + i])));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
  if (lane == 0) s_red[warp] = md;
  if (tid == 0) s_rot = 0;
  __syncthreads();
  everyone();
  md = s_red[0];
  for (int w = 1; w < warps; ++w) md = fmaxf(md, s_red[w]);
  // column pairs whose norms (eigenvalue estimates) are BOTH below the floor are left alone:
  // they are rounding noise of the largest eigenvalue, or lie below the rank cut-off, and
  // rotating them against each other only slows convergence
  const float floor1 = floor_rel * md;
  const float floor2 = floor1 * floor1;
  const float count_floor2 = (count_rel * md) * (count_rel * md);

  const int ne = (n + 1) & ~1;  // even number of players; index n (if any) is a bye
  const int m = ne - 1;
  const int half = ne / 2;
  int sweep = 0;
  bool converged = false;
  for (; sweep < max_sweeps; ++sweep) {
    int rot = 0;
    for (int round = 0; round < m; ++round) {
      for (int slot = gwarp; slot < half; slot += gwarps) {
        int u, v;
        if (slot == 0) {
          u = round;
          v = m;
        } else {
          u = round + slot;
          if (u >= m) u -= m;
          v = round - slot;
          if (v < 0) v += m;
        }
        if (u >= n || v >= n) continue;
        const int p = min(u, v), q = max(u, v);
        rot += jacobi_pair<R, CL != 1 && R <= 18>(W, J, n, p, q, lane, tol, floor2, count_floor2);
      }
      everyone();
    }
    if (lane == 0 && rot) {
      if constexpr (CL == 1) {
        atomicAdd(&s_rot, rot);
      } else {
        for (int t = 0; t < CL; ++t) atomicAdd(cooperative_groups::this_cluster().map_shared_rank(&s_rot, t), rot);
      }
    }
    everyone();
    const int total = s_rot;
    everyone();
    if (tid == 0) s_rot = 0;   // (next added to after a sweep's barriers)
    if (total == 0) {
      converged = true;
      break;
    }
  }
  everyone();
  if (rank == 0 && tid == 0 && !converged) atomicMax(&status[b], (int)TC_ERR_NOT_CONVERGED);

  // eigenvalues = column norms of W;  eigenvectors = columns of J, written as ZT[p][i]
  for (int p = gwarp; p < n; p += gwarps) {
    float a = 0.f;
    for (int r = lane; r < n; r += 32) {
      const float v = W[(size_t)p * n + r];
      a = fmaf(v, v, a);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    if (lane == 0) theta[(size_t)b * n + p] = sqrtf(a);
  }
  if constexpr (CL == 1) {
    float* out = ZTg + b * nn;
    for (size_t e = tid; e < nn; e += nt) out[e] = J[e];
  }
}

// ------------------------------------------------------------------------------------------
// The same sweeps for 97 to 660 columns, with W in the shared memory of a cluster, and J apart:
//   jacobi_sweep_kernel   a sweep over W.  Block `rank` holds the columns of its pairs (slots), a warp
//                         per slot.  In the tournament the first player of slot s moves to slot s - 1,
//                         the second to s + 1, so a pair's columns are written to where the next
//                         round reads them, those at the edges into the neighbouring block, and a
//                         cluster barrier ends the round.  The rotations of the sweep go to `rot`.
//   jacobi_replay_kernel  the sweep's rotations on J, whose rows do not depend on one another: eight
//                         rows per block in shared memory.
// Every number comes from the same operations in the same order as in jacobi_kernel.
// What bounds it is a round: 83 KB of W through each SM's shared memory and back, the scalar chain of a
// rotation, the barrier.  Measured, 2 images of 576, 30 sweeps: 77 ms (both matrices out of L2) ->
// 47 ms, 3 of them the replays.
// ------------------------------------------------------------------------------------------
struct JacobiState {
  float md;        // largest diagonal entry of the matrix
  int sweeps;      // sweeps done
  int converged;
};

__global__ void __launch_bounds__(1024) jacobi_begin_kernel(const float* __restrict__ Hin, int ldh, float* __restrict__ Wg,
                                                           float* __restrict__ Jg, int n, JacobiState* __restrict__ state) {
  __shared__ float s_red[32];
  const size_t b = blockIdx.y, nn = (size_t)n * n;
  const float* Hb = Hin + b * (size_t)n * ldh;
  pdl_wait();
  for (size_t e = blockIdx.x * 1024 + threadIdx.x; e < nn; e += (size_t)gridDim.x * 1024) {
    const int p = (int)(e / n), i = (int)(e % n);
    Wg[b * nn + e] = 0.5f * (Hb[(size_t)p * ldh + i] + Hb[(size_t)i * ldh + p]);
    Jg[b * nn + e] = (p == i) ? 1.f : 0.f;
  }
  if (blockIdx.x != 0) return;
  float md = 0.f;
  for (int i = threadIdx.x; i < n; i += 1024) md = fmaxf(md, fabsf(0.5f * (Hb[(size_t)i * ldh + i] + Hb[(size_t)i * ldh + i])));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) md = fmaxf(md, __shfl_xor_sync(0xffffffffu, md, o));
  if ((threadIdx.x & 31) == 0) s_red[threadIdx.x >> 5] = md;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < 32; ++w) md = fmaxf(md, s_red[w]);
    state[b].md = md;
    state[b].sweeps = 0;
    state[b].converged = 0;
  }
}

template <int R, int CL>
__global__ void __launch_bounds__(672) jacobi_sweep_kernel(float* __restrict__ Wg, float2* __restrict__ rot, int n, float tol,
                                                         float floor_rel, float count_rel, JacobiState* __restrict__ state) {
  extern __shared__ float sm[];   // [2 buffers][warps][first, second][32 R]
  __shared__ int s_rot;
  constexpr int LEN = 32 * R;
  const int rank = (int)(blockIdx.x % CL), b = blockIdx.x / CL, warps = blockDim.x / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int half = (n + 1) / 2, m = 2 * half - 1;
  const int slot = rank * warps + warp;
  const bool live = slot < half;
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  pdl_wait();
  const JacobiState st = state[b];
  if (st.converged) return;   // (all blocks of the cluster alike)
  float* W = Wg + (size_t)b * n * n;
  const float floor1 = floor_rel * st.md, floor2 = floor1 * floor1;
  const float count_floor2 = (count_rel * st.md) * (count_rel * st.md);
  auto local = [&](int w, int which, int buf) { return sm + (size_t)((buf * warps + w) * 2 + which) * LEN; };
  // a column to where it plays next, in this block or in a neighbour
  auto put = [&](const float (&x)[R], int s, int which, int buf) {
    if (s / warps == rank) {
      float* d = local(s % warps, which, buf);
#pragma unroll
      for (int i = 0; i < R; ++i) d[lane + 32 * i] = x[i];
    } else {
      float* d = cl.map_shared_rank(local(s % warps, which, buf), s / warps);
#pragma unroll
      for (int i = 0; i < R; ++i) d[lane + 32 * i] = x[i];
    }
  };
  auto players = [&](int round, int& u, int& v) {
    u = round + slot;
    if (u >= m) u -= m;
    v = round - slot;
    if (v < 0) v += m;
    if (slot == 0) {
      u = round;
      v = m;
    }
  };
  if (threadIdx.x == 0) s_rot = 0;
  float wu[R], wv[R];
  if (live) {
    int u, v;
    players(0, u, v);
    float *du = local(warp, 0, 0), *dv = local(warp, 1, 0);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = lane + 32 * i;
      du[r] = r < n ? W[(size_t)u * n + r] : 0.f;
      dv[r] = r < n && v < n ? W[(size_t)v * n + r] : 0.f;
    }
  }
  cl.sync();
  int count = 0;
  float2* out = rot + (size_t)b * m * half + slot;
  for (int round = 0; round < m; ++round) {
    if (live) {
      int u, v;
      players(round, u, v);
      const float *su = local(warp, 0, round & 1), *sv = local(warp, 1, round & 1);
      float a = 0.f, bq = 0.f, g = 0.f;
      // p is the column of the lower number
      const bool swap = u > v;
#pragma unroll
      for (int i = 0; i < R; ++i) {
        wu[i] = su[lane + 32 * i];
        wv[i] = sv[lane + 32 * i];
      }
#pragma unroll
      for (int i = 0; i < R; ++i) {
        a = fmaf(wu[i], wu[i], a);
        bq = fmaf(wv[i], wv[i], bq);
        g = fmaf(wu[i], wv[i], g);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        bq += __shfl_xor_sync(0xffffffffu, bq, o);
        g += __shfl_xor_sync(0xffffffffu, g, o);
      }
      if (swap) {
        const float t = a;
        a = bq;
        bq = t;
      }
      const float nn = sqrtf(a) * sqrtf(bq);
      float2 cs = make_float2(1.f, 0.f);
      if (v < n && fabsf(g) > tol * nn && fmaxf(a, bq) > floor2) {
        const float zeta = (bq - a) / (2.0f * g);
        const float t = copysignf(1.0f, zeta) / (fabsf(zeta) + sqrtf(fmaf(zeta, zeta, 1.0f)));
        const float c = rsqrtf(fmaf(t, t, 1.0f));
        const float s = c * t;
        cs = make_float2(c, s);
#pragma unroll
        for (int i = 0; i < R; ++i) {
          const float wp = swap ? wv[i] : wu[i], wq = swap ? wu[i] : wv[i];
          const float np = c * wp - s * wq, nq = fmaf(s, wp, c * wq);
          wu[i] = swap ? nq : np;
          wv[i] = swap ? np : nq;
        }
        count += fmaxf(a, bq) > count_floor2 ? 1 : 0;
      }
      if (lane == 0) out[(size_t)round * half] = cs;
      // slot 0: the first player turns into the second of slot 1, the second stays; the last slot: the
      // second player turns into the first
      const int next = (round + 1) & 1;
      put(wu, slot == 0 ? 1 : slot - 1, slot == 0 ? 1 : 0, next);
      put(wv, slot == 0 || slot == half - 1 ? slot : slot + 1, slot == half - 1 ? 0 : 1, next);
    }
    cl.sync();
  }
  if (lane == 0 && count) atomicAdd(cl.map_shared_rank(&s_rot, 0), count);
  if (live) {   // after m rounds the players are where they began
    int u, v;
    players(0, u, v);
    const float *su = local(warp, 0, m & 1), *sv = local(warp, 1, m & 1);
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int r = lane + 32 * i;
      if (r < n) {
        W[(size_t)u * n + r] = su[r];
        if (v < n) W[(size_t)v * n + r] = sv[r];
      }
    }
  }
  cl.sync();
  if (rank == 0 && threadIdx.x == 0) {
    state[b].sweeps = st.sweeps + 1;
    state[b].converged = s_rot == 0;
  }
}

constexpr int REPLAY_ROWS = 8;
// grid (row groups, images), 512 threads: 64 pairs x 8 rows
__global__ void __launch_bounds__(512) jacobi_replay_kernel(float* __restrict__ Jg, const float2* __restrict__ rot, int n, int sweep,
                                                           const JacobiState* __restrict__ state) {
  extern __shared__ float js[];   // [n + 1][8]
  constexpr int SLOTS = 6;        // of a thread: up to 64 x 6 pairs
  const int b = blockIdx.y, r0 = blockIdx.x * REPLAY_ROWS, row = threadIdx.x & 7, first = threadIdx.x >> 3;
  const int half = (n + 1) / 2, m = 2 * half - 1;
  pdl_wait();
  if (state[b].sweeps <= sweep) return;   // (the sweeps had ended before)
  float* J = Jg + (size_t)b * n * n;
  const bool there = r0 + row < n;
  for (int c = first; c < n; c += 64) js[c * 8 + row] = there ? J[(size_t)c * n + r0 + row] : 0.f;
  const float2* list = rot + (size_t)b * m * half;
  float2 cs[SLOTS];
#pragma unroll
  for (int k = 0; k < SLOTS; ++k) cs[k] = first + 64 * k < half ? __ldg(list + first + 64 * k) : make_float2(1.f, 0.f);
  __syncthreads();
  for (int round = 0; round < m; ++round) {
    float2 now[SLOTS];
#pragma unroll
    for (int k = 0; k < SLOTS; ++k) {
      now[k] = cs[k];
      if (round + 1 < m && first + 64 * k < half) cs[k] = __ldg(list + (size_t)(round + 1) * half + first + 64 * k);
    }
#pragma unroll
    for (int k = 0; k < SLOTS; ++k) {
      const int slot = first + 64 * k;
      if (slot >= half || now[k].y == 0.f) continue;
      int u = round + slot, v = round - slot;
      if (u >= m) u -= m;
      if (v < 0) v += m;
      if (slot == 0) {
        u = round;
        v = m;
      }
      const int p = min(u, v), q = max(u, v);
      const float c = now[k].x, s = now[k].y, jp = js[p * 8 + row], jq = js[q * 8 + row];
      js[p * 8 + row] = c * jp - s * jq;
      js[q * 8 + row] = fmaf(s, jp, c * jq);
    }
    __syncthreads();
  }
  if (there)
    for (int c = first; c < n; c += 64) J[(size_t)c * n + r0 + row] = js[c * 8 + row];
}

// eigenvalues = column norms of W; a warp per column
__global__ void __launch_bounds__(256) jacobi_end_kernel(const float* __restrict__ Wg, float* __restrict__ theta, int n,
                                                        const JacobiState* __restrict__ state, int32_t* __restrict__ status) {
  const int b = blockIdx.y, p = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0 && !state[b].converged) atomicMax(&status[b], (int)TC_ERR_NOT_CONVERGED);
  if (p >= n) return;
  float a = 0.f;
  for (int r = lane; r < n; r += 32) {
    const float v = Wg[(size_t)b * n * n + (size_t)p * n + r];
    a = fmaf(v, v, a);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
  if (lane == 0) theta[(size_t)b * n + p] = sqrtf(a);
}

typedef void (*jacobi_fn)(const float*, int, float*, float*, float*, int, int, float, int32_t*, float, float);

// (two matrices of up to 167 columns fit in shared memory)
static jacobi_fn pick_jacobi(int n, bool use_smem, int cl) {
  const int r = (n + 31) / 32;
  if (use_smem) {
    if (r <= 1) return jacobi_kernel<1, 1>;
    if (r <= 2) return jacobi_kernel<2, 1>;
    if (r <= 3) return jacobi_kernel<3, 1>;
    if (r <= 4) return jacobi_kernel<4, 1>;
    if (r <= 5) return jacobi_kernel<5, 1>;
    if (r <= 6) return jacobi_kernel<6, 1>;
    return nullptr;
  }
  if (r <= 6) return cl == 8 ? jacobi_kernel<6, 8> : jacobi_kernel<6, 16>;
  if (r <= 8) return cl == 8 ? jacobi_kernel<8, 8> : jacobi_kernel<8, 16>;
  if (r <= 10) return cl == 8 ? jacobi_kernel<10, 8> : jacobi_kernel<10, 16>;
  if (r <= 14) return jacobi_kernel<14, 16>;
  if (r <= 18) return jacobi_kernel<18, 16>;
  if (r <= 24) return jacobi_kernel<24, 16>;
  if (r <= 32) return jacobi_kernel<32, 16>;
  return nullptr;
}

constexpr size_t SMEM_LIMIT = 220 * 1024;  // leaves room for the static shared variables

typedef void (*sweep_fn)(float*, float2*, int, float, float, float, JacobiState*);
struct sweep_pick {
  sweep_fn fn;
  int len;   // floats of a column in shared memory
};
static sweep_pick pick_sweep(int n) {
  if (n <= 128) return {jacobi_sweep_kernel<4, 8>, 128};
  if (n <= 192) return {jacobi_sweep_kernel<6, 8>, 192};
  if (n <= 256) return {jacobi_sweep_kernel<8, 8>, 256};
  if (n <= 320) return {jacobi_sweep_kernel<10, 8>, 320};
  if (n <= 448) return {jacobi_sweep_kernel<14, 16>, 448};
  if (n <= 576) return {jacobi_sweep_kernel<18, 16>, 576};
  return {jacobi_sweep_kernel<21, 16>, 672};
}
// Bytes per image that the sweeps over a cluster's shared memory want (none: another size's kernel)
size_t jacobi_rot_bytes(int n) {
  if (n < 97 || n > 672) return 0;
  const size_t half = (n + 1) / 2;
  return ((2 * half - 1) * half * sizeof(float2) + sizeof(JacobiState) + 15) / 16 * 16;
}

static tc_status launch_jacobi(const float* H, int ldh, float* W, float* ZT, float* theta, int n, int batch,
                          int max_sweeps, float rank_tol, float2* rot, JacobiState* state, int32_t* status,
                          cudaStream_t st) {
  Scope scope_(KC_JACOBI, st);
  // off-diagonal threshold a little above the rounding noise of a length-n float32 dot product
  const float tol = fmaxf(1e-6f, 2.5f * sqrtf((float)n) * 1.1920929e-7f);
  // Eigenvalue floors, relative to the largest diagonal entry.  Column pairs that are both
  // under the float32 rounding level of that entry are never rotated; rotations between two
  // columns that are both under the eigenvalue rank_tol cuts at are done but do not count
  // towards "this sweep still rotated".
  const float floor_rel = 1e-6f;
  const float count_rel = fmaxf(floor_rel, rank_tol * rank_tol);
  const int pairs = (n + 1) / 2;
  // (a launch or two per sweep, so not for bounds on the sweeps that are none)
  if (rot != nullptr && max_sweeps <= 100) {
    const int cl = n <= 320 ? 8 : 16, warps = (pairs + cl - 1) / cl;
    const sweep_pick pk = pick_sweep(n);
    const size_t smem = (size_t)4 * warps * pk.len * sizeof(float);
    if (cudaFuncSetAttribute((const void*)pk.fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
        (cl > 8 && cudaFuncSetAttribute((const void*)pk.fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess))
      return TC_ERR_CUDA;
    launch_pdl(jacobi_begin_kernel, dim3(16, batch), dim3(1024), 0, st, 0, H, ldh, W, ZT, n, state);
    note_launch();
    for (int sweep = 0; sweep < max_sweeps; ++sweep) {
      if (launch_pdl(pk.fn, dim3((unsigned)(batch * cl)), dim3((unsigned)(warps * 32)), smem, st, cl, W, rot, n, tol, floor_rel,
                     count_rel, state) != cudaSuccess)
        return TC_ERR_CUDA;
      note_launch();
      launch_pdl(jacobi_replay_kernel, dim3((unsigned)((n + REPLAY_ROWS - 1) / REPLAY_ROWS), batch), dim3(512),
                 (size_t)n * REPLAY_ROWS * sizeof(float), st, 0, ZT, (const float2*)rot, n, sweep, (const JacobiState*)state);
      note_launch();
    }
    launch_pdl(jacobi_end_kernel, dim3((n + 7) / 8, batch), dim3(256), 0, st, 0, (const float*)W, theta, n,
               (const JacobiState*)state, status);
    note_launch();
    return TC_OK;
  }
  const size_t need = 2 * (size_t)n * n * sizeof(float);
  const bool use_smem = need <= SMEM_LIMIT;
  const size_t smem = use_smem ? need : 0;
  // up to 20 warps a block take a round's n / 2 pairs, one each up to 640 columns
  const int cl = use_smem ? 1 : pairs <= 160 ? 8 : 16;
  const int warps = use_smem ? 32 : min(JACOBI_CL_THREADS / 32, (pairs + cl - 1) / cl);
  jacobi_fn fn = pick_jacobi(n, use_smem, cl);
  if (fn == nullptr) return TC_ERR_UNSUPPORTED;
  if (use_smem && cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return TC_ERR_CUDA;
  if (cl > 8 && cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
    return TC_ERR_CUDA;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(batch * cl));
  cfg.blockDim = dim3((unsigned)(warps * 32));
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)cl;
  at.val.clusterDim.y = at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = cl > 1 ? 1 : 0;
  if (cudaLaunchKernelEx(&cfg, fn, H, ldh, W, ZT, theta, n, max_sweeps, tol, status, floor_rel, count_rel) != cudaSuccess)
    return TC_ERR_CUDA;
  note_launch();
  return TC_OK;
}

// Which solver decomposes an n x n matrix.  The vectors of the full solve come from Jacobi sweeps: they
// are orthogonal whatever the spectrum, and img_status says of every image whether its sweeps ended.
// So does a subspace wider than 224 with rank_tol under 1e-3: inverse iteration does not orthogonalise
// eigenvectors against each other, which is fine while the wanted eigenvalues (rank_tol^2 theta_max and
// up) stand clear of the float32 rounding level of the largest, about 1e-6 of it.  Eigenvalues alone
// need no such care.
static bool use_tridiag(int n, bool full, bool values_only, float rank_tol) {
  return eig_tridiag_supported(n) && (values_only || (!full && (rank_tol >= 1e-3f || n <= 224)));
}

// ==========================================================================================
// out [C][ldo] = in [R][C]^T per image, 32 x 32 tiles through shared memory.
// grid (C tiles, R tiles, batch), block (32, 8).
// ==========================================================================================
__global__ void __launch_bounds__(256) transpose_kernel(const float* __restrict__ in, int R, int C,
                                                       float* __restrict__ out, int ldo) {
  __shared__ float t[32][33];
  const int b = blockIdx.z, r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  const int tx = threadIdx.x, ty = threadIdx.y;
  pdl_wait();
  pdl_trigger();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int r = r0 + ty + 8 * i, c = c0 + tx;
    t[ty + 8 * i][tx] = (r < R && c < C) ? in[((size_t)b * R + r) * C + c] : 0.f;
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int c = c0 + ty + 8 * i, r = r0 + tx;
    if (r < R && c < C) out[((size_t)b * C + c) * ldo + r] = t[tx][ty + 8 * i];
  }
}

static void launch_transpose(const float* in, int R, int C, int batch, float* out, int ldo, cudaStream_t st, int cls) {
  Scope scope_(cls, st);
  dim3 grid((C + 31) / 32, (R + 31) / 32, batch), block(32, 8);
  { launch_pdl(transpose_kernel, grid, block, 0, st, 0, in, R, C, out, ldo); note_launch(); }
}

// ==========================================================================================
// Eq. 3-6 and the outputs that go with it.  One block per image.
//   theta [k]   eigenvalues of G (unsorted);  sigma_i = sqrt(theta_i)
//   PT [k][N]   PT[p][x] = component of token x along eigenvector p (u_xp)
//   C(x) = sum over p with sigma_p > rank_tol * sigma_max of |u_xp| sigma_p
// ==========================================================================================
__global__ void __launch_bounds__(256) ics_kernel(const float* __restrict__ theta,
                                                 const float* __restrict__ PT, int ldp, float* __restrict__ C,
                                                 float* __restrict__ sigma_sorted,
                                                 int32_t* __restrict__ rank_out,
                                                 int32_t* __restrict__ status, int N, int k, int q,
                                                 float rank_tol, int cap,
                                                 const float* __restrict__ G, int ldg,
                                                 const float* __restrict__ S, float* __restrict__ E, float lambda) {
  // k: vectors in PT (rows ldp floats apart); cap: bound on the rank that the caller gave (0: none):
  // singular values beyond it are reported as zero, and a rank that comes within eight of it as
  // TC_ERR_RANK_CAP.  G (subspace solve only): the Gram matrix, for the energy check below.
  // grid (token chunks of 64, images): every block ranks the k singular values again (k^2
  // comparisons, cheap) and sums Eq. 3-6 for its own tokens, four threads to a token (each a
  // quarter of the range of p, its loads in flight together); chunk 0 writes sigma and the rank.
  extern __shared__ float sig[];  // [k] sigma, then [k] weights (sigma or 0)
  float* wgt = sig + k;
  __shared__ float s_red[8];
  __shared__ int s_cnt[8];
  __shared__ float s_part[4][64];
  const int b = blockIdx.y, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool writer = blockIdx.x == 0;
  pdl_wait();
  pdl_trigger();
  float mx = 0.f;
  for (int p = tid; p < k; p += 256) {
    const float s = sqrtf(fmaxf(theta[(size_t)b * k + p], 0.f));
    sig[p] = s;
    mx = fmaxf(mx, s);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (lane == 0) s_red[warp] = mx;
  __syncthreads();
  float smax = s_red[0];
#pragma unroll
  for (int w = 1; w < 8; ++w) smax = fmaxf(smax, s_red[w]);
  const float cut = rank_tol * smax;
  // O has at most q = min(N, d) non-zero singular values: only the q largest eigenvalues of G
  // can be one, whatever rounding left in the others.
  int cnt = 0;
  for (int p = tid; p < k; p += 256) {
    const float s = sig[p];
    int pos = 0;
    for (int o = 0; o < k; ++o) pos += (sig[o] > s) || (sig[o] == s && o < p);
    const bool on = (s > cut) && (pos < q);
    wgt[p] = on ? s : 0.f;
    cnt += on;
    if (writer && sigma_sorted && pos < q) sigma_sorted[(size_t)b * q + pos] = (cap == 0 || pos < cap) ? s : 0.f;
  }
  if (writer && sigma_sorted)
    for (int p = k + tid; p < q; p += 256) sigma_sorted[(size_t)b * q + p] = 0.f;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) cnt += __shfl_xor_sync(0xffffffffu, cnt, o);
  if (lane == 0) s_cnt[warp] = cnt;
  __syncthreads();
  if (writer && tid == 0) {
    int r = 0;
    for (int w = 0; w < 8; ++w) r += s_cnt[w];
    if (rank_out) rank_out[b] = r;
    if (cap > 0 && r > cap - 8) atomicMax(&status[b], (int)TC_ERR_RANK_CAP);
  }
  if (writer && G != nullptr && warp == 0) {
    // What the subspace did not capture: trace(G) - sum(theta) is the energy of O outside it.
    // If the directions left out were all under the rank cut-off, that is at most
    // (q - k) (rank_tol sigma_1)^2; more means a direction above the cut-off was missed (a
    // rank above the hint that the count above could not see), and Eq. 3-6 would be truncated.
    float tr = 0.f, st = 0.f;
    const float* Gb = G + (size_t)b * N * ldg;
    for (int x0 = 0; x0 < N; x0 += 256) {  // eight loads in flight
      float dgl[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int x = x0 + u * 32 + lane;
        dgl[u] = (x < N) ? Gb[(size_t)x * ldg + x] : 0.f;
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) tr += dgl[u];
    }
    for (int p = lane; p < k; p += 32) st += sig[p] * sig[p];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      tr += __shfl_xor_sync(0xffffffffu, tr, o);
      st += __shfl_xor_sync(0xffffffffu, st, o);
    }
    const float allow = (float)max(q - k, 0) * cut * cut + 1e-5f * tr;
    if (lane == 0 && tr - st > allow) atomicMax(&status[b], (int)TC_ERR_RANK_CAP);
  }
  const float* PTb = PT + (size_t)b * k * ldp;
  const int xl = tid & 63, part = tid >> 6;
  const int x = blockIdx.x * 64 + xl;
  const int per = (k + 3) >> 2;
  const int p_lo = part * per, p_hi = min(k, p_lo + per);
  float acc = 0.f;
  if (x < N) {
    // terms of a quarter in the order p = p_lo, p_lo + 1, ...; twelve loads in flight
    int p = p_lo;
    for (; p + 11 < p_hi; p += 12) {
      float v[12];
#pragma unroll
      for (int u = 0; u < 12; ++u) v[u] = PTb[(size_t)(p + u) * ldp + x];
#pragma unroll
      for (int u = 0; u < 12; ++u) acc = fmaf(fabsf(v[u]), wgt[p + u], acc);
    }
    for (; p < p_hi; ++p) acc = fmaf(fabsf(PTb[(size_t)p * ldp + x]), wgt[p], acc);
  }
  s_part[part][xl] = acc;
  __syncthreads();
  if (part == 0 && x < N) {
    const float c = (s_part[0][xl] + s_part[1][xl]) + (s_part[2][xl] + s_part[3][xl]);
    C[(size_t)b * N + x] = c;
    if (E != nullptr) E[(size_t)b * N + x] = (1.f - lambda) * c + lambda * S[(size_t)b * N + x];   // Eq. 3-8
  }
}

__global__ void fill_i32_kernel(int32_t* p, int n, int v) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

void fill_i32(int32_t* p, int n, int v, cudaStream_t st) {
  Scope scope_(KC_FILL, st);
  { fill_i32_kernel<<<(n + 255) / 256, 256, 0, st>>>(p, n, v); note_launch(); }
}

// ==========================================================================================
// The whole of Eq. 3-5 / 3-6 for a batch, given G in the workspace.
// ==========================================================================================
tc_status launch_ics(const Dims& D, const Plan& P, char* ws, int b0, const void* O, const ScoreIo& io,
                     cudaStream_t st) {
  int32_t* img_status = io.status;
  // D.B images starting at image b0 of the workspace arrays; O and the outputs already point at
  // image b0.
  const int B = D.B, N = D.N, k = D.k;
  const int q = min(D.N, D.d);
  const int ldn = D.ldn, cap = (D.cap > 0 && D.cap < N) ? D.cap : 0;
  const size_t sG = (size_t)N * ldn, sY = (size_t)N * k, sT = (size_t)k * ldn, sK = (size_t)k * k;
  float* G = (float*)(ws + P.G) + b0 * sG;
  float* W = (float*)(ws + P.W + b0 * jacobi_work_bytes(k));
  float* ZT = (float*)(ws + P.ZT) + b0 * sK;
  float* theta = (float*)(ws + P.sigma) + (size_t)b0 * k;
  auto scores = [&](const float* PT, int ldp, const float* Gc) {
    if (io.s_ready) cudaStreamWaitEvent(st, io.s_ready, 0);
    Scope scope_(KC_ICS, st);
    { launch_pdl(ics_kernel, dim3((N + 63) / 64, B), dim3(256), 2 * (size_t)k * sizeof(float), st, 0,
          theta, PT, ldp, io.C, io.sigma, io.rank, img_status, N, k, q, D.rank_tol, cap, Gc, ldn, io.S,
          D.score_norm == TC_NORM_NONE ? io.E : nullptr, D.lambda); note_launch(); }
  };

  if (D.full) {
    if (io.g_ready) cudaStreamWaitEvent(st, io.g_ready, 0);
    if (use_tridiag(N, cap == 0, io.values_only, D.rank_tol)) {   // (a bound that left no subspace is not the full solve)
      tc_status e = launch_eig_tridiag(G, sG, ldn, N, B, D.rank_tol, theta, ZT, sK, N, W, img_status, st);
      if (e != TC_OK) return e;
    } else {
      const size_t rb = jacobi_rot_bytes(N), half = (N + 1) / 2;
      // (the batch's lists, then its states; groups have theirs apart)
      float2* rot = rb ? (float2*)(ws + P.rot + b0 * rb) : nullptr;
      JacobiState* jst = rb ? (JacobiState*)(rot + (size_t)B * (2 * half - 1) * half) : nullptr;
      const tc_status e = launch_jacobi(G, ldn, W, ZT, theta, N, B, D.max_sweeps, D.rank_tol, rot, jst, img_status, st);
      if (e != TC_OK) return e;
    }
    scores(ZT, N, nullptr);
    return TC_OK;
  }
  auto sketch_into = [&](float* Y0) {
    Scope scope_(KC_SKETCH, st);
    const int L = 16 / D.esz;
    if (k % L == 0 && k / L <= 256 && (size_t)D.d * sizeof(float) <= 48 * 1024) {
      const int kg = k / L;
      const int rows = max(1, 256 / kg);
      dim3 block(kg, rows), grid((N + rows - 1) / rows, B);
      const size_t smem = (size_t)D.d * sizeof(float);
      TC_WITH_STORAGE_TYPE(D,
        launch_pdl(sketch_vec_kernel<T, 16 / sizeof(T)>, grid, block, smem, st, 0, (const T*)O, Y0, N, D.d, k);
        note_launch(););
    } else {
      dim3 grid(N, B);
      const int threads = (k + 31) / 32 * 32;
      TC_WITH_STORAGE_TYPE(D,
        launch_pdl(sketch_kernel<T>, grid, dim3(threads), 0, st, 0, (const T*)O, Y0, N, D.d, k);
        note_launch(););
    }
  };
  if (D.tcp) {
    // ---- the products on the tensor cores (gemm_f32x3.cu: C = A B^T, both operands with the
    //      contraction index contiguous).  Every tall panel is therefore kept twice, row-major
    //      [N][k] and transposed [k][ldn]; a product writes whichever forms its consumers read.
    float* Ar = (float*)(ws + P.PA) + b0 * sY;
    float* At = (float*)(ws + P.PA) + P.panel_T_off / sizeof(float) + b0 * sT;
    float* Br = (float*)(ws + P.PB) + b0 * sY;
    float* Bt = (float*)(ws + P.PB) + P.panel_T_off / sizeof(float) + b0 * sT;
    float* Sk = (float*)(ws + P.Sk) + b0 * sK;
    float* Hk = (float*)(ws + P.Hk) + b0 * sK;
    float* Rinv = (float*)(ws + P.Rinv) + b0 * sK;
    float* Pk = (float*)(ws + P.Pk) + (size_t)b0 * chol_panel_floats(k);
    float* Es = (float*)(ws + P.Es + b0 * jacobi_work_bytes(k));
    tc_status err = TC_OK;
    const auto rows = [&](const float* p) { return F32x3Operand{p, k, sY}; };    // [N][k]
    const auto cols = [&](const float* p) { return F32x3Operand{p, ldn, sT}; };  // [k][N]
    const auto small = [&](const float* p) { return F32x3Operand{p, k, sK}; };   // [k][k]
    const F32x3Operand gram{G, ldn, sG};
    auto mm = [&](const F32x3Operand& A_, const F32x3Operand& B_, int M_, int K_, const F32x3Result& R, int cls) {
      if (err == TC_OK) err = launch_gemm_f32x3(A_, B_, M_, k, K_, B, D.call_B, R, img_status, st, cls);
    };
    const auto tall = [&](float* c, float* ct) { return F32x3Result{c, k, sY, ct, ldn, sT}; };
    const auto square = [&](float* c) { return F32x3Result{c, k, sK, nullptr, 0, 0}; };
    // one Cholesky-QR pass  dst = src R^{-1}  with  R^T R = src^T src + shift
    auto pass = [&](const float* srcR, const float* srcT, float* dstR, float* dstT, float shift_rel) {
      mm(cols(srcT), cols(srcT), k, N, square(Sk), KC_GEMM_TN);
      if (err == TC_OK) err = launch_chol_inv(Sk, Rinv, Pk, k, B, D.call_B, shift_rel, img_status, st);
      mm(rows(srcR), small(Rinv), N, k, tall(dstR, dstT), KC_GEMM);   // (Y R^{-1})[x][c] = Y[x][:] . R^{-T}[c][:]
    };
    // 1. sketch of the column space of O, in both forms
    sketch_into(Ar);
    launch_transpose(Ar, N, k, B, At, ldn, st, KC_SKETCH);
    // 2. a well-conditioned basis Q0 of the sketch (only its transposed form is read)
    pass(Ar, At, nullptr, Bt, 1e-6f);
    // 3. Y1 = G Q0, then two passes: the first (shifted) brings the condition number from ~1e7
    //    down to ~1e3, the second leaves a basis whose departure from orthonormality lies in the
    //    directions under the rank cut-off; the Ritz values above it are unaffected.  The widths of
    //    the package's configurations, chosen close to the rank, stop there; others, which may hold
    //    many directions under the cut-off, take a third so that the values there are right as well.
    if (io.g_ready) cudaStreamWaitEvent(st, io.g_ready, 0);
    mm(gram, cols(Bt), N, N, tall(Ar, At), KC_GEMM_GQ);
    pass(Ar, At, Br, Bt, 1e-6f);
    if (!((k == 128 || k == 144 || k == 160 || k == 192) && k == D.cap && (N & 3) == 0)) {
      pass(Br, Bt, Ar, At, 1e-6f);
      std::swap(Ar, Br);
      std::swap(At, Bt);
    }
    pass(Br, Bt, Ar, At, 1e-7f);  // Q1 in set A
    // 4. Rayleigh-Ritz:  T = G Q1 (kept transposed),  H = Q1^T T
    mm(gram, cols(At), N, N, tall(nullptr, Bt), KC_GEMM_GQ);
    mm(cols(At), cols(Bt), k, N, square(Hk), KC_GEMM_TN);
    float* Zk = Sk;  // the k x k matrix of the passes is free now
    if (err != TC_OK) return err;
    err = launch_eig_tridiag(Hk, sK, k, k, B, D.rank_tol, theta, Zk, sK, k, Es, img_status, st);
    // 5. eigenvectors of G in the subspace, U = Q1 Z, written transposed:
    //    PT[p][x] = sum_i ZT[p][i] Q1[x][i]
    float* PT = Bt;
    mm(rows(Ar), small(Zk), N, k, tall(nullptr, PT), KC_GEMM);
    if (err != TC_OK) return err;
    scores(PT, ldn, G);
    return TC_OK;
  }
  float* Y0 = (float*)(ws + P.Y0) + b0 * sY;
  float* Y1 = (float*)(ws + P.Y1) + b0 * sY;
  float* Y2 = (float*)(ws + P.Y2) + b0 * sY;
  float* Sm = (float*)(ws + P.Sm) + b0 * sK;
  float* Rinv = (float*)(ws + P.Rinv) + b0 * sK;
  float* Hm = (float*)(ws + P.Hm) + b0 * sK;

  // 1. sketch of the column space of O
  sketch_into(Y0);
  // one Cholesky-QR pass: dst = src R^{-1},  R^T R = src^T src (+ shift)
  auto cholqr_pass = [&](const float* src, float* dst, float shift_rel) {
    gemm<float, float, true, false>(src, src, Sm, k, k, N, k, k, k, sY, sY, sK, B, st, KC_GEMM_TN, GEMM_SYM);
    launch_chol_inv_f32(Sm, Rinv, W, k, B, shift_rel, img_status, st);
    gemm<float, float, false, true>(src, Rinv, dst, N, k, k, k, k, k, sY, sK, sY, B, st, KC_GEMM, GEMM_B_UPPER);
  };
  const float kShift = 1e-6f;
  // 2. a well-conditioned (not orthonormal) basis Q0 of the sketch: one shifted pass takes the
  //    condition number from ~1e3 to a few units, which is all the next product needs
  cholqr_pass(Y0, Y1, kShift);
  { float* t = Y0; Y0 = Y1; Y1 = t; }  // Q0 in Y0
  // 3. one multiplication by G sharpens the subspace:  Y1 = G Q0, then orthonormalise
  if (io.g_ready) cudaStreamWaitEvent(st, io.g_ready, 0);
  gemm<float, float, false, false>(G, Y0, Y1, N, k, N, ldn, k, k, sG, sY, sY, B, st, KC_GEMM_GQ);
  cholqr_pass(Y1, Y2, kShift);
  cholqr_pass(Y2, Y1, kShift);
  cholqr_pass(Y1, Y2, 0.f);  // Q1 in Y2
  // 4. Rayleigh-Ritz:  H = Q1^T G Q1
  gemm<float, float, false, false>(G, Y2, Y1, N, k, N, ldn, k, k, sG, sY, sY, B, st, KC_GEMM_GQ);   // T = G Q1
  gemm<float, float, true, false>(Y2, Y1, Hm, k, k, N, k, k, k, sY, sY, sK, B, st, KC_GEMM_TN);   // H = Q1^T T
  if (use_tridiag(k, false, io.values_only, D.rank_tol)) {
    tc_status e = launch_eig_tridiag(Hm, sK, k, k, B, D.rank_tol, theta, ZT, sK, k, W, img_status, st);
    if (e != TC_OK) return e;
  } else {
    const tc_status e = launch_jacobi(Hm, k, W, ZT, theta, k, B, D.max_sweeps, D.rank_tol, nullptr, nullptr, img_status, st);
    if (e != TC_OK) return e;
  }
  // 5. eigenvectors of G restricted to the subspace:  PT[p][x] = sum_i ZT[p][i] Q1[x][i]
  gemm<float, float, false, true>(ZT, Y2, Y0, k, N, k, k, k, N, sK, sY, sY, B, st);
  scores(Y0, N, G);
  return TC_OK;
}

}  // namespace tc
