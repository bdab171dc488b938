// Internal declarations shared by the translation units of libtokencarve.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stddef.h>
#include <stdint.h>

#include "pdl.cuh"
#include "tokencarve.h"

#include <atomic>

namespace tc {

// test hook (tc_test_fail_tensor_maps): while set, every tensor-map encode is refused, which is
// how a launcher's refusal after the group streams were forked is exercised without a GPU fault
inline std::atomic<int> g_refuse_encode{0};


// Counts of Sec. 3.3.1 / Eq. 3-9 plus everything the launchers derive from tc_params.
struct Dims {
  int B, N, d, H, dh, T;
  int call_B;     // images of the call (B: of the group at hand)
  int keep, M, P, nA, nB;
  int cap;        // rank_cap as given (0 or >= N: none)
  int k;          // dimension of the decomposition: N for the full solve, else rank_cap, on the tensor
                  // cores rounded up to a multiple of 16
  bool full;      // the Gram matrix itself is decomposed
  bool tcp;       // the subspace solve runs its products on the tensor cores
  int ldn;        // pitch in floats of G's rows and of transposed panels: N rounded up to a multiple of 4
  int esz;        // bytes per element of O, A, X, K, V
  bool f16;       // float16 storage
  bool bf16;      // bfloat16 storage (neither: float32)
  int sim_src;    // Eq. 3-10 features: 0 rows of O (the paper), 1 rows of X, 2 head-mean of K
  bool wmerge;    // merge with the IPGS scores as weights instead of the plain mean
  int chunks;     // row chunks of the attention column-mean
  int max_sweeps;
  float lambda, rank_tol;
  int score_norm;
};

tc_status make_dims(const tc_params* p, Dims* out);

// Offsets (bytes) of every scratch array inside the caller's workspace.
struct Plan {
  size_t s_part;   // [B, chunks, N] f32   partial column sums of A
  size_t S, C, E;  // [B, N] f32 each
  size_t sigma;    // [B, k] f32 (unsorted eigenvalue norms theta)
  size_t G;        // [B, N, ldn] f32
  size_t Y0, Y1, Y2;  // [B, N, k] f32 each (subspace solve only)
  size_t Sm, Rinv, Hm;  // [B, k, k] f32 each (subspace solve only)
  size_t W, ZT;    // [B] work array of the eigen-solver; [B, k, k] f32 eigenvectors
  size_t rot;      // [B] rotations of a Jacobi sweep (full solve)
  size_t setA, setB, best_val, best_dst, msrc, mdst, kept;  // int32 / f32 lists
  size_t rank;     // [B] int32
  size_t flags;    // [B] int32 device status scratch
  size_t Kmean;    // [B, N, dh] f32: head-mean keys (sim_src == 2 only)
  // tensor-core subspace solve (Dims::tcp)
  size_t PA, PB;   // two sets of tall panels: [B][N][k] row-major and, panel_T_off bytes
                   // further on, [B][k][ldn] transposed
  size_t panel_T_off;
  size_t Sk, Hk;   // [B][k][k] f32: Y^T Y (later the eigenvectors) and the projected matrix
  size_t Es;       // [B] scratch of the tridiagonal solver
  size_t Pk;       // [B][chol_panel_floats(k)] f32: panel of the blocked Cholesky factorisation
  size_t total;
};

Plan make_plan(const Dims& D);

// value rounded to the nearest TF32 (low 13 mantissa bits zero)
__device__ __forceinline__ float tf32_round(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return __uint_as_float(r);
}

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// Runs `...` with T bound to the storage type of the call.
#define TC_WITH_STORAGE_TYPE(D, ...)      \
  do {                                    \
    if ((D).bf16) {                       \
      using T = __nv_bfloat16;            \
      __VA_ARGS__                         \
    } else if ((D).f16) {                 \
      using T = __half;                   \
      __VA_ARGS__                         \
    } else {                              \
      using T = float;                    \
      __VA_ARGS__                         \
    }                                     \
  } while (0)

// Running count of kernels this library has launched (host side, all streams).
void note_launch(int n = 1);

// Kernel classes for the optional event profile (tc_profile_begin / tc_profile_end).
enum KernelClass {
  KC_FILL = 0, KC_ATTN, KC_GRAM, KC_SKETCH, KC_GEMM, KC_CHOL, KC_JACOBI, KC_ICS, KC_COMBINE,
  KC_PRUNE, KC_MATCH, KC_MSEL, KC_COMPACT, KC_GEMM_GQ, KC_GEMM_TN, KC_COUNT
};
// While a profile is open, brackets the launches made in its lifetime with two CUDA events
// on `st`; otherwise does nothing.
struct Scope {
  int slot;
  cudaStream_t st;
  Scope(int cls, cudaStream_t st);
  ~Scope();
};

// ---- launchers (each only enqueues on `st`) ---------------------------------------------
// Eq. 3-7: column means of A over heads and query rows.
void launch_attn_colsum(const Dims& D, const void* A, float* s_part, cudaStream_t st);
// ... and S from them.
void launch_attn_finish(const Dims& D, const float* s_part, float* S, cudaStream_t st);
// Eq. 3-8 on normalised terms (score_norm == TC_NORM_SUM1).
void launch_combine(const Dims& D, const float* C, const float* S, float* E, cudaStream_t st);
// Stage I prune + Eq. 3-9 split.
void launch_prune(const Dims& D, const float* E, int32_t* setA, int32_t* setB, cudaStream_t st);
// Eq. 3-10 best match per Set-B token, from the Gram matrix.
// (status [B]: receives TC_ERR_INVALID_ARG for an image whose lists hold a token number outside
// [0, N); such an entry is skipped, never used as an address.  The same for the launchers below.)
void launch_match_gram(const Dims& D, const float* G, int ldg, const int32_t* setA, const int32_t* setB,
                       float* best_val, int32_t* best_dst, int32_t* status, cudaStream_t st);
// top-M of the best similarities, merge lists, kept list.
void launch_merge_select(const Dims& D, const int32_t* setA, const int32_t* setB,
                         const float* best_val, const int32_t* best_dst, int32_t* msrc,
                         int32_t* mdst, int32_t* kept, int32_t* status, cudaStream_t st);
// merge + gather of X, K, V.
// E: the per-token weights [B, N] of the score-weighted merge, or null for the plain mean.
void launch_compact(const Dims& D, const void* X, const void* K, const void* V,
                    const int32_t* kept, const int32_t* msrc, const int32_t* mdst, void* Xo,
                    void* Ko, void* Vo, const float* E, int32_t* status, cudaStream_t st);
// Km [B, N, dh] float32 = mean over the heads of K [B, H, N, dh].
void launch_mean_heads(const Dims& D, const void* K, float* Km, cudaStream_t st);

// Sec. 3.2: rows idx[b][0..n_sub) of O gathered into Os [B, n_sub, d] (D describes O).
void launch_gather_rows(const Dims& D, int n_sub, const void* O, const int32_t* idx, void* Os,
                        int32_t* status, cudaStream_t st);
void fill_i32(int32_t* p, int n, int v, cudaStream_t st);
// Sec. 3.1 / Conclusion: [system, compacted visual, prompt] rows and their original positions.
void launch_reassemble(const Dims& D, int n_sys, int n_text, const void* Hs, const void* Xo,
                       const int32_t* kept, void* Ho, int32_t* pos, cudaStream_t st);

// Conclusion: rotary tables cos / sin [rows][head_dim / 2] of the given position IDs.
void launch_rope_tables(const int32_t* pos, long long rows, int head_dim, double base, float* cosv,
                        float* sinv, cudaStream_t st);

// Layer-2 probe (Eq. 3-1 / 3-2): visual rows of the attention output and the probe rows'
// attention to the visual tokens, from Q, K, V [B, H, L, dh] (16-bit storage, dh = 128).
size_t probe_workspace_bytes(int B, int H, int L, int dh);
tc_status launch_probe(int B, int H, int dh, int L, int n_sys, int n_vis, int probe_start, int n_probe,
                       const void* Q, const void* K, const void* V, void* O, void* A, void* ws,
                       int32_t* status, cudaStream_t st, int bf);

// G = O O^T (float32 out, rows ldg floats apart).
tc_status launch_gram(const Dims& D, const void* O, float* G, int ldg, int32_t* status, cudaStream_t st);

// C [batch][M][W] = A B^T on the tensor cores, float32-accurate, for A [batch][M][K] and B [batch][W][K]
// with the contraction index contiguous; W, pitches and strides (in floats) multiples of four, bases
// 16-byte aligned.  C and / or its transpose CT [batch][W][M] are written (either may be null).
// of_batch: images of the whole call that these are a part of.
struct F32x3Operand {
  const float* p;
  int ld;          // floats between rows
  size_t stride;   // floats between images
  int rows = -1;   // rows that exist, the others read as zero (-1: all of M or W)
};
struct F32x3Result {
  float* C;
  int ld;
  size_t stride;
  float* CT;
  int ldT;
  size_t strideT;
  int rows_t = -1;        // rows of C that go to CT (-1: all)
  bool subtract = false;  // C -= A B^T, C counting as zero in rows zero_from .. zero_to - 1
  int zero_from = 0, zero_to = 0;
  bool symmetric = false; // A and B are the same: C is to be symmetric bit for bit
};
tc_status launch_gemm_f32x3(const F32x3Operand& A, const F32x3Operand& B, int M, int W, int K, int batch,
                            int of_batch, const F32x3Result& R, int32_t* status, cudaStream_t st, int cls);

// RinvT [batch][k][k] = L^{-1} (zero above the diagonal) with L L^T = S + shift_rel max_i S_ii I, for
// S [batch][k][k] symmetric (overwritten), k a multiple of 16.  A pivot well below zero (or no number)
// is reported as TC_ERR_BREAKDOWN.  Above CHOL_BLOCK_MAX the factorisation is blocked and needs the
// panel [batch][chol_panel_floats(k)].
constexpr int CHOL_BLOCK_MAX = 192;
constexpr int TCP_MAX = 640;  // widest subspace whose products run on the tensor cores
size_t chol_panel_floats(int k);
tc_status launch_chol_inv(float* S, float* RinvT, float* panel, int k, int batch, int of_batch, float shift_rel,
                          int32_t* status, cudaStream_t st);

// RinvT as above for any k up to 1024, by plain float32 multiply-adds in the order of the textbook
// loops; a pivot that is not positive is replaced and reported.  F: [batch][k][k] scratch.
void launch_chol_inv_f32(float* S, float* RinvT, float* F, int k, int batch, float shift_rel, int32_t* status,
                         cudaStream_t st);

// Eigen-decomposition of the symmetric part of H [batch][n][ldh], 3 <= n <= EIG_TRIDIAG_MAX:
// theta [batch][n] ascending, ZT [batch][n][ldz] with the eigenvectors in its rows (zero rows for
// eigenvalues under a quarter of the rank cut-off rank_tol^2 theta_max).  scratch: batch *
// eig_tridiag_scratch_bytes(n) bytes, 16-byte aligned.
constexpr int EIG_TRIDIAG_MAX = 768;
bool eig_tridiag_supported(int n);
size_t eig_tridiag_scratch_bytes(int n);
tc_status launch_eig_tridiag(const float* H, size_t sH, int ldh, int n, int batch, float rank_tol, float* theta,
                             float* ZT, size_t sZ, int ldz, void* scratch, int32_t* status, cudaStream_t st);

// bytes per image of the work array of either eigen-solver (the Jacobi work matrix is k x k)
size_t jacobi_rot_bytes(int n);   // rotations of a sweep, per image
inline size_t jacobi_work_bytes(int k) { return align_up(eig_tridiag_scratch_bytes(k), 256); }

// Eigen-decomposition of G and Eq. 3-6:  C, theta (unsorted), then sorted sigma / rank; on the raw
// terms (score_norm == TC_NORM_NONE) Eq. 3-8 as well.  Everything points at image b0 of the batch.
struct ScoreIo {
  float* C;                       // out
  const float* S = nullptr;       // Eq. 3-7, for E
  float* E = nullptr;             // out, may be null
  float* sigma = nullptr;         // out, may be null
  int32_t* rank = nullptr;        // out, may be null
  int32_t* status;
  bool values_only = false;       // the caller reads no eigenvectors (C), only sigma and the rank
  cudaEvent_t g_ready = nullptr;  // after it G is complete, where it is built on another stream
  cudaEvent_t s_ready = nullptr;  // after it S is
};
tc_status launch_ics(const Dims& D, const Plan& P, char* ws, int b0, const void* O, const ScoreIo& io,
                     cudaStream_t st);

}  // namespace tc
