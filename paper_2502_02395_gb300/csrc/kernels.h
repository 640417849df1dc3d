// Launchers of the device kernels (internal).
#pragma once

#include <atomic>

#include "h2_internal.h"

namespace h2 {

// Number of kernels this library has launched (reported by h2_stats), and of
// those this thread launched (what a capture holds: other threads go on).
struct LaunchCount {
  std::atomic<long long> all{0};
  inline static thread_local long long mine = 0;
  void operator++() { *this += 1; }
  void operator+=(long long n) { all += n, mine += n; }
};
extern LaunchCount g_launches;
// Tensor-core GEMM kernel form of the factorization's main chain
// (projection, Schur update), process-wide (H2_OPT_TC_KERNEL): 0 one CTA per
// batch entry, 1 a persistent grid of two CTAs per SM, 2 (default) the
// persistent warp-specialized kernel with two TMEM accumulators.  The coupling
// products on their own stream always use form 0, so that they keep sharing
// the SMs with the main chain.
extern std::atomic<int> g_tc_kernel;
// The substitution's per-box steps: 1 the streamed persistent form
// (bulk-copy ring) on levels with at least one box per SM, 2 on every level
// of a supported shape, 0 (default) never (row-split kernels); process-wide
// (H2_OPT_BOX_STREAM).
extern std::atomic<int> g_box_stream;
// Launch shapes of the substitution (h2_autotune): CTAs per SM targeted by
// the per-box row splits (default 1) and of the TMA-fed pair kernels
// (default 3; at most 3 fit their shared-memory rings).
extern std::atomic<int> g_box_ctas_per_sm;
extern std::atomic<int> g_pair_ctas_per_sm;

int num_sms();  // of the current device

// Lets kernel f be launched with as much dynamic shared memory as the device
// allows (once per kernel and device; safe from several threads).
void allow_smem(const void* f);

// The first failed launch of this thread since the last look, and none from
// then on.  (cudaGetLastError alone does not do: a cudaFuncSetAttribute that
// succeeds resets the runtime's record.)
cudaError_t take_launch_error();
// whether there is one
bool launch_error_pending();
void note_launch(cudaError_t e);

// kernels_factor.cu
void launch_eval_blocks(const KernelFn& G, const double* pts, int64_t npairs, const int64_t* ptr, const int32_t* pi,
                        const int32_t* pj, const int64_t* idx, int n, double* out, cudaStream_t st);
template <typename S, typename T>
void launch_convert(const S* in, T* out, int64_t n, cudaStream_t st);
template <typename T, typename TB>
void gemm_simt(int M, int N, int K, const T* A, int64_t sA, const int32_t* ia, int lda, bool tA, const TB* B,
               int64_t sB, const int32_t* ib, int ldb, bool tB, T* C, int64_t sC, const int32_t* ic, int ldc,
               T alpha, T beta, int64_t batch, cudaStream_t st);
template <typename T>
// true when the compact-WY factor Tw was formed too (Tw non-NULL, FP32 register form)
bool launch_qr_panel(int nb, int D, int K, const T* Xin, T* Vout, T* tau, T* Tm, T* gscr, cudaStream_t st,
                     T* Tw = nullptr);
template <typename T>
void launch_wy_tfactor(int nb, int K, const T* S, const T* tau, T* Tw, cudaStream_t st);
template <typename T>
void launch_perm_identity(int nb, int D, int K, T* U, cudaStream_t st);
// U = [Q[:, K:] Q[:, :K]], Q = I - W1 V^T (W1 D x K row-major, V D x K
// column-major), as column-major U, row-major Ur and 16-bit U16 (NULL: none)
// (any D, K; with padding, Dp and Kp > their logical sizes, rs: where the
// logical rows lie; the padding itself is launch_form_u_pads')
void launch_form_u(int64_t nb, int D, int K, const float* W1, const float* V, float* U, float* Ur, void* u16,
                   int bf16, int Dp, int Kp, PadSeg rs, cudaStream_t st);
// a3: the inverses of the R x R blocks (FP64: their LU factors too, on stream
// side).  True when piv holds the pivot rows and wants launch_pivot_sequence.
// (FP64: piv has room for 2 nb R entries.)
template <typename T>
bool launch_lu_inverse(int nb, int D, int R, const T* Ablk, const int32_t* diag_idx, double* lu, T* luT,
                       int32_t* piv, T* Ainv, int32_t* status, int level, cudaStream_t st, cudaStream_t side);
// the FP16/BF16 factorizations' a3 in FP64: FP32 blocks in, FP32 inverse out
// (scratch lu, inv: nb * R * R each)
bool launch_lu_inverse_f64_for_f32(int nb, int D, int R, const float* Ablk, const int32_t* diag_idx, double* lu,
                                   double* inv, int32_t* piv, float* Ainv, int32_t* status, int level,
                                   cudaStream_t st);
void launch_pivot_sequence(int nb, int R, int32_t* piv, cudaStream_t st);
template <typename T>
void launch_merge(int D, int K, int64_t NP, const T* Ahat, const int32_t* ni, const int32_t* nj,
                  const int32_t* ndst, int64_t FP, const T* Shat, const int32_t* fi, const int32_t* fj,
                  const int32_t* fdst, T* Apar, cudaStream_t st);

// kernels_tc.cu: tensor-core (tcgen05 + TMA) batched GEMM
//   C_b = alpha * (*alpha_dev) * A_b B_b^T, A_b = matrix ia[b] (rowsA x K,
//   K-major, 16-bit) of the nA-matrix array A, B_b likewise, FP32
//   accumulation; out_mode 0: FP32 row-major C, 1: 16-bit C^T, 3: FP32
//   C += result (read-modify-write).
// gemm_tc returns false (and launches nothing) for unsupported shapes.
bool gemm_tc_supported(int M, int N, int K, int lda, int ldb, int ldc);
bool gemm_tc(int ab_bf16, int M, int N, int K, const void* A, int64_t nA, int rowsA, int lda, const int32_t* ia,
             const void* B, int64_t nB, int rowsB, int ldb, const int32_t* ib, void* C, int64_t sC,
             const int32_t* ic, int ldc, int out_mode, int out_bf16, float alpha, const float* alpha_dev,
             int64_t batch, int32_t* err, cudaStream_t st, void* C2 = nullptr, int qsplit = -1,
             const int32_t* qi = nullptr, const int32_t* qj = nullptr, unsigned int* amax_ss = nullptr,
             int64_t rowsA_total = 0,  // rowsA_total > 0: the rows A's tensor map spans (else nA * rowsA)
             int form = -1);           // kernel form 0 / 1 / 2 (g_tc_kernel's meaning); -1: g_tc_kernel
// 2-D tensor map over a rows x cols 16-bit array (row stride ld elements)
// with box_rows x box_cols tiles, no swizzle (dense row-major tiles in
// shared memory).  False if the driver or the shape does not allow it.
bool make_tile_map(CUtensorMap* tm, const void* base, int bf16, uint64_t rows, uint64_t cols, uint64_t ld,
                   uint32_t box_rows, uint32_t box_cols);
// One CTA whose thread 0 waits (bounded by timeout_ns) on an mbarrier that
// nothing completes, then sets *flag = 1: the self-test of the bounded waits.
void launch_wait_selftest(unsigned long long timeout_ns, int32_t* flag, cudaStream_t st);
template <typename S>
void launch_amax_blocks(const S* base, int64_t nblk, int64_t stride, int rows, int cols, int ld, unsigned int* out,
                        cudaStream_t st, const int32_t* idx = nullptr);  // idx: block q is base + idx[q] stride
// Scale of a 16-bit copy: the largest power of two s with max |in| s <= target,
// to scale[0] (1 / s to scale[1]); inv (optional) = 1 / (other s) or, squared,
// 1 / (other s s).  amax NULL: s = 1, nothing is written.
struct LowpScale {
  const unsigned int* amax = nullptr;
  float target = 1.0f;
  float* scale = nullptr;
  const float* other = nullptr;
  float* inv = nullptr;
  bool squared = false;
};
template <typename S>
void launch_to_lowp(int bf16, const S* in, void* out, int64_t n, const LowpScale& sc, cudaStream_t st);
void launch_merge_lowp(int D, int K, int64_t NP, const float* Ahat, const int32_t* ni, const int32_t* nj,
                       const int32_t* ndst, int64_t FP, const float* Shat, const int32_t* fi, const int32_t* fj,
                       const int32_t* fdst, void* Apar, const unsigned int* am, const unsigned int* am2, float* scale,
                       int bf16, cudaStream_t st, const int32_t* mirror = nullptr, int skip_lower = 0);
// 16-bit D x D blocks dst[k] = (block src[k])^T outside the SS quadrant
void launch_transpose16_blocks(int D, int R, int64_t n, const int32_t* dst, const int32_t* src, void* A,
                               cudaStream_t st);

// kernels_solve.cu: substitution (Eq. 24-31 and its mirror), H^2 matvec,
// refinement vector operations
// Ahat of level L in storage type TS (T itself, or 16-bit scaled by s with
// iscale -> 1/s on the device; iscale NULL means 1)
// The children of a level's boxes as the first forward step reads them:
// c (nb_c * D), the SR pair sums in part, the near-pair ranges ptr, the
// 16-bit scale of Ahat (NULL: 1) and the child level's D, R, K.  c NULL:
// the input is the level's own vin (leaf level).
template <typename T>
struct ChildIn {
  const T* c = nullptr;
  const T* part = nullptr;
  const int64_t* ptr = nullptr;
  const float* iscale = nullptr;
  int D = 0, R = 0, K = 0;
};
template <typename T>
void launch_fwd1(const DevLevel& L, const FacLevel<T>& F, const ChildIn<T>& ch, cudaStream_t st);

template <typename T, typename TS>
void launch_fwd2(const DevLevel& L, const FacLevel<T>& F, const TS* Ahat, const float* iscale, cudaStream_t st);
template <typename T, typename TS>
void launch_fwd3(const DevLevel& L, const FacLevel<T>& F, const TS* Ahat, const float* iscale, T* parent_vin,
                 cudaStream_t st);
template <typename T, typename TS>
void launch_bwd1(const DevLevel& L, const FacLevel<T>& F, const TS* Ahat, const float* iscale, const T* parent_x,
                 cudaStream_t st);
template <typename T, typename TS>
void launch_bwd2(const DevLevel& L, const FacLevel<T>& F, const TS* Ahat, const float* iscale, const T* parent_x,
                 cudaStream_t st);
// The cluster form (a pair step and the per-box step after it in one launch)
// of levels with few boxes: the CTAs per box a level takes it with (0: not at
// all), and its four steps.
// launch_cl_up: level L's SR sums and the parent's first step ([M1; U^S] with
// dimensions D1, R1 into u and c; at the root M1 = the inverse, R1 = D1).
template <typename T, typename TS>
int subst_clustered(const DevLevel& L, const TS* Ahat);
template <typename T, typename TS>
void launch_cl_fwd2(const DevLevel& L, int CS, const FacLevel<T>& F, const TS* Ahat, const float* iscale, cudaStream_t st);
template <typename T, typename TS>
void launch_cl_up(const DevLevel& L, int CS, const FacLevel<T>& F, const TS* Ahat, const float* iscale, int D1, int R1,
                  const T* M1, const T* U, T* u, T* c, cudaStream_t st);
template <typename T, typename TS>
void launch_cl_bwd1(const DevLevel& L, int CS, const FacLevel<T>& F, const TS* Ahat, const float* iscale, const T* parent_x,
                    cudaStream_t st);
template <typename T, typename TS>
void launch_cl_bwd2(const DevLevel& L, int CS, const FacLevel<T>& F, const TS* Ahat, const float* iscale, const T* parent_x,
                    cudaStream_t st);
template <typename T>
void launch_gemv_rows(int nb, int n, const T* M, const T* x, T* y, cudaStream_t st);
template <typename T>
void launch_transpose_pairs(int D, int64_t n, const int32_t* dst, const int32_t* src, T* A, cudaStream_t st);
template <typename T>
void launch_transpose_blocks(int64_t nb, int D, const T* in, T* out, cudaStream_t st);  // out_b = in_b^T (D x D)  // y = M x, M n x n row-major

template <typename T>
void launch_matvec_up(const DevLevel& L, const T* X, const T* x, T* xh, cudaStream_t st);
// out rows = base + X yh + sums of partial products (see mv_rows_kernel)
template <typename T>
void launch_matvec_rows(int nb, int D, int K, const T* X, const T* yh, const T* base, T* out, int seg,
                        const int64_t* ptr, const int32_t* ent, const T* part, bool pdl, cudaStream_t st);
// Block rows of several levels in one launch (see mv_block_rows_kernel): per
// level nb boxes of n rows, lists ptr / fj, blocks M, input x, basis X (n x K
// with coefficients yh, or NULL), output; nch and cta0 are the launcher's.
template <typename T>
struct BlockRowLevel {
  const int64_t* ptr;
  const int32_t* fj;
  const T *M, *x, *X, *yh;
  T* out;
  int nb, n, K, nch, cta0;
};
constexpr int kMaxRowLevels = 32;
template <typename T>
struct BlockRowArgs {
  int nlev;
  BlockRowLevel<T> lv[kMaxRowLevels];
};
template <typename T>
void launch_matvec_block_rows(BlockRowArgs<T> a, cudaStream_t st);
// The FP64 matvec with each FP64 matrix held as an FP32 pair (hi = fl32, lo
// = fl32 of the rest) and FP32-pair arithmetic throughout: the input vector
// is split once (launch_split_df), the basis coefficients xhat / yhat of
// every level and the leaf partial products stay FP32 pairs, and only the
// leaf output is converted to FP64.
// up: xhat_i = X_i^T z_i (z: the leaf input or the children's xhat)
void launch_matvec_up_df(const DevLevel& L, const float* Xh, const float* Xl, const float* zh, const float* zl,
                         float* oh, float* ol, cudaStream_t st);
// couplings of all levels in one launch: per level its far lists, the
// couplings S (hi / lo), xhat and yhat pairs; CTAs cta0 .. cta0 + nb nch - 1
// (nch 64-row chunks per box)
struct FarDfLevel {
  const int64_t* ptr;
  const int32_t* fj;
  const float *Sh, *Sl, *xh, *xl;
  float *yh, *yl;
  int nb, K, nch, cta0;
};
constexpr int kMaxFarDfLevels = 32;
struct FarDfArgs {
  int nlev;
  FarDfLevel lv[kMaxFarDfLevels];
};
void launch_matvec_far_df_all(const FarDfArgs& a, cudaStream_t st);
// rows in pairs (see mv_rows_kernel and RowsDf): out = base + X yh + sums of
// partial products; as pairs into oh / ol, or as FP64 into y (ny rows a box)
void launch_matvec_rows_df(int nb, int D, int K, const float* Xh, const float* Xl, const float* yhh, const float* yhl,
                           const float* bh, const float* bl, int seg, const int64_t* ptr, const int32_t* ent,
                           const float* ph, const float* pl, float* oh, float* ol, double* y, int ny, cudaStream_t st);
// leaf, general near lists: y_i = X_i yhat_i + sum_{near j} A_ij x_j, ny rows a
// box in y
void launch_matvec_leaf_df(const DevLevel& L, const float* Ah, const float* Al, const float* Xh, const float* Xl,
                           const float* xh, const float* xl, const float* yhh, const float* yhl, double* y, int ny,
                           cudaStream_t st);
// h = fl32(v), l = fl32(v - h); v has n entries in segments of p.len, h and l
// nb segments of p.str (the rest zero)
void launch_split_df(const double* v, float* h, float* l, int64_t n, PadSeg p, cudaStream_t st);
// Leaf matvec on the stored (i <= j) halves of symmetric leaf near blocks:
// per stored pair k = (ui[k], uj[k]) the partial products [A x_j; A^T x_i]
// into part (2 D per pair), then per box y = X yh + its partial products.
bool sym_supported(int n);  // n a multiple of 4, at most 256
// (pdl: launched to overlap its predecessor; off where events bracket it)
// (min_n, max_n: the smallest and largest block, multiples of 4 up to 256)
void launch_matvec_sym_pairs(int min_n, int max_n, int64_t npu, const SymPair* desc, const float* A, const float* x,
                             float* part, bool pdl, cudaStream_t st, const GmState* state = nullptr,
                             unsigned long long* stamp = nullptr);  // (times of iteration state->j)
void launch_matvec_sym_pairs_df(int min_n, int max_n, int64_t npu, const SymPair* desc, const float* Ah,
                                const float* Al, const float* xh, const float* xl, float* ph, float* pl,
                                cudaStream_t st);
// FP32 copies of nblk blocks (block k from in[idx[k]], or in[k]): a block of
// rows x cols entries whose logical rows and columns lie at rs and cs, zeros
// elsewhere; hi = fl32(v) and, lo non-NULL, lo = fl32(v - hi).  di / dj
// non-NULL: blocks with di[k] == dj[k] get 1 on the padding's diagonal.
template <typename Ti>
void launch_pad_blocks(const Ti* in, const int32_t* idx, int64_t nblk, int rows, PadSeg rs, int cols, PadSeg cs,
                       float* hi, float* lo, const int32_t* di, const int32_t* dj, cudaStream_t st);
// the padding's part of U and Ur (zeros, and one 1 per padding row and
// column) for D x D blocks with R complement columns, of which Rl and Kl
// columns and the rows at rs are logical
void launch_form_u_pads(int64_t nb, int D, int R, int Rl, int Kl, PadSeg rs, float* U, float* Ur, cudaStream_t st);

void launch_gather(const int64_t* slot, const double* src, double* dst, int64_t nslots, cudaStream_t st);
void launch_scatter(const int64_t* slot, const double* src, double* dst, int64_t nslots, cudaStream_t st);
void launch_residual(const double* b, const double* y, double* r, int64_t n, cudaStream_t st);
template <typename T>
void launch_norm2(const T* v, int64_t n, double* out, cudaStream_t st);  // out[0] = sum v^2 (FP64), out[1..256] scratch
template <typename Ti, typename To>
void launch_scaled_copy(const Ti* in, const double* nrm2, bool inverse, To* out, int64_t n, cudaStream_t st);
// (the FP32 vectors of the next three have padded boxes: segment p)
void launch_pad_scaled_copy(const double* in, const double* nrm2, float* out, int64_t n, PadSeg p, cudaStream_t st);
template <typename T>
void launch_scale_to(const double* in, const double* norm2, T* out, int64_t n, PadSeg p, cudaStream_t st);
template <typename T>
void launch_axpy_from(const T* d, const double* norm2, double* x, int64_t n, PadSeg p, cudaStream_t st);
// x += sum_v coef[v] V_v for padded FP32 vectors V_v, ldv apart
void launch_pad_axpy(const float* V, int64_t ldv, int nv, const double* coef, double* x, int64_t n, PadSeg p,
                     cudaStream_t st);
void launch_unpad(const float* in, double* out, int64_t n, PadSeg p, cudaStream_t st);
// One inner FGMRES iteration's vector work (classical Gram-Schmidt applied
// twice, FP32 vectors with FP32-pair sums), the iteration's index j read from
// state->j so that the same launches serve every iteration of a cycle: Z_j =
// xs; w -= V (V^T w) twice; V_j+1 = vin = w / ||w||; h1, h2, ||w||^2 and the
// iteration count to pinned host memory.  n entries per vector, m0 the
// restart; part holds (2 (m0 + 1) + 1) * kOrthCtas doubles.
constexpr int kOrthCtas = 2 * 152;
struct OrthArgs {
  float *V, *Z, *w, *vin;
  const float* xs;
  int64_t n;
  int m0, ctas;
  double *part, *h;  // h: h1 (m0 + 2), h2 (m0 + 2) on the device
  GmState* state;
  unsigned long long* stamp;
  double* host;              // pinned: h1, h2, ||w||^2
  unsigned long long* flag;  // pinned
};
int orth_ctas(int64_t n);
void launch_orth(const OrthArgs& a, cudaStream_t st);
// the cycle's start: V_0 = vin = r / sqrt(nrm2), j = 0, times cleared
void launch_gm_start(const float* r, const double* nrm2, float* V, float* vin, int64_t n, int m0, GmState* state,
                     unsigned long long* stamp, cudaStream_t st);
// x += sum_{v < k} y[1 + v] V_v with k = y[0] (device), padded FP32 vectors
void launch_pad_axpy_dev(const float* V, int64_t ldv, const double* y, double* x, int64_t n, PadSeg p,
                         cudaStream_t st);
// GMRES: out[v] (+)= V_v . w for v < nv (part: nv * 128 scratch); w += sign sum_v coef[v] V_v;
// w = src / sqrt(nrm2[0])
template <typename T>
void launch_multi_dot(const T* V, int64_t ldv, int nv, const T* w, int64_t n, double* part, double* out,
                      bool accumulate, cudaStream_t st);
template <typename T, typename TW>
void launch_multi_axpy(const T* V, int64_t ldv, int nv, const double* coef, double sign, TW* w, int64_t n,
                       cudaStream_t st);

}  // namespace h2
