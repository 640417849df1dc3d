// Factorization kernels of the H^2-ULV library (sm_103a).
//
//   eval_blocks_kernel     dense kernel blocks G(B_i, B_j) of the leaf near
//                          pairs and couplings G(SK_i, SK_j) (Algorithm 1),
//                          evaluated from the points
//   gemm_f32_tile_kernel,  SIMT batched GEMM C = alpha op(A) op(B) + beta C in
//   gemm_batched_kernel    FP32 and in FP64
//   qr_reg_kernel,         Householder QR of X^orth (FP32; FP64; any size), its
//   qr_cluster_kernel,     compact WY factor and the explicit U = [U^R U^S]
//   qr_panel_kernel        (Eq. 6-7)
//   gj_rows_kernel,        partial-pivot elimination of Ahat_ii^RR (Algorithm
//   gj_cluster_kernel,     2, with LU in place of Cholesky) and the explicit
//   lu_inverse_kernel      inverse (Ahat_ii^RR)^-1 used by the Schur update and by
//                          the substitution of Eq. 31
//   merge_kernel           children's SS blocks / couplings into the parent
//                          near blocks (the merge of Algorithm 2)
#include <type_traits>

#include "h2_internal.h"
#include "kernels.h"
#include "ptx_util.h"

namespace h2 {

// ------------------------------------------------------------------------
// block evaluation
// ------------------------------------------------------------------------
// out[q] = G(idx[pi[q]], idx[pj[q]]) for the pairs q of a list sorted by (i, j)
// with CSR ptr over i.  One CTA per 32 x 32 tile of a pair.  Bound by the FP64
// pipe (a square root, a division and often an exponential per entry), so
// each tile of a symmetric kernel is evaluated once: the pair i < j writes it
// to its mirror (j, i) too, transposed through shared memory, and a pair
// i > j with a mirror writes nothing (N = 16384: 3.1 ms instead of 5.6 ms with
// every entry evaluated).  Pairs without a mirror (an imported list that is
// not closed) evaluate their own tile.
__device__ __forceinline__ int64_t find_pair(const int64_t* __restrict__ ptr, const int32_t* __restrict__ pi,
                                             const int32_t* __restrict__ pj, int i, int j) {
  int64_t lo = ptr[i], hi = ptr[i + 1];
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if (pj[mid] < j) lo = mid + 1;
    else hi = mid;
  }
  return lo < ptr[i + 1] && pi[lo] == i && pj[lo] == j ? lo : -1;
}
__global__ void __launch_bounds__(256) eval_blocks_kernel(KernelFn G, const double* __restrict__ pts, int64_t ntile,
                                                          int nt, const int64_t* __restrict__ ptr,
                                                          const int32_t* __restrict__ pi,
                                                          const int32_t* __restrict__ pj,
                                                          const int64_t* __restrict__ idx, int n,
                                                          double* __restrict__ out) {
  __shared__ double tile[32][33];
  __shared__ double xa[32][3], xb[32][3];
  __shared__ int64_t ia[32], ib[32];
  const int tid = threadIdx.x, x = tid & 31, y0 = tid >> 5;
  for (int64_t w = blockIdx.x; w < ntile; w += gridDim.x) {
    const int64_t q = w / (nt * nt);
    const int t = (int)(w - q * (nt * nt)), tr = t / nt * 32, tc = t % nt * 32;
    const int i = pi[q], j = pj[q];
    const int64_t m = i == j ? -1 : find_pair(ptr, pi, pj, j, i);
    if (i > j && m >= 0 && find_pair(ptr, pi, pj, i, j) == q) continue;  // written by its mirror
    if (tid < 64) {
      const int u = (tid < 32 ? tr : tc) + x;
      const int64_t p = u < n ? idx[(int64_t)(tid < 32 ? i : j) * n + u] : -1;
      (tid < 32 ? ia : ib)[x] = p;
      for (int d = 0; d < 3; ++d) (tid < 32 ? xa : xb)[x][d] = p >= 0 ? pts[3 * p + d] : 0.0;
    }
    __syncthreads();
    for (int y = y0; y < 32; y += 8) {
      const int r = tr + y, c = tc + x;
      if (r < n && c < n) {
        const int64_t a = ia[y], b = ib[x];
        const double v = (a < 0 || b < 0) ? ((a < 0 && b < 0 && i == j && r == c) ? 1.0 : 0.0)
                                          : (a == b ? G.diag(xa[y]) : G.off(xa[y], xb[x]));
        out[(q * n + r) * n + c] = v;
        tile[y][x] = v;
      }
    }
    __syncthreads();
    if (m >= 0 && i < j)
      for (int y = y0; y < 32; y += 8) {
        const int r = tc + y, c = tr + x;
        if (r < n && c < n) out[(m * n + r) * n + c] = tile[x][y];
      }
    __syncthreads();
  }
}

void launch_eval_blocks(const KernelFn& G, const double* pts, int64_t npairs, const int64_t* ptr, const int32_t* pi,
                        const int32_t* pj, const int64_t* idx, int n, double* out, cudaStream_t st) {
  if (npairs == 0 || n == 0) return;
  const int nt = (n + 31) / 32;
  const int64_t ntile = npairs * nt * nt;
  ++g_launches;
  eval_blocks_kernel<<<(unsigned)std::min<int64_t>(ntile, 152 * 64), 256, 0, st>>>(G, pts, ntile, nt, ptr, pi, pj, idx,
                                                                                   n, out);
}

// ------------------------------------------------------------------------
// conversions
// ------------------------------------------------------------------------
template <typename S, typename T>
__global__ void convert_kernel(const S* __restrict__ in, T* __restrict__ out, int64_t n) {
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x)
    out[e] = (T)in[e];
}
template <typename S, typename T>
void launch_convert(const S* in, T* out, int64_t n, cudaStream_t st) {
  if (n == 0) return;
  int blocks = (int)std::min<int64_t>((n + 255) / 256, 152 * 32);
  ++g_launches;
  convert_kernel<S, T><<<blocks, 256, 0, st>>>(in, out, n);
}
template void launch_convert<double, float>(const double*, float*, int64_t, cudaStream_t);
template void launch_convert<double, double>(const double*, double*, int64_t, cudaStream_t);
template void launch_convert<float, double>(const float*, double*, int64_t, cudaStream_t);
template void launch_convert<float, float>(const float*, float*, int64_t, cudaStream_t);

// ------------------------------------------------------------------------
// SIMT batched GEMM (row-major operands):
//   op(A)(m,k) = tA ? A[k*lda+m] : A[m*lda+k]
//   op(B)(k,n) = tB ? B[n*ldb+k] : B[k*ldb+n]
//   C(m,n)     = C[m*ldc+n]
// Batch b uses A + (ia ? ia[b] : b) * sA, likewise B and C.  Bound by the FP64
// pipe in FP64 (300 products of 256^3 in 8.2 ms, 1.23 of 1.25 TFLOP/s).  Sums of
// 7-bit digits on the tensor cores took 0.96 ms, but a digit form holds a row in
// fixed point below its largest entry: the small entries of a graded row are
// lost, and of the second product of a projection a third to a half of the
// entries had no bound as good as an FP64 sum's.
// ------------------------------------------------------------------------
template <typename T, typename TB>
__global__ void __launch_bounds__(256)
gemm_batched_kernel(int M, int N, int K, const T* __restrict__ A, int64_t sA, const int32_t* __restrict__ ia,
                    int lda, int tA, const TB* __restrict__ B, int64_t sB, const int32_t* __restrict__ ib,
                    int ldb, int tB, T* __restrict__ C, int64_t sC, const int32_t* __restrict__ ic, int ldc,
                    T alpha, T beta, int64_t batch) {
  constexpr int BM = 64, BN = 64, BK = 16;
  __shared__ T As[BK][BM + 1];
  __shared__ T Bs[BK][BN + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  for (int64_t b = blockIdx.z; b < batch; b += gridDim.z) {
    const T* Ab = A + (ia ? (int64_t)ia[b] : b) * sA;
    const TB* Bb = B + (ib ? (int64_t)ib[b] : b) * sB;
    T* Cb = C + (ic ? (int64_t)ic[b] : b) * sC;
    T acc[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
    for (int k0 = 0; k0 < K; k0 += BK) {
      for (int e = threadIdx.x; e < BM * BK; e += 256) {
        int mm, kk;
        if (tA) { mm = e % BM; kk = e / BM; } else { kk = e % BK; mm = e / BK; }
        int gm = m0 + mm, gk = k0 + kk;
        T v = T(0);
        if (gm < M && gk < K) v = tA ? Ab[(int64_t)gk * lda + gm] : Ab[(int64_t)gm * lda + gk];
        As[kk][mm] = v;
      }
      for (int e = threadIdx.x; e < BN * BK; e += 256) {
        int nn, kk;
        if (tB) { kk = e % BK; nn = e / BK; } else { nn = e % BN; kk = e / BN; }
        int gn = n0 + nn, gk = k0 + kk;
        T v = T(0);
        if (gn < N && gk < K) v = (T)(tB ? Bb[(int64_t)gn * ldb + gk] : Bb[(int64_t)gk * ldb + gn]);
        Bs[kk][nn] = v;
      }
      __syncthreads();
#pragma unroll
      for (int kk = 0; kk < BK; ++kk) {
        T a[4], bb[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
        for (int j = 0; j < 4; ++j) bb[j] = Bs[kk][tx + 16 * j];
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], bb[j], acc[i][j]);
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      int gm = m0 + ty + 16 * i;
      if (gm >= M) continue;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        int gn = n0 + tx + 16 * j;
        if (gn >= N) continue;
        T* cp = Cb + (int64_t)gm * ldc + gn;
        T r = alpha * acc[i][j];
        if (beta != T(0)) r = fma(beta, *cp, r);
        *cp = r;
      }
    }
  }
}

// FP32 form for tile-sized problems: 128 x 128 tiles, BK = 8, 256 threads
// each holding an 8 x 8 block of C (rows ty*4 + {0..3, 64..67}, columns
// tx*4 + {0..3, 64..67}) so that every shared-memory read is a 16-byte
// vector; the next k-slice is fetched into registers while the current one
// is used, and two shared buffers leave one barrier per slice.  Bound by the
// FP32 pipe's issue: the products go two at a time through fma.rn.f32x2 (the
// same roundings as two fmaf), 4000 products of 256 x 256 blocks in 2.66
// instead of 3.18 ms (50 TFLOP/s).  Tiles fitted to the block (104 x 104 for
// 200 x 200, 169 threads) measured the same as 128 x 128 ones.
// H = 1: 64 x 64 tiles, BK = 16, a 4 x 4 block a thread, the same sums, for
// batches whose 128 x 128 tiles leave SMs idle (there a tile's chain of slices
// is the time: 16 products 128 x 128 x 128 in 10 instead of 17 us, U of 16 boxes
// of 256 in 9 instead of 22).
template <int H>
struct G2 {
  static constexpr int BM = 64 * H, BN = BM, BK = H == 2 ? 8 : 16, LD = BM + 4;
  static constexpr int KQ = BK / 4, MQ = BM / 4;  // float4 pieces of a slice's row (k contiguous), of its column
};

template <int H>
__device__ __forceinline__ void g2_load_a(const float* __restrict__ Ab, int lda, int tA, int M, int K, int m0, int k0,
                                          bool vec, float (&ra)[4]) {
  const int t = threadIdx.x;
  if (!tA) {  // A[m * lda + k]: 4 consecutive k of row m
    const int m = m0 + t / G2<H>::KQ, k = k0 + (t % G2<H>::KQ) * 4;
    if (vec && m < M && k + 3 < K) {
      const float4 v = *reinterpret_cast<const float4*>(Ab + (int64_t)m * lda + k);
      ra[0] = v.x, ra[1] = v.y, ra[2] = v.z, ra[3] = v.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) ra[e] = (m < M && k + e < K) ? Ab[(int64_t)m * lda + k + e] : 0.0f;
    }
  } else {  // A[k * lda + m]: 4 consecutive m of row k
    const int k = k0 + t / G2<H>::MQ, m = m0 + (t % G2<H>::MQ) * 4;
    if (vec && k < K && m + 3 < M) {
      const float4 v = *reinterpret_cast<const float4*>(Ab + (int64_t)k * lda + m);
      ra[0] = v.x, ra[1] = v.y, ra[2] = v.z, ra[3] = v.w;
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e) ra[e] = (k < K && m + e < M) ? Ab[(int64_t)k * lda + m + e] : 0.0f;
    }
  }
}
template <int H>
__device__ __forceinline__ void g2_store_a(float (*As)[G2<H>::LD], int tA, const float (&ra)[4]) {
  const int t = threadIdx.x;
  if (!tA) {
    const int m = t / G2<H>::KQ, k = (t % G2<H>::KQ) * 4;
#pragma unroll
    for (int e = 0; e < 4; ++e) As[k + e][m] = ra[e];
  } else {
    const int k = t / G2<H>::MQ, m = (t % G2<H>::MQ) * 4;
    *reinterpret_cast<float4*>(&As[k][m]) = make_float4(ra[0], ra[1], ra[2], ra[3]);
  }
}

// acc = op(A)[m0.., :] op(B)[:, n0..] for one 64 H x 64 H tile (thread layout
// of the tile kernel below); As / Bs are the CTA's two shared buffers.
template <int H>
__device__ __forceinline__ void g2_mainloop(int M, int N, int K, const float* __restrict__ Ab, int lda, int tA,
                                            const float* __restrict__ Bb, int ldb, int tB, int m0, int n0, int vecA,
                                            int vecB, float (*As)[G2<H>::BK][G2<H>::LD], float (*Bs)[G2<H>::BK][G2<H>::LD],
                                            float (&acc)[4 * H][4 * H]) {
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  // op(B)(k, n) tile: B[k * ldb + n] (!tB) or B[n * ldb + k] (tB), stored as
  // Bs[k][n]; the same code as A with the roles of m and n exchanged
  auto load_b = [&](int k0, float (&rb)[4]) {
    if (tB) {  // B[n * ldb + k]: 4 consecutive k of row n
      const int n = n0 + t / G2<H>::KQ, k = k0 + (t % G2<H>::KQ) * 4;
      if (vecB && n < N && k + 3 < K) {
        const float4 v = *reinterpret_cast<const float4*>(Bb + (int64_t)n * ldb + k);
        rb[0] = v.x, rb[1] = v.y, rb[2] = v.z, rb[3] = v.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) rb[e] = (n < N && k + e < K) ? Bb[(int64_t)n * ldb + k + e] : 0.0f;
      }
    } else {  // B[k * ldb + n]: 4 consecutive n of row k
      const int k = k0 + t / G2<H>::MQ, n = n0 + (t % G2<H>::MQ) * 4;
      if (vecB && k < K && n + 3 < N) {
        const float4 v = *reinterpret_cast<const float4*>(Bb + (int64_t)k * ldb + n);
        rb[0] = v.x, rb[1] = v.y, rb[2] = v.z, rb[3] = v.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) rb[e] = (k < K && n + e < N) ? Bb[(int64_t)k * ldb + n + e] : 0.0f;
      }
    }
  };
  auto store_b = [&](float (*Bsb)[G2<H>::LD], const float (&rb)[4]) {
    if (tB) {
      const int n = t / G2<H>::KQ, k = (t % G2<H>::KQ) * 4;
#pragma unroll
      for (int e = 0; e < 4; ++e) Bsb[k + e][n] = rb[e];
    } else {
      const int k = t / G2<H>::MQ, n = (t % G2<H>::MQ) * 4;
      *reinterpret_cast<float4*>(&Bsb[k][n]) = make_float4(rb[0], rb[1], rb[2], rb[3]);
    }
  };
  uint64_t c2[4 * H][2 * H];  // pairs of neighbouring columns
#pragma unroll
  for (int i = 0; i < 4 * H; ++i)
#pragma unroll
    for (int j = 0; j < 2 * H; ++j) c2[i][j] = 0;
  float ra[4], rb[4];
  g2_load_a<H>(Ab, lda, tA, M, K, m0, 0, vecA, ra);
  load_b(0, rb);
  g2_store_a<H>(As[0], tA, ra);
  store_b(Bs[0], rb);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += G2<H>::BK) {
    const bool more = k0 + G2<H>::BK < K;
    if (more) {
      g2_load_a<H>(Ab, lda, tA, M, K, m0, k0 + G2<H>::BK, vecA, ra);
      load_b(k0 + G2<H>::BK, rb);
    }
#pragma unroll
    for (int kk = 0; kk < G2<H>::BK; ++kk) {
      float av[4 * H];
      uint64_t bv[2 * H];
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const float4 a = *reinterpret_cast<const float4*>(&As[buf][kk][ty * 4 + 64 * h]);
        const ulonglong2 b = *reinterpret_cast<const ulonglong2*>(&Bs[buf][kk][tx * 4 + 64 * h]);
        av[4 * h] = a.x, av[4 * h + 1] = a.y, av[4 * h + 2] = a.z, av[4 * h + 3] = a.w;
        bv[2 * h] = b.x, bv[2 * h + 1] = b.y;
      }
#pragma unroll
      for (int i = 0; i < 4 * H; ++i) {
        uint64_t aa;
        asm("mov.b64 %0, {%1, %1};" : "=l"(aa) : "f"(av[i]));
#pragma unroll
        for (int j = 0; j < 2 * H; ++j) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c2[i][j]) : "l"(aa), "l"(bv[j]));
      }
    }
    if (more) {
      g2_store_a<H>(As[buf ^ 1], tA, ra);
      store_b(Bs[buf ^ 1], rb);
    }
    __syncthreads();
    buf ^= 1;
  }
#pragma unroll
  for (int i = 0; i < 4 * H; ++i)
#pragma unroll
    for (int j = 0; j < 2 * H; ++j)
      asm("mov.b64 {%0, %1}, %2;" : "=f"(acc[i][2 * j]), "=f"(acc[i][2 * j + 1]) : "l"(c2[i][j]));
}

template <int H>
__global__ void __launch_bounds__(256, H == 2 ? 2 : 4)
gemm_f32_tile_kernel(int M, int N, int K, const float* __restrict__ A, int64_t sA, const int32_t* __restrict__ ia,
                     int lda, int tA, const float* __restrict__ B, int64_t sB, const int32_t* __restrict__ ib, int ldb,
                     int tB, float* __restrict__ C, int64_t sC, const int32_t* __restrict__ ic, int ldc, float alpha,
                     float beta, int64_t batch, int vecA, int vecB, int vecC) {
  __shared__ __align__(16) float As[2][G2<H>::BK][G2<H>::LD];
  __shared__ __align__(16) float Bs[2][G2<H>::BK][G2<H>::LD];
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int m0 = blockIdx.y * G2<H>::BM, n0 = blockIdx.x * G2<H>::BN;
  for (int64_t b = blockIdx.z; b < batch; b += gridDim.z) {
    const float* Ab = A + (ia ? (int64_t)ia[b] : b) * sA;
    const float* Bb = B + (ib ? (int64_t)ib[b] : b) * sB;
    float* Cb = C + (ic ? (int64_t)ic[b] : b) * sC;
    float acc[4 * H][4 * H];
    g2_mainloop<H>(M, N, K, Ab, lda, tA, Bb, ldb, tB, m0, n0, vecA, vecB, As, Bs, acc);
#pragma unroll
    for (int i = 0; i < 4 * H; ++i) {
      const int m = m0 + ty * 4 + (i & 3) + (i >> 2) * 64;
      if (m >= M) continue;
#pragma unroll
      for (int h = 0; h < H; ++h) {
        const int n = n0 + tx * 4 + h * 64;
        float* cp = Cb + (int64_t)m * ldc + n;
        float v[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) v[e] = alpha * acc[i][h * 4 + e];
        if (vecC && n + 3 < N) {
          if (beta != 0.0f) {
            const float4 o = *reinterpret_cast<const float4*>(cp);
            v[0] = fmaf(beta, o.x, v[0]), v[1] = fmaf(beta, o.y, v[1]), v[2] = fmaf(beta, o.z, v[2]),
            v[3] = fmaf(beta, o.w, v[3]);
          }
          *reinterpret_cast<float4*>(cp) = make_float4(v[0], v[1], v[2], v[3]);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (n + e < N) cp[e] = (beta != 0.0f) ? fmaf(beta, cp[e], v[e]) : v[e];
        }
      }
    }
  }
}

// U from the compact WY form in one pass: Q = I - W1 V^T (W1 = V Tw, D x K
// row-major; V column-major D x K) and U = [Q[:, K:] Q[:, :K]] written three
// ways: column-major U, row-major Ur and the 16-bit column-major copy U16
// (u16 NULL: none).  Tiles and main loop of the tile GEMM; column n of Q is
// column n - K of U for n >= K and n + R otherwise.  VEC: D and K are
// multiples of 4 and nothing is padded, so each thread's 4 x 4 groups lie
// wholly inside or outside the block and on one side of column K and are
// stored as vectors; otherwise entry by entry, row m at its place of rs and
// U's columns behind Rp = Dp - Kp complement columns (no 16-bit copy).
template <bool VEC, int H>
__global__ void __launch_bounds__(256, H == 2 ? 2 : 4) form_u_kernel(int D, int K, const float* __restrict__ W1,
                                                        const float* __restrict__ V, float* __restrict__ U,
                                                        float* __restrict__ Ur, void* __restrict__ u16, int bf16,
                                                        int64_t nb, int Dp, int Kp, PadSeg rs, int vecA, int vecB) {
  __shared__ __align__(16) float As[2][G2<H>::BK][G2<H>::LD];
  __shared__ __align__(16) float Bs[2][G2<H>::BK][G2<H>::LD];
  const int t = threadIdx.x, tx = t & 15, ty = t >> 4;
  const int m0 = blockIdx.y * G2<H>::BM, n0 = blockIdx.x * G2<H>::BN;
  const int R = D - K;
  for (int64_t b = blockIdx.z; b < nb; b += gridDim.z) {
    const float* Ab = W1 + b * (int64_t)D * K;
    const float* Bb = V + b * (int64_t)D * K;  // V^T row-major K x D
    float acc[4 * H][4 * H];
    g2_mainloop<H>(D, D, K, Ab, K, 0, Bb, D, 0, m0, n0, vecA, vecB, As, Bs, acc);
    if constexpr (!VEC) {
      float* Uo = U + b * (int64_t)Dp * Dp;
      float* Uro = Ur + b * (int64_t)Dp * Dp;
#pragma unroll
      for (int i = 0; i < 4 * H; ++i) {
        const int m = m0 + ty * 4 + (i & 3) + (i >> 2) * 64;
        if (m >= D) continue;
        const int mp = m / rs.len * rs.str + m % rs.len;
#pragma unroll
        for (int j = 0; j < 4 * H; ++j) {
          const int n = n0 + tx * 4 + (j & 3) + (j >> 2) * 64;
          if (n >= D) continue;
          const int cp = n >= K ? n - K : Dp - Kp + n;
          const float q = (m == n ? 1.0f : 0.0f) - acc[i][j];
          Uo[(int64_t)cp * Dp + mp] = q;
          Uro[(int64_t)mp * Dp + cp] = q;
        }
      }
      continue;
    }
    float* Ub = U + b * (int64_t)D * D;
    float* Urb = Ur + b * (int64_t)D * D;
    uint16_t* U16b = u16 ? reinterpret_cast<uint16_t*>(u16) + b * (int64_t)D * D : nullptr;
    // three passes over the thread's four 4 x 4 groups (rows mb.., columns
    // nbase..), one output each, to keep few addresses live
#pragma unroll
    for (int pass = 0; pass < 3; ++pass) {
      if (pass == 2 && !U16b) break;
#pragma unroll
      for (int g = 0; g < H * H; ++g) {
        const int q4 = g / H, h = g % H;
        const int mb = m0 + ty * 4 + q4 * 64, nbase = n0 + tx * 4 + h * 64;
        if (mb >= D || nbase >= D) continue;
        const int cb = nbase >= K ? nbase - K : nbase + R;  // U column of Q column nbase
        auto q = [&](int r, int e) {
          return (mb + r == nbase + e ? 1.0f : 0.0f) - acc[q4 * 4 + r][h * 4 + e];
        };
        if (pass == 0) {
#pragma unroll
          for (int r = 0; r < 4; ++r)
            *reinterpret_cast<float4*>(Urb + (int64_t)(mb + r) * D + cb) =
                make_float4(q(r, 0), q(r, 1), q(r, 2), q(r, 3));
        } else if (pass == 1) {
#pragma unroll
          for (int e = 0; e < 4; ++e)
            *reinterpret_cast<float4*>(Ub + (int64_t)(cb + e) * D + mb) = make_float4(q(0, e), q(1, e), q(2, e), q(3, e));
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            uint32_t w0, w1;
            if (bf16) {
              __nv_bfloat162 x0 = __floats2bfloat162_rn(q(0, e), q(1, e)), x1 = __floats2bfloat162_rn(q(2, e), q(3, e));
              w0 = *reinterpret_cast<uint32_t*>(&x0), w1 = *reinterpret_cast<uint32_t*>(&x1);
            } else {
              __half2 x0 = __floats2half2_rn(q(0, e), q(1, e)), x1 = __floats2half2_rn(q(2, e), q(3, e));
              w0 = *reinterpret_cast<uint32_t*>(&x0), w1 = *reinterpret_cast<uint32_t*>(&x1);
            }
            *reinterpret_cast<uint2*>(U16b + (int64_t)(cb + e) * D + mb) = make_uint2(w0, w1);
          }
        }
      }
    }
  }
}
void launch_form_u(int64_t nb, int D, int K, const float* W1, const float* V, float* U, float* Ur, void* u16,
                   int bf16, int Dp, int Kp, PadSeg rs, cudaStream_t st) {
  if (nb == 0 || D == 0) return;
  // (64 x 64 tiles while 128 x 128 ones leave SMs idle)
  const int64_t big = nb * ((D + 127) / 128) * ((D + 127) / 128);
  const int bm = big < num_sms() ? 64 : 128;
  const dim3 g((D + bm - 1) / bm, (D + bm - 1) / bm, (unsigned)std::min<int64_t>(nb, 65535));
  const bool vec = D % 4 == 0 && K % 4 == 0 && Dp == D;
  auto go = vec ? (bm == 64 ? form_u_kernel<true, 1> : form_u_kernel<true, 2>)
                : (bm == 64 ? form_u_kernel<false, 1> : form_u_kernel<false, 2>);
  ++g_launches;
  go<<<g, 256, 0, st>>>(D, K, W1, V, U, Ur, vec ? u16 : nullptr, bf16, nb, Dp, Kp, rs, vec || K % 4 == 0,
                        vec || D % 4 == 0);
}

static bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

template <typename T, typename TB>
void gemm_simt(int M, int N, int K, const T* A, int64_t sA, const int32_t* ia, int lda, bool tA, const TB* B,
               int64_t sB, const int32_t* ib, int ldb, bool tB, T* C, int64_t sC, const int32_t* ic, int ldc,
               T alpha, T beta, int64_t batch, cudaStream_t st) {
  if (batch == 0 || M == 0 || N == 0) return;
  if constexpr (std::is_same<T, float>::value && std::is_same<TB, float>::value) {
    // 16-byte vector access needs 4-element strides and aligned bases
    const int vecA = (lda % 4 == 0) && (sA % 4 == 0) && aligned16(A);
    const int vecB = (ldb % 4 == 0) && (sB % 4 == 0) && aligned16(B);
    const int vecC = (ldc % 4 == 0) && (sC % 4 == 0) && aligned16(C);
    // (64 x 64 tiles while 128 x 128 ones leave SMs idle)
    const int64_t big = batch * ((M + 127) / 128) * ((N + 127) / 128);
    const int bm = big < num_sms() ? 64 : 128;
    const dim3 g2((N + bm - 1) / bm, (M + bm - 1) / bm, (unsigned)std::min<int64_t>(batch, 65535));
    auto go = bm == 64 ? gemm_f32_tile_kernel<1> : gemm_f32_tile_kernel<2>;
    ++g_launches;
    go<<<g2, 256, 0, st>>>(M, N, K, A, sA, ia, lda, tA, B, sB, ib, ldb, tB, C, sC, ic, ldc, alpha, beta, batch, vecA,
                           vecB, vecC);
    return;
  }
  dim3 grid((N + 63) / 64, (M + 63) / 64, (unsigned)std::min<int64_t>(batch, 65535));
  ++g_launches;
  gemm_batched_kernel<T, TB><<<grid, 256, 0, st>>>(M, N, K, A, sA, ia, lda, tA, B, sB, ib, ldb, tB, C, sC, ic, ldc,
                                                   alpha, beta, batch);
}
template void gemm_simt<double, double>(int, int, int, const double*, int64_t, const int32_t*, int, bool,
                                        const double*, int64_t, const int32_t*, int, bool, double*, int64_t,
                                        const int32_t*, int, double, double, int64_t, cudaStream_t);
template void gemm_simt<float, float>(int, int, int, const float*, int64_t, const int32_t*, int, bool,
                                      const float*, int64_t, const int32_t*, int, bool, float*, int64_t,
                                      const int32_t*, int, float, float, int64_t, cudaStream_t);

// ------------------------------------------------------------------------
// a1: complement bases (Eq. 6-7) in three steps:
//   qr_panel_kernel   Householder QR of X^orth (LAPACK geqr2 conventions:
//                     beta = -sign(alpha) |x|), one CTA per box, the panel in
//                     shared memory when it fits.  Writes the reflectors V
//                     (column-major D x K, unit diagonal stored), tau and
//                     T_i = R (row-major K x K, X^orth = U^S T_i).
//   wy_tfactor_kernel the triangular factor of the compact WY form
//                     H_0 ... H_{K-1} = I - V Tw V^T (LAPACK larft, forward,
//                     columnwise) from S = V^T V.
//   identity + GEMMs  U = [Q[:, K:] Q[:, :K]] with Q = I - V Tw V^T, formed
//                     by batched GEMMs (in the caller).
// ------------------------------------------------------------------------
template <typename T>
__device__ T block_sum2(T v, T* sbuf) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (lane == 0) sbuf[warp] = v;
  __syncthreads();
  T t = T(0);
  for (int w = 0; w < nw; ++w) t += sbuf[w];
  __syncthreads();
  return t;
}

// Xin: row-major D x K per box.  Vout: column-major D x K per box.
template <typename T>
__global__ void __launch_bounds__(512) qr_panel_kernel(int D, int K, const T* __restrict__ Xin, T* __restrict__ Vout,
                                                       T* __restrict__ tau_out, T* __restrict__ Tm, T* __restrict__ gscr,
                                                       int use_smem) {
  extern __shared__ __align__(16) unsigned char smraw[];
  __shared__ T red[32];
  __shared__ T s_tau, s_scal, s_beta;
  const int box = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  T* X = use_smem ? reinterpret_cast<T*>(smraw) : gscr + (size_t)box * D * K;  // column-major, ld = D
  const T* src = Xin + (size_t)box * D * K;
  for (int e = tid; e < D * K; e += blockDim.x) {
    const int r = e / K, a = e - r * K;
    X[a * D + r] = src[e];
  }
  __syncthreads();
  for (int k = 0; k < K; ++k) {
    T* xk = X + k * D;
    T part = T(0);
    for (int r = k + 1 + tid; r < D; r += blockDim.x) part += xk[r] * xk[r];
    const T xn2 = block_sum2(part, red);
    if (tid == 0) {
      const T alpha = xk[k];
      if (xn2 == T(0)) {
        s_tau = T(0);
      } else {
        const T beta = -copysign(sqrt(alpha * alpha + xn2), alpha);
        s_tau = (beta - alpha) / beta;
        s_scal = T(1) / (alpha - beta);
        s_beta = beta;
      }
    }
    __syncthreads();
    const T tk = s_tau;
    if (tk != T(0)) {
      const T scal = s_scal;
      for (int r = k + 1 + tid; r < D; r += blockDim.x) xk[r] *= scal;
      __syncthreads();
      for (int j = k + 1 + warp; j < K; j += nw) {
        T* xj = X + j * D;
        const T xjk = xj[k];
        T w = T(0);
        for (int r = k + 1 + lane; r < D; r += 32) w += xk[r] * xj[r];
        for (int o = 16; o; o >>= 1) w += __shfl_xor_sync(0xffffffffu, w, o);
        w = tk * (w + xjk);
        if (lane == 0) xj[k] = xjk - w;
        for (int r = k + 1 + lane; r < D; r += 32) xj[r] -= w * xk[r];
      }
      if (tid == 0) xk[k] = s_beta;
    }
    if (tid == 0) tau_out[(size_t)box * K + k] = tk;
    __syncthreads();
  }
  // R (row-major, upper) and V (column-major, unit diagonal, zeros above)
  T* Rb = Tm + (size_t)box * K * K;
  for (int e = tid; e < K * K; e += blockDim.x) {
    const int a = e / K, b = e - a * K;
    Rb[e] = (b >= a) ? X[b * D + a] : T(0);
  }
  T* Vb = Vout + (size_t)box * D * K;
  for (int e = tid; e < D * K; e += blockDim.x) {
    const int a = e / D, r = e - a * D;
    Vb[e] = (r > a) ? X[a * D + r] : (r == a ? T(1) : T(0));
  }
}

// Tw (row-major K x K, upper): for i = 0..K-1:
//   Tw[0:i, i] = -tau_i Tw[0:i, 0:i] S[0:i, i];  Tw[i, i] = tau_i
// S = V^T V (row-major K x K per box).  Step i: warp w computes the rows
// r = w, w + nwarps, ... of the new column, its lanes splitting the dot
// product over c in [r, i) (Tw is upper triangular).
template <typename T>
__global__ void __launch_bounds__(256) wy_tfactor_kernel(int K, const T* __restrict__ S, const T* __restrict__ tau,
                                                         T* __restrict__ Tw, int use_smem) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int box = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nw = blockDim.x >> 5;
  // K x K row-major working triangle: shared memory when it fits, else the
  // output block itself; w (K entries) always in shared memory
  T* Ts = use_smem ? reinterpret_cast<T*>(smraw) : Tw + (size_t)box * K * K;
  T* w = use_smem ? Ts + K * K : reinterpret_cast<T*>(smraw);
  const T* Sb = S + (size_t)box * K * K;
  const T* tb = tau + (size_t)box * K;
  for (int e = tid; e < K * K; e += blockDim.x) Ts[e] = T(0);
  __syncthreads();
  for (int i = 0; i < K; ++i) {
    for (int r = tid; r < i; r += blockDim.x) w[r] = Sb[r * K + i];
    __syncthreads();
    const T ti = tb[i];
    for (int r = warp; r < i; r += nw) {
      T sacc = T(0);
      for (int c = r + lane; c < i; c += 32) sacc += Ts[r * K + c] * w[c];
      for (int o = 16; o; o >>= 1) sacc += __shfl_xor_sync(0xffffffffu, sacc, o);
      if (lane == 0) Ts[r * K + i] = -ti * sacc;
    }
    if (tid == 0) Ts[i * K + i] = ti;
    __syncthreads();
  }
  T* out = Tw + (size_t)box * K * K;
  if (use_smem)
    for (int e = tid; e < K * K; e += blockDim.x) out[e] = Ts[e];
}

// C[r0.., c0..] = alpha A B for the 4 x 4 tile at (r0, c0) of an h x h
// product of shared-memory operands (row-major, leading dimensions lda, ldb,
// ldc).
template <typename T>
__device__ __forceinline__ void smem_mm4(const T* A, int lda, const T* B, int ldb, T* C, int ldc, int h, T alpha,
                                         int r0, int c0) {
  T acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = T(0);
#pragma unroll 4
  for (int k = 0; k < h; ++k) {
    T a[4], bv[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) a[i] = A[(r0 + i) * lda + k];
#pragma unroll
    for (int j = 0; j < 4; ++j) bv[j] = B[k * ldb + c0 + j];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fma(a[i], bv[j], acc[i][j]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) C[(r0 + i) * ldc + c0 + j] = alpha * acc[i][j];
}

// The same factor from the identity Tw^-1 = striu(S) + diag(1 / tau) of the
// compact WY form (tau_k = 0, a reflector equal to I, gives a zero row and
// column k of Tw: M is made the identity there and Tw_kk set to 0).  M is
// padded to Kp (a power of two, 8 <= Kp <= 128) with the identity and
// inverted in shared memory by recursive 2 x 2 blocking: the 8 x 8
// diagonal blocks by back substitution (one thread per column), then for
// b = 16 .. Kp every diagonal block [T11 T12; 0 T22] gets
// T12 = -T11 (M12 T22) from its two already inverted halves (dense 4 x 4
// register-tiled products; the zeros of the triangles are multiplied too).
// In place: Ms (Kp x Kp upper triangular, leading dimension Kp + 1) becomes
// its inverse; Xs is Kp * Kp / 4 scratch; every thread of the CTA calls it
// (Kp a power of two, 8 <= Kp <= 128; at least Kp threads).
template <typename T>
__device__ void tri_inverse_smem(int Kp, T* Ms, T* Xs) {
  const int ld = Kp + 1, tid = threadIdx.x;
  // 8 x 8 diagonal blocks: thread (q, j) solves M_qq x = e_j
  {
    const int nq = Kp / 8;
    T x[8];
    const int q = tid >> 3, j = tid & 7;
    if (q < nq) {
      const T* Mq = Ms + (size_t)(q * 8) * ld + q * 8;
#pragma unroll
      for (int i = 7; i >= 0; --i) {
        T acc = (i == j) ? T(1) : T(0);
#pragma unroll
        for (int k = i + 1; k < 8; ++k) acc -= Mq[i * ld + k] * x[k];
        x[i] = (i <= j) ? acc / Mq[i * ld + i] : T(0);
      }
    }
    __syncthreads();
    if (q < nq) {
      T* Mq = Ms + (size_t)(q * 8) * ld + q * 8;
#pragma unroll
      for (int i = 0; i < 8; ++i) Mq[i * ld + j] = x[i];
    }
    __syncthreads();
  }
  // the block products in 4 x 4 register tiles, one per thread
  for (int b = 16; b <= Kp; b *= 2) {
    const int h = b / 2, nb = Kp / b, hh = h * h, tw = h / 4, tpb = tw * tw;
    // X_q = M12 T22
    for (int e = tid; e < nb * tpb; e += blockDim.x) {
      const int q = e / tpb, rc = e - q * tpb, r0 = (rc / tw) * 4, c0 = (rc % tw) * 4;
      smem_mm4<T>(Ms + (size_t)(q * b) * ld + q * b + h, ld, Ms + (size_t)(q * b + h) * ld + q * b + h, ld,
                  Xs + (size_t)q * hh, h, h, T(1), r0, c0);
    }
    __syncthreads();
    // T12 = -T11 X_q, in place of M12
    for (int e = tid; e < nb * tpb; e += blockDim.x) {
      const int q = e / tpb, rc = e - q * tpb, r0 = (rc / tw) * 4, c0 = (rc % tw) * 4;
      smem_mm4<T>(Ms + (size_t)(q * b) * ld + q * b, ld, Xs + (size_t)q * hh, h,
                  Ms + (size_t)(q * b) * ld + q * b + h, ld, h, T(-1), r0, c0);
    }
    __syncthreads();
  }
}

template <typename T>
__global__ void __launch_bounds__(256) wy_tinv_kernel(int K, int Kp, const T* __restrict__ S,
                                                      const T* __restrict__ tau, T* __restrict__ Tw) {
  extern __shared__ __align__(16) unsigned char smraw[];
  const int ld = Kp + 1;
  T* Ms = reinterpret_cast<T*>(smraw);  // Kp x ld
  T* Xs = Ms + (size_t)Kp * ld;           // Kp * Kp / 4 scratch
  const int box = blockIdx.x, tid = threadIdx.x;
  const T* Sb = S + (size_t)box * K * K;
  const T* tb = tau + (size_t)box * K;
  for (int e = tid; e < Kp * Kp; e += blockDim.x) {
    const int r = e / Kp, c = e - r * Kp;
    T v = T(0);
    if (r >= K || c >= K) {
      v = (r == c) ? T(1) : T(0);
    } else {
      const bool zr = tb[r] == T(0), zc = tb[c] == T(0);
      if (r == c) v = zr ? T(1) : T(1) / tb[r];
      else if (c > r && !zr && !zc) v = Sb[r * K + c];
    }
    Ms[r * ld + c] = v;
  }
  __syncthreads();
  tri_inverse_smem<T>(Kp, Ms, Xs);
  T* out = Tw + (size_t)box * K * K;
  for (int e = tid; e < K * K; e += blockDim.x) {
    const int r = e / K, c = e - r * K;
    out[e] = (r == c && tb[r] == T(0)) ? T(0) : Ms[r * ld + c];
  }
}

// U (column-major D x D): column c' holds e_{perm(c')}, perm(c') = K + c'
// for c' < R = D - K, c' - R otherwise ([Q[:, K:] Q[:, :K]] of Q = I).
template <typename T>
__global__ void perm_identity_kernel(int nb, int D, int K, T* __restrict__ U) {
  const int R = D - K;
  const int64_t n = (int64_t)nb * D * D;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < n; e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t q = e % ((int64_t)D * D);
    const int cp = (int)(q / D), r = (int)(q % D);
    const int src = cp < R ? K + cp : cp - R;
    U[e] = (r == src) ? T(1) : T(0);
  }
}

// Sums of CPW (8) per-lane values over the warp, left in d in every lane.  A transposed butterfly: at xor-distance 16, 8 and 4
// each lane keeps half of its remaining values and adds its partner's copy
// of them (4 + 2 + 1 shuffles), two plain steps finish one column per group
// of four lanes, and one shuffle per column brings every sum back.
template <int CPW>
__device__ __forceinline__ void qr_reduce_cols(float (&d)[CPW]) {
  static_assert(CPW == 8, "the butterfly is written for 8 columns");
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const bool up = lane & 16;
    const float mine = up ? d[q + 4] : d[q], other = up ? d[q] : d[q + 4];
    d[q] = mine + __shfl_xor_sync(0xffffffffu, other, 16);
  }
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const bool up = lane & 8;
    const float mine = up ? d[q + 2] : d[q], other = up ? d[q] : d[q + 2];
    d[q] = mine + __shfl_xor_sync(0xffffffffu, other, 8);
  }
  {
    const bool up = lane & 4;
    const float mine = up ? d[1] : d[0], other = up ? d[0] : d[1];
    d[0] = mine + __shfl_xor_sync(0xffffffffu, other, 4);
  }
  d[0] += __shfl_xor_sync(0xffffffffu, d[0], 2);
  d[0] += __shfl_xor_sync(0xffffffffu, d[0], 1);
  // lane l now holds the sum of column 4 * bit4(l) + 2 * bit3(l) + bit2(l)
  const float t = d[0];
#pragma unroll
  for (int c = 0; c < 8; ++c) d[c] = __shfl_sync(0xffffffffu, t, ((c >> 2) << 4) | (((c >> 1) & 1) << 3) | ((c & 1) << 2));
}

// Householder reflector of one register-held column (rows lane + 32 s) at
// pivot row k, by the warp that owns it: the column becomes beta at row k and
// v below it (v_k = 1 implied); v (zeros above k) goes to vb (this lane's rows
// together), tau to *stau.
template <int RPL>
__device__ __forceinline__ void qr_reflector(float (&xc)[RPL], int k, int lane, float* vb, float* stau) {
  float alpha = 0.0f, part = 0.0f;
#pragma unroll
  for (int s = 0; s < RPL; ++s) {
    const int r = lane + 32 * s;
    if (r == k) alpha = xc[s];
    if (r > k) part = fmaf(xc[s], xc[s], part);
  }
  alpha = __shfl_sync(0xffffffffu, alpha, k & 31);
  for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  float tau = 0.0f, beta = alpha, scal = 0.0f;
  if (part != 0.0f) {
    beta = -copysignf(sqrtf(fmaf(alpha, alpha, part)), alpha);
    tau = (beta - alpha) / beta;
    scal = 1.0f / (alpha - beta);
  }
  float v[RPL];
#pragma unroll
  for (int s = 0; s < RPL; ++s) {
    const int r = lane + 32 * s;
    v[s] = 0.0f;
    if (r == k) {
      v[s] = 1.0f;
      xc[s] = beta;
    } else if (r > k && tau != 0.0f) {
      xc[s] *= scal;
      v[s] = xc[s];
    }
  }
#pragma unroll
  for (int s = 0; s < RPL; s += 4)
    *reinterpret_cast<float4*>(vb + lane * RPL + s) = make_float4(v[s], v[s + 1], v[s + 2], v[s + 3]);
  if (lane == 0) *stau = tau;
}
// Barriers 1 and 2 of 512 threads: arrive without waiting, or wait.
__device__ __forceinline__ void qr_arrive(int id) { asm volatile("barrier.cta.arrive %0, 512;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void qr_wait(int id) { asm volatile("barrier.cta.sync %0, 512;" ::"r"(id) : "memory"); }

// two floats in one register pair
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t p, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(p));
}

// The same factorization in FP32 with the panel in registers: column j belongs to
// warp j mod 16 and lane l holds rows l, l + 32, ... (D <= 32 RPL, K <= 128).
// Step k: v_k and tau lie in shared memory (two buffers).  The warp of column k
// + 1 updates that column first, forms its reflector, publishes it and arrives
// at step k + 1's barrier without waiting, then catches up with its other
// columns; the other warps update theirs (w = tau v^T x_j, lane-local
// products, one warp reduction for eight columns, x_j -= w v) and wait
// there.  A warp's finished columns (j < k) give the Gram entries v_j^T v_k
// instead, so that after the last step the compact-WY factor Tw = (striu(V^T V) +
// diag(1 / tau))^-1 (zero-tau rows and columns masked, as in wy_tinv_kernel) is
// inverted in shared memory by the same CTA (Tw NULL: no factor).  Two barriers
// alternate: the next publisher has passed the barrier at which everybody
// else had read the buffer it overwrites (the last publisher read it before it arrived).
// Bound by the chain of the reflectors (update of one column, two reductions, a
// square root, a division) and the issue of the updates.  Ten levels of 262144
// points (1024 to 2 boxes of 256 x 128) 3.87 ms; with a barrier between every
// reflector and its updates, columns contiguous and scalar products 5.07 ms; a
// cluster of 2 to 8 CTAs a box was slower (0.27 - 0.42 ms a level against 0.19).
template <int RPL>
__global__ void __launch_bounds__(512) qr_reg_kernel(int D, int K, int Kp, const float* __restrict__ Xin,
                                                     float* __restrict__ Vout, float* __restrict__ tau_out,
                                                     float* __restrict__ Tm, float* __restrict__ Tw) {
  constexpr int NW = 16, CPW = 8;
  extern __shared__ __align__(16) unsigned char qsm[];
  float* vsb = reinterpret_cast<float*>(qsm);          // 2 x RPL * 32
  float* s_tau = vsb + 2 * RPL * 32;                    // 2 (+2 pad)
  float* tau_s = s_tau + 4;                             // Kp
  float* scr = tau_s + Kp;                              // max(32 x 129, Kp^2 / 4): load tile, then Xs
  const int nscr = (32 * 129 > Kp * Kp / 4) ? 32 * 129 : Kp * Kp / 4;
  float* Gm = scr + nscr;                               // Kp x (Kp + 1): Gram entries, then Tw
  const int ldg = Kp + 1;
  float(*tile)[NW * CPW + 1] = reinterpret_cast<float(*)[NW * CPW + 1]>(scr);
  const int box = blockIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const float* src = Xin + (size_t)box * D * K;  // row-major D x K
  uint64_t x2[CPW / 2][RPL];  // columns 2 q and 2 q + 1 of this warp (fma.rn.f32x2: the roundings of two fmaf)
  // load through shared memory, 32 rows at a time (coalesced reads)
#pragma unroll
  for (int s = 0; s < RPL; ++s) {
    for (int e = threadIdx.x; e < 32 * K; e += blockDim.x) {
      const int rr = e / K, cc = e - rr * K, r = 32 * s + rr;
      tile[rr][cc] = (r < D) ? src[(size_t)r * K + cc] : 0.0f;
    }
    __syncthreads();
#pragma unroll
    for (int q = 0; q < CPW / 2; ++q) {
      const int j = warp + 2 * NW * q;
      x2[q][s] = pack2((j < K) ? tile[lane][j] : 0.0f, (j + NW < K) ? tile[lane][j + NW] : 0.0f);
    }
    __syncthreads();
  }
  const bool gram = Tw != nullptr;
  // column c (a constant) as a copy, and back
  auto get = [&](int c, float(&xc)[RPL]) {
#pragma unroll
    for (int s = 0; s < RPL; ++s) {
      float lo, hi;
      unpack2(x2[c / 2][s], lo, hi);
      xc[s] = c % 2 ? hi : lo;
    }
  };
  auto put = [&](int c, const float(&xc)[RPL]) {
#pragma unroll
    for (int s = 0; s < RPL; ++s) {
      float lo, hi;
      unpack2(x2[c / 2][s], lo, hi);
      x2[c / 2][s] = c % 2 ? pack2(lo, xc[s]) : pack2(xc[s], hi);
    }
  };
  if (warp == 0) {
    float xc[RPL];
    get(0, xc);
    qr_reflector<RPL>(xc, 0, lane, vsb, s_tau);
    put(0, xc);
    qr_arrive(1);
  }
#pragma unroll
  for (int kc = 0; kc < CPW; ++kc) {
    for (int w = 0; w < NW; ++w) {
      const int k = NW * kc + w, buf = k & 1;
      if (k >= K) break;
      if (warp == w) __syncwarp();  // (published v_k and arrived itself)
      else qr_wait(buf + 1);
      const float tk = s_tau[buf];
      float v[RPL];
#pragma unroll
      for (int s = 0; s < RPL; s += 4) {
        const float4 t = *reinterpret_cast<const float4*>(vsb + buf * RPL * 32 + lane * RPL + s);
        v[s] = t.x, v[s + 1] = t.y, v[s + 2] = t.z, v[s + 3] = t.w;
      }
      if (threadIdx.x == 0) tau_out[(size_t)box * K + k] = tk, tau_s[k] = tk;
      // the next column first
      auto ahead = [&](int c) {
        float xc[RPL], d = 0.0f;
        get(c, xc);
#pragma unroll
        for (int s = 0; s < RPL; ++s) d = fmaf(v[s], xc[s], d);
        for (int o = 16; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        const float dj = d * tk;
        if (tk != 0.0f)
#pragma unroll
          for (int s = 0; s < RPL; ++s) xc[s] = fmaf(-dj, v[s], xc[s]);
        qr_reflector<RPL>(xc, k + 1, lane, vsb + (buf ^ 1) * RPL * 32, &s_tau[buf ^ 1]);
        qr_arrive((buf ^ 1) + 1);
        put(c, xc);
      };
      const bool next0 = k + 1 < K && w + 1 < NW && warp == w + 1;
      const bool next1 = kc + 1 < CPW && k + 1 < K && w + 1 == NW && warp == 0;
      if (next0) ahead(kc);
      if (kc + 1 < CPW)
        if (next1) ahead(kc + 1);
      if (tk == 0.0f) continue;
      uint64_t vv[RPL], d2[CPW / 2];
#pragma unroll
      for (int s = 0; s < RPL; ++s) vv[s] = pack2(v[s], v[s]);
      float d[CPW];
#pragma unroll
      for (int q = 0; q < CPW / 2; ++q) {
        d2[q] = 0;
#pragma unroll
        for (int s = 0; s < RPL; ++s) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d2[q]) : "l"(vv[s]), "l"(x2[q][s]));
        unpack2(d2[q], d[2 * q], d[2 * q + 1]);
      }
      qr_reduce_cols<CPW>(d);
      float u[CPW];  // -tau w, 0 for the columns that are finished or ahead
#pragma unroll
      for (int c = 0; c < CPW; ++c) {
        const bool after = c > kc ? !(c == kc + 1 && next1) : (c == kc && warp > w && !next0);
        u[c] = after ? -(d[c] * tk) : 0.0f;
        if (gram && lane == 0 && (c < kc || (c == kc && warp < w))) Gm[(warp + NW * c) * ldg + k] = d[c];
      }
#pragma unroll
      for (int q = 0; q < CPW / 2; ++q) {
        if (2 * q + 1 < kc) continue;
        const uint64_t uu = pack2(u[2 * q], u[2 * q + 1]);
#pragma unroll
        for (int s = 0; s < RPL; ++s) asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(x2[q][s]) : "l"(uu), "l"(vv[s]));
      }
    }
  }
  // R (row-major, upper) and V (column-major, unit diagonal, zeros above)
  float* Rb = Tm + (size_t)box * K * K;
  float* Vb = Vout + (size_t)box * D * K;
#pragma unroll
  for (int c = 0; c < CPW; ++c) {
    const int j = warp + NW * c;
    if (j >= K) continue;
    float xc[RPL];
    get(c, xc);
#pragma unroll
    for (int s = 0; s < RPL; ++s) {
      const int r = lane + 32 * s;
      if (r < K) Rb[(size_t)r * K + j] = (r <= j) ? xc[s] : 0.0f;
      if (r < D) Vb[(size_t)j * D + r] = (r > j) ? xc[s] : (r == j ? 1.0f : 0.0f);
    }
  }
  if (!gram) return;
  // M = striu(G) + diag(1 / tau), padded to Kp with the identity, in place
  __syncthreads();
  for (int e = threadIdx.x; e < Kp * Kp; e += blockDim.x) {
    const int r = e / Kp, c = e - r * Kp;
    float v = 0.0f;
    if (r >= K || c >= K) {
      v = (r == c) ? 1.0f : 0.0f;
    } else {
      const bool zr = tau_s[r] == 0.0f, zc = tau_s[c] == 0.0f;
      if (r == c) v = zr ? 1.0f : 1.0f / tau_s[r];
      else if (c > r && !zr && !zc) v = Gm[r * ldg + c];
    }
    Gm[r * ldg + c] = v;
  }
  __syncthreads();
  tri_inverse_smem<float>(Kp, Gm, scr);
  float* out = Tw + (size_t)box * K * K;
  for (int e = threadIdx.x; e < K * K; e += blockDim.x) {
    const int r = e / K, c = e - r * K;
    out[e] = (r == c && tau_s[r] == 0.0f) ? 0.0f : Gm[r * ldg + c];
  }
}

// The same factorization in FP64, a thread-block cluster of C CTAs per box and
// the panel in registers: column j belongs to warp j mod G (G = 16 C), lane l
// holds rows l, l + 32, ... (D <= 256, K <= CW G).  Step k: the warp of column k
// + 1 updates that column first, forms its reflector and writes it to every
// CTA of the cluster (distributed shared memory, two buffers) while the others
// still update; one cluster barrier a step.  Bound by the FP64 pipe (2
// multiply-adds per clock and SM: 5 M per 256 x 128 box) where a level has many
// boxes, by the chain of the steps (two reductions, a square root and a
// division in FP64) where it has few; C is the largest that leaves one CTA an
// SM.  256 x 128: 1.06 ms for 32 boxes, 1.1 ms for 16 to 2; with one CTA per box
// and the panel in global memory 3.4 - 3.9 ms.
template <int CW>
__global__ void __launch_bounds__(512, 1) qr_cluster_kernel(int D, int K, int C, const double* __restrict__ Xin,
                                                            double* __restrict__ Vout, double* __restrict__ tau_out,
                                                            double* __restrict__ Tm) {
  constexpr int NR = 8;
  __shared__ __align__(16) double vb[2][32 * NR];
  __shared__ double tb[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int rank = (int)cluster_rank(), box = blockIdx.x / C, g = rank * 16 + warp, G = 16 * C;
  const double* src = Xin + (size_t)box * D * K;  // row-major D x K
  double x[CW][NR];
#pragma unroll
  for (int c = 0; c < CW; ++c)
#pragma unroll
    for (int s = 0; s < NR; ++s) {
      const int r = lane + 32 * s, j = g + G * c;
      x[c][s] = (r < D && j < K) ? src[(size_t)r * K + j] : 0.0;
    }
  // reflector of this warp's column k = g + G * kc, to buffer k & 1 of every CTA
  auto reflect = [&](int k) {
    const int kc = k / G, s0 = k >> 5;
    double xc[NR];
#pragma unroll
    for (int s = 0; s < NR; ++s) {
      xc[s] = x[0][s];
#pragma unroll
      for (int c = 1; c < CW; ++c) xc[s] = kc == c ? x[c][s] : xc[s];
    }
    double alpha = 0.0, p0 = 0.0, p1 = 0.0;
#pragma unroll
    for (int s = 0; s < NR; ++s) {
      const int r = lane + 32 * s;
      if (s == s0) alpha = xc[s];
      const double v = r > k ? xc[s] : 0.0;
      if (s >= s0) (s & 1 ? p1 : p0) = fma(v, v, s & 1 ? p1 : p0);
    }
    alpha = __shfl_sync(0xffffffffu, alpha, k & 31);
    double part = p0 + p1;
    for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
    double tau = 0.0, beta = alpha, scal = 0.0;
    if (part != 0.0) {
      beta = -copysign(sqrt(fma(alpha, alpha, part)), alpha);
      tau = (beta - alpha) / beta;
      scal = 1.0 / (alpha - beta);
    }
#pragma unroll
    for (int s = 0; s < NR; ++s) {
      const int r = lane + 32 * s;
      double v = r == k ? 1.0 : 0.0;
      if (r == k) {
        xc[s] = beta;
      } else if (r > k && tau != 0.0) {
        xc[s] *= scal;
        v = xc[s];
      }
      for (int q = 0; q < C; ++q) st_cluster(cluster_map(&vb[k & 1][r], q), v);
#pragma unroll
      for (int c = 0; c < CW; ++c)
        if (kc == c) x[c][s] = xc[s];
    }
    if (lane < C) st_cluster(cluster_map(&tb[k & 1], lane), tau);
    if (lane == 0) tau_out[(size_t)box * K + k] = tau;
  };
  cluster_sync();  // every CTA runs (its shared memory may be written)
  if (g == 0) reflect(0);
  for (int k = 0; k < K; ++k) {
    cluster_sync();
    const double tk = tb[k & 1];
    double v[NR];
#pragma unroll
    for (int s = 0; s < NR; ++s) v[s] = vb[k & 1][lane + 32 * s];
    const int s0 = k >> 5;
    const bool next = k + 1 < K && (k + 1) % G == g;
    const int nc = next ? (k + 1) / G : -1;
    // column c's update with reflector k
    auto update = [&](int c) {
      double d0 = 0.0, d1 = 0.0;
#pragma unroll
      for (int s = 0; s < NR; ++s)
        if (s >= s0) (s & 1 ? d1 : d0) = fma(v[s], x[c][s], s & 1 ? d1 : d0);
      double d = d0 + d1;
      for (int o = 16; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
      d *= -tk;
#pragma unroll
      for (int s = 0; s < NR; ++s)
        if (s >= s0) x[c][s] = fma(d, v[s], x[c][s]);
    };
    if (next) {
      if (tk != 0.0) {
#pragma unroll
        for (int c = 0; c < CW; ++c)
          if (c == nc) update(c);
      }
      reflect(k + 1);
    }
    if (tk != 0.0) {
#pragma unroll
      for (int c = 0; c < CW; ++c)
        if (c != nc && g + G * c > k && g + G * c < K) update(c);
    }
  }
  cluster_sync();  // no CTA leaves while its buffers may be written
  double* Rb = Tm + (size_t)box * K * K;
  double* Vb = Vout + (size_t)box * D * K;
#pragma unroll
  for (int c = 0; c < CW; ++c) {
    const int j = g + G * c;
    if (j >= K) continue;
#pragma unroll
    for (int s = 0; s < NR; ++s) {
      const int r = lane + 32 * s;
      if (r < K) Rb[(size_t)r * K + j] = (r <= j) ? x[c][s] : 0.0;
      if (r < D) Vb[(size_t)j * D + r] = (r > j) ? x[c][s] : (r == j ? 1.0 : 0.0);
    }
  }
}
template <int CW>
static void launch_qr_cluster(int nb, int D, int K, int C, const double* Xin, double* Vout, double* tau, double* Tm,
                              cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nb * C));
  cfg.blockDim = dim3(512);
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = (unsigned)C;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  ++g_launches;
  note_launch(cudaLaunchKernelEx(&cfg, qr_cluster_kernel<CW>, D, K, C, Xin, Vout, tau, Tm));
}

template <typename T>
bool launch_qr_panel(int nb, int D, int K, const T* Xin, T* Vout, T* tau, T* Tm, T* gscr, cudaStream_t st, T* Tw) {
  if (nb == 0 || K == 0) return false;
  if (std::is_same<T, float>::value && D <= 256 && K <= 128) {
    int Kp = 8;
    while (Kp < K) Kp *= 2;
    const size_t nscr = std::max<size_t>(32 * 129, (size_t)Kp * Kp / 4);
    const size_t sm = sizeof(float) * (2 * 256 + 4 + Kp + nscr + (Tw ? (size_t)Kp * (Kp + 1) : 0));
    allow_smem((const void*)qr_reg_kernel<8>);
    ++g_launches;
    qr_reg_kernel<8><<<nb, 512, sm, st>>>(D, K, Kp, reinterpret_cast<const float*>(Xin),
                                          reinterpret_cast<float*>(Vout), reinterpret_cast<float*>(tau),
                                          reinterpret_cast<float*>(Tm), reinterpret_cast<float*>(Tw));
    return Tw != nullptr;
  }
  if constexpr (std::is_same<T, double>::value)
    if (D <= 256 && K <= 128) {
      // C = 2, 4 or 8 CTAs a box with 64 / C or fewer doubles of the panel a thread
      int C = 8;
      while (C > 2 && nb * C > num_sms()) C /= 2;
      const int cw = (K + 16 * C - 1) / (16 * C);
      auto go = cw <= 1 ? launch_qr_cluster<1> : cw <= 2 ? launch_qr_cluster<2> : launch_qr_cluster<4>;
      go(nb, D, K, C, Xin, Vout, tau, Tm, st);
      return false;
    }
  const size_t sm = sizeof(T) * (size_t)D * K;
  const int use = sm <= 200 * 1024;
  allow_smem((const void*)qr_panel_kernel<T>);
  ++g_launches;
  qr_panel_kernel<T><<<nb, 512, use ? sm : 0, st>>>(D, K, Xin, Vout, tau, Tm, gscr, use);
  return false;
}
template <typename T>
void launch_wy_tfactor(int nb, int K, const T* S, const T* tau, T* Tw, cudaStream_t st) {
  if (nb == 0 || K == 0) return;
  if (K <= 128) {
    int Kp = 8;
    while (Kp < K) Kp *= 2;
    const size_t sm = sizeof(T) * ((size_t)Kp * (Kp + 1) + (size_t)Kp * Kp / 4);
    allow_smem((const void*)wy_tinv_kernel<T>);
    ++g_launches;
    wy_tinv_kernel<T><<<nb, 256, sm, st>>>(K, Kp, S, tau, Tw);
    return;
  }
  size_t sm = sizeof(T) * ((size_t)K * K + K);
  const int use = sm <= 200 * 1024;
  if (!use) sm = sizeof(T) * (size_t)K;
  allow_smem((const void*)wy_tfactor_kernel<T>);
  ++g_launches;
  wy_tfactor_kernel<T><<<nb, 256, sm, st>>>(K, S, tau, Tw, use);
}
template <typename T>
void launch_perm_identity(int nb, int D, int K, T* U, cudaStream_t st) {
  const int64_t n = (int64_t)nb * D * D;
  if (n == 0) return;
  ++g_launches;
  perm_identity_kernel<T><<<(int)std::min<int64_t>((n + 255) / 256, 152 * 32), 256, 0, st>>>(nb, D, K, U);
}
#define H2_INST_QR(T)                                                                                         \
  template bool launch_qr_panel<T>(int, int, int, const T*, T*, T*, T*, T*, cudaStream_t, T*);                \
  template void launch_wy_tfactor<T>(int, int, const T*, const T*, T*, cudaStream_t);                          \
  template void launch_perm_identity<T>(int, int, int, T*, cudaStream_t);
H2_INST_QR(double)
H2_INST_QR(float)

// ------------------------------------------------------------------------
// a3: partial-pivot LU of Ahat_ii^RR (rows/cols 0..R of a D x D row-major
// block), LAPACK getf2 conventions (the first largest |pivot|; whole-row
// interchanges), in the factorization's precision T (FP64 for the FP64
// factorization, FP32 for the mixed-precision one).
//   luT  column-major R x R in T (L unit lower, U upper), piv LAPACK-style
//        (for T = double this is the lu array itself)
//   M    working copy: shared memory (ld = R + 1) when it fits, else luT
// A zero pivot records (level, box) in status[0..1]; the rest of that box's
// factorization is then undefined.
// ------------------------------------------------------------------------
// (TI: the type Ablk is stored in; the factorization runs in T)
template <typename T, typename TI = T>
__global__ void __launch_bounds__(256)
lu_factor_kernel(int D, int R, const TI* __restrict__ Ablk, const int32_t* __restrict__ diag_idx,
                 T* __restrict__ luT, int32_t* __restrict__ piv, int32_t* __restrict__ status, int level,
                 int use_smem) {
  extern __shared__ __align__(16) unsigned char sm_raw[];
  __shared__ int s_p;
  __shared__ T s_inv;
  const int box = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const TI* A = Ablk + (size_t)(diag_idx ? diag_idx[box] : box) * D * D;
  T* G = luT + (size_t)box * R * R;
  T* M = use_smem ? reinterpret_cast<T*>(sm_raw) : G;
  const int ld = use_smem ? R + 1 : R;
  int32_t* pv = piv + (size_t)box * R;
  for (int r = warp; r < R; r += 8)
    for (int c = lane; c < R; c += 32) M[c * ld + r] = static_cast<T>(A[(size_t)r * D + c]);
  __syncthreads();
  int bad = 0;
  for (int k = 0; k < R; ++k) {
    if (warp == 0) {
      T best = T(-1);
      int bi = k;
      for (int r = k + lane; r < R; r += 32) {
        T a = fabs(M[k * ld + r]);
        if (a > best) { best = a; bi = r; }
      }
      for (int o = 16; o; o >>= 1) {
        T ob = __shfl_down_sync(0xffffffffu, best, o);
        int oi = __shfl_down_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (lane == 0) {
        s_p = bi;
        pv[k] = bi;
        T d = M[k * ld + bi];
        s_inv = d != T(0) ? T(1) / d : T(0);
      }
    }
    __syncthreads();
    const int p = s_p;
    const T inv = s_inv;
    if (inv == T(0)) {
      bad = 1;
      break;
    }
    if (p != k)
      for (int c = tid; c < R; c += 256) {
        T t = M[c * ld + k];
        M[c * ld + k] = M[c * ld + p];
        M[c * ld + p] = t;
      }
    __syncthreads();
    for (int r = k + 1 + tid; r < R; r += 256) M[k * ld + r] *= inv;
    __syncthreads();
    for (int c = k + 1 + warp; c < R; c += 8) {
      const T f = M[c * ld + k];
      if (f != T(0))
        for (int r = k + 1 + lane; r < R; r += 32) M[c * ld + r] = fma(-M[k * ld + r], f, M[c * ld + r]);
    }
    __syncthreads();
  }
  if (bad) {
    if (tid == 0 && atomicCAS(status, 0, level + 1) == 0) status[1] = box;
    return;
  }
  if (use_smem)
    for (int c = warp; c < R; c += 8)
      for (int r = lane; r < R; r += 32) G[c * R + r] = M[c * ld + r];
}

// ------------------------------------------------------------------------
// a3 (cont.): Ainv = (P L U)^-1 = U^-1 L^-1 P^T in T, from the factors luT.
// Y starts as P^T (row r = e_perm[r]), then the unit-lower forward sweep and
// the upper backward sweep over all columns at once (row k is final when
// step k starts; the division by U(k,k) is applied to every row at the end).
// mode 2: factors and Y in shared memory; 1: factors only; 0: neither.
// ------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(256)
lu_inverse_kernel(int R, const T* __restrict__ luT, const int32_t* __restrict__ piv, T* __restrict__ Ainv, int mode) {
  extern __shared__ unsigned char sm_raw[];
  __shared__ int s_perm[1024];
  const int box = blockIdx.x, tid = threadIdx.x, tx = tid & 31, ty = tid >> 5;
  const T* src = luT + (size_t)box * R * R;
  const int ld = mode ? R + 1 : R;
  T* F = mode ? reinterpret_cast<T*>(sm_raw) : const_cast<T*>(src);
  T* Yg = Ainv + (size_t)box * R * R;
  T* Y = (mode == 2) ? F + R * (R + 1) : Yg;
  if (mode)
    for (int c = ty; c < R; c += 8)
      for (int r = tx; r < R; r += 32) F[c * ld + r] = src[c * R + r];
  if (tid == 0) {
    for (int r = 0; r < R; ++r) s_perm[r] = r;
    for (int k = 0; k < R; ++k) {
      int p = piv[(size_t)box * R + k];
      int t = s_perm[k];
      s_perm[k] = s_perm[p];
      s_perm[p] = t;
    }
  }
  __syncthreads();
  for (int r = ty; r < R; r += 8)
    for (int b = tx; b < R; b += 32) Y[r * R + b] = (b == s_perm[r]) ? T(1) : T(0);
  for (int k = 0; k < R - 1; ++k) {
    __syncthreads();
    for (int r = k + 1 + ty; r < R; r += 8) {
      const T l = F[k * ld + r];
      if (l != T(0))
        for (int b = tx; b < R; b += 32) Y[r * R + b] = fma(-l, Y[k * R + b], Y[r * R + b]);
    }
  }
  for (int k = R - 1; k > 0; --k) {
    __syncthreads();
    const T dk = T(1) / F[k * ld + k];
    for (int r = ty; r < k; r += 8) {
      const T u = F[k * ld + r] * dk;
      if (u != T(0))
        for (int b = tx; b < R; b += 32) Y[r * R + b] = fma(-u, Y[k * R + b], Y[r * R + b]);
    }
  }
  __syncthreads();
  for (int r = ty; r < R; r += 8) {
    const T dr = T(1) / F[r * ld + r];
    for (int b = tx; b < R; b += 32) Yg[r * R + b] = Y[r * R + b] * dr;
  }
}

// ------------------------------------------------------------------------
// a3 for R <= 256: (Ahat_ii^RR)^-1 by Gauss-Jordan elimination with partial
// pivoting (FP32 for the FP16/BF16 factorizations, FP64 for FP64 ones and for
// H2_OPT_RR_LU_FP64), or the LU factors in getf2's sense (LU), the block in
// registers.  A cluster of CL CTAs holds a box: CTA q columns 32 CPL q .., its
// warp w rows RPW w .. RPW w + RPW - 1, lane l columns CPL l .. CPL l + CPL - 1
// of them.  Step k:
//   (a) the lanes holding column k publish its entries f_r and each warp its
//       largest |f_r| among rows not yet used as pivots (the first on ties:
//       LAPACK's choice), in every CTA of the cluster; barrier (of the cluster);
//   (b) every warp finds the pivot row p; its warp publishes the row (each CTA
//       its columns), scaled so that column k becomes 1 / f_p; barrier (CTA);
//   (c) every other row takes a_r -= f_r (row p), its column k read as 0 (LU:
//       only rows not used yet, column k becomes the multiplier f_r / f_p).
// Rows are never moved: with pivot(k) the row of step k,
//   Ainv[k][pivot(j)] = a[pivot(k)][j];   LU: row k of the factors = a[pivot(k)].
// Buffers alternate with the step, so two barriers a step suffice.  A zero or
// non-finite pivot is seen by all threads at the same step, records (level,
// box) in status[0..1] and leaves the box's output undefined.  The pivot rows
// go to piv; pivot_sequence_kernel turns them into LAPACK's interchanges.
// Bound by the latency of a step (two barriers, a shuffle reduction, a
// reciprocal: 0.7 us at R = 128) in FP32 and by the FP64 pipe in FP64.  FP32:
// 128 x 128 in 92 us, 256 x 256 in 346 us; a panel form in which one warp ran 16
// steps at a time took 165 us, and 256 x 256 with four CTAs a box and the pivot
// column read from the owner 436 us.  FP64: 128 x 128 in 0.6 ms (inverse) and 0.8
// ms (LU), 256 x 256 in 2.0 and 2.1 ms; the LU of one 256 x 256 root by one CTA in
// global memory and its inverse took 20.6 ms.
// ------------------------------------------------------------------------
__device__ __forceinline__ float rcp_pivot(float v) { return __frcp_rn(v); }
__device__ __forceinline__ double rcp_pivot(double v) { return 1.0 / v; }

template <typename T, typename TI, typename TO, int NW, int RPW, int CPL, int CL, bool LU>
__global__ void __launch_bounds__(32 * NW, (sizeof(T) == 4 && RPW * CPL <= 32) ? 2 : 1)
    gj_rows_kernel(int D, int R, const TI* __restrict__ Ablk, const int32_t* __restrict__ diag_idx,
                   TO* __restrict__ out, int32_t* __restrict__ piv, int32_t* __restrict__ status, int level) {
  constexpr int NR = NW * RPW, NC = 32 * CPL;
  __shared__ __align__(16) T f[2][NR];
  __shared__ __align__(16) T prow[2][NC];
  __shared__ T cv[2][NW];
  __shared__ int cr[2][NW];
  __shared__ int pr_of[NR], step_of[NR];  // pivot(k), and its inverse
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int q = CL > 1 ? (int)cluster_rank() : 0, box = blockIdx.x / CL;
  const int r0 = RPW * warp, c0 = NC * q + CPL * lane;
  const TI* A = Ablk + (size_t)(diag_idx ? diag_idx[box] : box) * D * D;
  T a[RPW][CPL];
  unsigned used = 0;
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    if (r0 + i >= R) used |= 1u << i;
#pragma unroll
    for (int j = 0; j < CPL; ++j)
      a[i][j] = (r0 + i < R && c0 + j < R) ? static_cast<T>(A[(size_t)(r0 + i) * D + c0 + j]) : T(0);
  }
  if constexpr (CL > 1) cluster_sync();  // every CTA runs
  bool ok = true;
  for (int kc = 0; kc * CPL < R && ok; ++kc) {
#pragma unroll
    for (int jk = 0; jk < CPL; ++jk) {
      const int k = kc * CPL + jk, buf = k & 1;
      if (k >= R || !ok) break;
      if (kc / 32 == q) {
        if (lane == (kc & 31)) {
          T bv = T(0), best = T(-1);
          int br = -1;
#pragma unroll
          for (int i = 0; i < RPW; ++i) {
            const T v = a[i][jk];
            if (!((used >> i) & 1u) && fabs(v) > best) best = fabs(v), bv = v, br = r0 + i;
            f[buf][r0 + i] = v;
            if constexpr (!LU) a[i][jk] = T(0);  // (column k is read as 0 by the update)
          }
          cv[buf][warp] = bv, cr[buf][warp] = br;
        }
        if constexpr (CL > 1) {
          // to the other CTAs, an entry per lane
          __syncwarp();
          if (lane < RPW) {
            const T v = f[buf][r0 + lane];
#pragma unroll
            for (int o = 1; o < CL; ++o) st_cluster(cluster_map(&f[buf][r0 + lane], (q + o) % CL), v);
          } else if (lane < RPW + CL - 1) {
            const int cta = (q + 1 + lane - RPW) % CL;
            st_cluster(cluster_map(&cv[buf][warp], cta), cv[buf][warp]);
            st_cluster(cluster_map(&cr[buf][warp], cta), cr[buf][warp]);
          }
        }
      }
      if constexpr (CL > 1) cluster_sync();
      else __syncthreads();
      // the pivot: the candidate of largest size, the lowest row on ties
      const int pc = lane < NW ? cr[buf][lane] : -1;
      const T vc = lane < NW ? cv[buf][lane] : T(0);
      int src;
      if constexpr (sizeof(T) == 4) {
        // (sizes order as their bits; NaN candidates are never published)
        const unsigned key = pc >= 0 ? __float_as_uint(fabsf(vc)) : 0u;
        const unsigned top = __reduce_max_sync(0xffffffffu, key);
        const unsigned at = __ballot_sync(0xffffffffu, pc >= 0 && key == top);
        src = at ? __ffs(at) - 1 : 0;  // (warps are in row order)
      } else {
        long long key = pc >= 0 ? __double_as_longlong(fabs(vc)) : -1;
        src = lane;
#pragma unroll
        for (int o = NW / 2; o > 0; o >>= 1) {
          const long long ok2 = __shfl_xor_sync(0xffffffffu, key, o);
          const int os = __shfl_xor_sync(0xffffffffu, src, o);
          if (ok2 > key || (ok2 == key && os < src)) key = ok2, src = os;
        }
        src = __shfl_sync(0xffffffffu, src, 0);
      }
      const int p = __shfl_sync(0xffffffffu, pc, src);
      const T pv = __shfl_sync(0xffffffffu, vc, src);
      if (p < 0 || pv == T(0) || !isfinite(pv)) {
        ok = false;
        break;
      }
      const T inv = rcp_pivot(pv);
      const int ip = p - r0;  // in 0 .. RPW - 1 in its warp
      if (ip >= 0 && ip < RPW) {
#pragma unroll
        for (int j = 0; j < CPL; ++j) {
          T v = a[0][j];
#pragma unroll
          for (int i = 1; i < RPW; ++i) v = i == ip ? a[i][j] : v;
          if constexpr (!LU) v = (j == jk && c0 + j == k) ? inv : v * inv;
          prow[buf][CPL * lane + j] = v;
        }
        used |= 1u << ip;
        if (lane == 0) pr_of[k] = p, step_of[p] = k;
      }
      __syncthreads();
      T pr[CPL];
#pragma unroll
      for (int j = 0; j < CPL; ++j) pr[j] = prow[buf][CPL * lane + j];
      if constexpr (!LU) {
        T fr[RPW];
#pragma unroll
        for (int i = 0; i < RPW; ++i) fr[i] = f[buf][r0 + i];
        if (ip >= 0 && ip < RPW) {
#pragma unroll
          for (int i = 0; i < RPW; ++i)
#pragma unroll
            for (int j = 0; j < CPL; ++j) a[i][j] = i == ip ? pr[j] : fma(-fr[i], pr[j], a[i][j]);
        } else {
#pragma unroll
          for (int i = 0; i < RPW; ++i)
#pragma unroll
            for (int j = 0; j < CPL; ++j) a[i][j] = fma(-fr[i], pr[j], a[i][j]);
        }
      } else {
#pragma unroll
        for (int i = 0; i < RPW; ++i) {
          if ((used >> i) & 1u) continue;
          const T l = f[buf][r0 + i] * inv;
#pragma unroll
          for (int j = 0; j < CPL; ++j) {
            const int c = c0 + j;
            if (c > k) a[i][j] = fma(-l, pr[j], a[i][j]);
            else if (j == jk && c == k) a[i][j] = l;
          }
        }
      }
    }
  }
  if constexpr (CL > 1) cluster_sync();  // no CTA leaves while another may still write to it
  if (!ok) {
    if (q == 0) {
      for (int k = tid; k < R; k += blockDim.x) piv[(size_t)box * R + k] = k;  // (a valid sequence)
      if (tid == 0 && atomicCAS(status, 0, level + 1) == 0) status[1] = box;
    }
    return;
  }
  __syncthreads();
  TO* ob = out + (size_t)box * R * R;
#pragma unroll
  for (int i = 0; i < RPW; ++i) {
    if (r0 + i >= R) continue;
    const int sr = step_of[r0 + i];
#pragma unroll
    for (int j = 0; j < CPL; ++j)
      if (c0 + j < R) {
        if constexpr (LU) ob[(size_t)(c0 + j) * R + sr] = static_cast<TO>(a[i][j]);
        else ob[(size_t)sr * R + pr_of[c0 + j]] = static_cast<TO>(a[i][j]);
      }
  }
  if (q == 0)
    for (int k = tid; k < R; k += blockDim.x) piv[(size_t)box * R + k] = pr_of[k];
}

// LAPACK's interchange sequence of the pivot rows in piv, in place (R <= 256):
// one thread per box, beside the factorization's chain.
__global__ void __launch_bounds__(32) pivot_sequence_kernel(int R, int32_t* __restrict__ piv) {
  __shared__ int pos[256], rowat[256], pr[256];
  int32_t* pv = piv + (size_t)blockIdx.x * R;
  for (int r = threadIdx.x; r < R; r += 32) pos[r] = r, rowat[r] = r, pr[r] = pv[r];
  __syncwarp();
  if (threadIdx.x == 0)
    for (int k = 0; k < R; ++k) {
      const int r = pr[k], at = pos[r], rk = rowat[k];
      pv[k] = at;
      rowat[k] = r, rowat[at] = rk;
      pos[r] = k, pos[rk] = at;
    }
}
void launch_pivot_sequence(int nb, int R, int32_t* piv, cudaStream_t st) {
  if (nb == 0 || R == 0) return;
  ++g_launches;
  pivot_sequence_kernel<<<nb, 32, 0, st>>>(R, piv);
}

template <typename T, typename TI, typename TO, int NW, int RPW, int CPL, int CL, bool LU>
static void launch_gj_rows_t(int nb, int D, int R, const TI* A, const int32_t* diag_idx, TO* out, int32_t* piv,
                             int32_t* status, int level, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nb * CL));
  cfg.blockDim = dim3(32 * NW);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = CL;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = CL > 1 ? 1 : 0;
  ++g_launches;
  note_launch(cudaLaunchKernelEx(&cfg, gj_rows_kernel<T, TI, TO, NW, RPW, CPL, CL, LU>, D, R, A, diag_idx, out, piv,
                                 status, level));
}
// false for R > 256.  FP64 spreads a box over more CTAs (its time is the FP64
// pipe's); few rows take fewer warps (a barrier's cost goes with them).
template <typename T, typename TI, typename TO, bool LU>
static bool launch_gj_rows(int nb, int D, int R, const TI* A, const int32_t* di, TO* out, int32_t* piv,
                           int32_t* status, int level, cudaStream_t st) {
  if (R > 256) return false;
  if constexpr (sizeof(T) == 4) {
    if (R <= 32) launch_gj_rows_t<T, TI, TO, 4, 8, 1, 1, LU>(nb, D, R, A, di, out, piv, status, level, st);
    else if (R <= 64) launch_gj_rows_t<T, TI, TO, 8, 8, 2, 1, LU>(nb, D, R, A, di, out, piv, status, level, st);
    else if (R <= 128) launch_gj_rows_t<T, TI, TO, 16, 8, 4, 1, LU>(nb, D, R, A, di, out, piv, status, level, st);
    else launch_gj_rows_t<T, TI, TO, 16, 16, 4, 2, LU>(nb, D, R, A, di, out, piv, status, level, st);
  } else {
    if (R <= 32) launch_gj_rows_t<T, TI, TO, 4, 8, 1, 1, LU>(nb, D, R, A, di, out, piv, status, level, st);
    else if (R <= 64) launch_gj_rows_t<T, TI, TO, 8, 8, 1, 2, LU>(nb, D, R, A, di, out, piv, status, level, st);
    else if (R <= 128) launch_gj_rows_t<T, TI, TO, 16, 8, 1, 4, LU>(nb, D, R, A, di, out, piv, status, level, st);
    else launch_gj_rows_t<T, TI, TO, 16, 16, 1, 8, LU>(nb, D, R, A, di, out, piv, status, level, st);
  }
  return true;
}

// ------------------------------------------------------------------------
// The same in-place elimination in FP32 for 256 < R <= 512: the columns are
// split over a cluster of CL CTAs (thread-block cluster, distributed shared
// memory).  CTA q of a box holds the columns [q W, (q + 1) W), W = Rp / CL,
// as TR x TC register tiles, thread t at tile (t % G, q W / TC + t / G).
// Step k: the CTA owning column k picks the pivot row among the unused rows
// and publishes (p, a_pk) and column k in its shared memory, in the buffer
// of the step's parity; one cluster barrier; every CTA reads them from the
// owner, scales its part of row p and eliminates column k from its other
// rows.  The owner rewrites a buffer two steps later, after every CTA has
// passed the next barrier, so one cluster barrier per step suffices.  A
// failed pivot is seen by every CTA at the same step; all of them leave
// after one more cluster barrier, so that no CTA exits while another may
// still read its shared memory.
// ------------------------------------------------------------------------
template <typename T>
struct __align__(16) GjcShared {
  T fcol[2][512];  // the owner's column k, by step parity
  T fl[512];       // this CTA's copy of it
  T P[512];        // the scaled pivot row (this CTA's columns)
  T pvs[2];        // a_pk, by step parity
  int ps[2];       // p, by step parity
  int prow[512], pinv[512], rowat[512];
};

__host__ __device__ inline int gj_group(int ntr) {
  int g = 1;
  while (g < ntr) g <<= 1;
  return g;
}

template <typename T, int TR, int TC, int J>
__device__ __forceinline__ bool gjc_step(GjcShared<T>& sh, T (&a)[TR][TC], unsigned& used, int kc, int oq, int kcl,
                                         int q, int G, int Rp, bool has, int tr, int tc, int tcl, int r0, int c0) {
  const int t = threadIdx.x, k = kc * TC + J, b = k & 1;
  if (q == oq) {
    // (a) the owner warp of column k: the first largest |a_rk| over unused rows
    if ((t >> 5) == ((kcl * G) >> 5)) {
      T best = T(-1), sv = T(0);
      int bi = -1;
      if (has && tcl == kcl) {
#pragma unroll
        for (int i = 0; i < TR; ++i) {
          const T v = fabs(a[i][J]);
          if (!((used >> i) & 1u) && v > best) best = v, sv = a[i][J], bi = r0 + i;
        }
      }
      for (int o = G >> 1; o > 0; o >>= 1) {
        const T ob = __shfl_xor_sync(0xffffffffu, best, o), os = __shfl_xor_sync(0xffffffffu, sv, o);
        const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
        if (ob > best || (ob == best && oi >= 0 && (bi < 0 || oi < bi))) best = ob, sv = os, bi = oi;
      }
      if (tcl == kcl && tr == 0) sh.ps[b] = bi, sh.pvs[b] = sv;
    }
    if (has && tcl == kcl) {
#pragma unroll
      for (int i = 0; i < TR; ++i) sh.fcol[b][r0 + i] = a[i][J];
    }
  }
  cluster_sync();
  const int p = ld_cluster(cluster_map(&sh.ps[b], (uint32_t)oq), int());
  const T pv = ld_cluster(cluster_map(&sh.pvs[b], (uint32_t)oq), T());
  if (p < 0 || pv == T(0) || !isfinite(pv)) return false;
  const T inv = rcp_pivot(pv);
  if (t == 0) sh.prow[k] = p;
  // (b) column k from the owner; this CTA's part of the scaled pivot row
  {
    constexpr int PER = 16 / (int)sizeof(T);
    const uint32_t src = cluster_map(&sh.fcol[b][0], (uint32_t)oq);
    for (int e = t; e < Rp / PER; e += blockDim.x)
      *reinterpret_cast<uint4*>(&sh.fl[e * PER]) = ld_cluster_v4(src + 16u * (uint32_t)e);
  }
  if (has && tr == p / TR) {
#pragma unroll
    for (int i = 0; i < TR; ++i)
      if (r0 + i == p) {
#pragma unroll
        for (int jj = 0; jj < TC; ++jj) {
          const T v = ((jj == J && c0 + jj == k) ? T(1) : a[i][jj]) * inv;
          a[i][jj] = v;
          sh.P[c0 + jj] = v;
        }
        used |= 1u << i;
      }
  }
  __syncthreads();
  // (c) eliminate column k from every other row
  if (has) {
    T pr[TC];
#pragma unroll
    for (int jj = 0; jj < TC; ++jj) pr[jj] = sh.P[c0 + jj];
    const bool own = (tc == kc);
#pragma unroll
    for (int i = 0; i < TR; ++i) {
      const T f = (r0 + i == p) ? T(0) : sh.fl[r0 + i];
      if (own && r0 + i != p) a[i][J] = T(0);
#pragma unroll
      for (int jj = 0; jj < TC; ++jj) a[i][jj] = fma(-f, pr[jj], a[i][jj]);
    }
  }
  return true;
}

template <typename T, int TR, int TC, int J>
__device__ __forceinline__ void gjc_steps(bool& ok, GjcShared<T>& sh, T (&a)[TR][TC], unsigned& used, int kc, int oq,
                                          int kcl, int q, int G, int Rp, int left, bool has, int tr, int tc, int tcl,
                                          int r0, int c0) {
  if constexpr (J < TC) {
    if (ok && left > J) ok = gjc_step<T, TR, TC, J>(sh, a, used, kc, oq, kcl, q, G, Rp, has, tr, tc, tcl, r0, c0);
    gjc_steps<T, TR, TC, J + 1>(ok, sh, a, used, kc, oq, kcl, q, G, Rp, left, has, tr, tc, tcl, r0, c0);
  }
}

template <typename T, int TR, int TC, int CL, int NT>
__global__ void __cluster_dims__(CL, 1, 1) __launch_bounds__(NT, 1)
    gj_cluster_kernel(int D, int R, int Rp, const float* __restrict__ Ablk, const int32_t* __restrict__ diag_idx,
                      float* __restrict__ Ainv, int32_t* __restrict__ piv, int32_t* __restrict__ status, int level) {
  __shared__ GjcShared<T> sh;
  const int q = (int)cluster_rank();
  const int box = blockIdx.x / CL, t = threadIdx.x;
  const int W = Rp / CL, ntr = Rp / TR, ntcl = W / TC, G = gj_group(ntr);
  const int tr = t % G, tcl = t / G;
  const bool has = tr < ntr && tcl < ntcl;
  const int tc = q * ntcl + tcl;
  const int r0 = tr * TR, c0 = tc * TC;
  const float* A = Ablk + (size_t)(diag_idx ? diag_idx[box] : box) * D * D;
  T a[TR][TC];
  unsigned used = 0;
#pragma unroll
  for (int i = 0; i < TR; ++i) {
    const int r = r0 + i;
    if (!has || r >= R) used |= 1u << i;
#pragma unroll
    for (int j = 0; j < TC; ++j) {
      const int c = c0 + j;
      a[i][j] = (has && r < R && c < R) ? static_cast<T>(A[(size_t)r * D + c]) : T(0);
    }
  }
  bool ok = true;
  const int nkc = (R + TC - 1) / TC;
  for (int kc = 0; kc < nkc && ok; ++kc) {
    const int oq = kc / ntcl;
    gjc_steps<T, TR, TC, 0>(ok, sh, a, used, kc, oq, kc - oq * ntcl, q, G, Rp, R - kc * TC, has, tr, tc, tcl, r0,
                            c0);
  }
  cluster_sync();
  if (!ok) {
    if (q == 0 && t == 0 && atomicCAS(status, 0, level + 1) == 0) status[1] = box;
    return;
  }
  // unscramble this CTA's columns: Ainv[k][prow[j]] = a[prow[k]][j]
  for (int k = t; k < R; k += blockDim.x) sh.pinv[sh.prow[k]] = k;
  __syncthreads();
  if (has) {
    float* out = Ainv + (size_t)box * R * R;
#pragma unroll
    for (int i = 0; i < TR; ++i) {
      const int r = r0 + i;
      if (r >= R) continue;
      const size_t row = (size_t)sh.pinv[r] * R;
#pragma unroll
      for (int jj = 0; jj < TC; ++jj)
        if (c0 + jj < R) out[row + sh.prow[c0 + jj]] = static_cast<float>(a[i][jj]);
    }
  }
  if (q == 0) {
    // LAPACK-style interchange sequence of the same pivots
    __syncthreads();
    if (t == 0) {
      int* pos = sh.pinv;
      for (int r = 0; r < R; ++r) pos[r] = r, sh.rowat[r] = r;
      int32_t* pv_out = piv + (size_t)box * R;
      for (int k = 0; k < R; ++k) {
        const int r = sh.prow[k], qq = pos[r], rk = sh.rowat[k];
        pv_out[k] = qq;
        sh.rowat[k] = r, sh.rowat[qq] = rk;
        pos[r] = k, pos[rk] = qq;
      }
    }
  }
}

// Inverses of nb blocks by the cluster kernel: FP32 elimination for
// 256 < R <= 512.  False: R not covered.
static bool launch_gj_cluster(int nb, int D, int R, const float* Ablk, const int32_t* diag_idx, float* Ainv,
                              int32_t* piv, int32_t* status, int level, cudaStream_t st) {
  if (R <= 256 || R > 512) return false;
  ++g_launches;
  gj_cluster_kernel<float, 16, 4, 8, 512><<<nb * 8, 512, 0, st>>>(D, R, (R + 31) / 32 * 32, Ablk, diag_idx, Ainv, piv,
                                                                   status, level);
  return true;
}

template <typename T>
bool launch_lu_inverse(int nb, int D, int R, const T* Ablk, const int32_t* diag_idx, double* lu, T* luT,
                       int32_t* piv, T* Ainv, int32_t* status, int level, cudaStream_t st, cudaStream_t side) {
  if (nb == 0 || R == 0) return false;
  (void)lu;  // for T = double, luT is the lu array
  if constexpr (std::is_same<T, float>::value) {
    // mixed precision: the inverse directly, no LU factors kept
    if (launch_gj_rows<float, float, float, false>(nb, D, R, Ablk, diag_idx, Ainv, piv, status, level, st)) return true;
    if (launch_gj_cluster(nb, D, R, Ablk, diag_idx, Ainv, piv, status, level, st)) return false;
  } else {
    // the inverse on the chain, the factors (kept for inspection) beside it;
    // both pick the same pivots
    if (launch_gj_rows<double, double, double, true>(nb, D, R, Ablk, diag_idx, luT, piv, status, level, side)) {
      launch_pivot_sequence(nb, R, piv, side);
      launch_gj_rows<double, double, double, false>(nb, D, R, Ablk, diag_idx, Ainv, piv + (size_t)nb * R, status, level,
                                                    st);
      return false;
    }
  }
  const size_t cap = 220 * 1024;
  size_t sm1 = sizeof(T) * (size_t)R * (R + 1);
  int use = sm1 <= cap;
  allow_smem((const void*)lu_factor_kernel<T>);
  ++g_launches;
  lu_factor_kernel<T><<<nb, 256, use ? sm1 : 0, st>>>(D, R, Ablk, diag_idx, luT, piv, status, level, use);
  if (R > 1024) return false;  // the permutation table holds 1024 rows; larger blocks are rejected by the caller
  size_t f = sizeof(T) * (size_t)R * (R + 1), y = sizeof(T) * (size_t)R * R;
  int mode = (f + y <= cap) ? 2 : (f <= cap ? 1 : 0);
  size_t sm = mode == 2 ? f + y : (mode == 1 ? f : 0);
  allow_smem((const void*)lu_inverse_kernel<T>);
  ++g_launches;
  lu_inverse_kernel<T><<<nb, 256, sm, st>>>(R, luT, piv, Ainv, mode);
  return false;
}
bool launch_lu_inverse_f64_for_f32(int nb, int D, int R, const float* Ablk, const int32_t* diag_idx, double* lu,
                                   double* inv, int32_t* piv, float* Ainv, int32_t* status, int level,
                                   cudaStream_t st) {
  if (nb == 0 || R == 0 || R > 1024) return false;
  if (launch_gj_rows<double, float, float, false>(nb, D, R, Ablk, diag_idx, Ainv, piv, status, level, st)) return true;
  const size_t cap = 220 * 1024;
  const size_t sm1 = sizeof(double) * (size_t)R * (R + 1);
  const int use = sm1 <= cap;
  allow_smem((const void*)lu_factor_kernel<double, float>);
  ++g_launches;
  lu_factor_kernel<double, float><<<nb, 256, use ? sm1 : 0, st>>>(D, R, Ablk, diag_idx, lu, piv, status, level, use);
  const size_t f = sizeof(double) * (size_t)R * (R + 1), y = sizeof(double) * (size_t)R * R;
  const int mode = (f + y <= cap) ? 2 : (f <= cap ? 1 : 0);
  const size_t sm = mode == 2 ? f + y : (mode == 1 ? f : 0);
  allow_smem((const void*)lu_inverse_kernel<double>);
  ++g_launches;
  lu_inverse_kernel<double><<<nb, 256, sm, st>>>(R, lu, piv, inv, mode);
  launch_convert<double, float>(inv, Ainv, (int64_t)nb * R * R, st);
  return false;
}

template bool launch_lu_inverse<double>(int, int, int, const double*, const int32_t*, double*, double*, int32_t*,
                                        double*, int32_t*, int, cudaStream_t, cudaStream_t);
template bool launch_lu_inverse<float>(int, int, int, const float*, const int32_t*, double*, float*, int32_t*,
                                       float*, int32_t*, int, cudaStream_t, cudaStream_t);

// ------------------------------------------------------------------------
// a6: merge.  Child pair q of level l (near: its SS part of Ahat; far: Shat)
// goes to quadrant (i%2, j%2) of parent near block dst[q] (D_{l-1} = 2K).
// ------------------------------------------------------------------------
template <typename T>
__global__ void merge_kernel(int D, int K, int64_t NP, const T* __restrict__ Ahat,
                             const int32_t* __restrict__ ni, const int32_t* __restrict__ nj,
                             const int32_t* __restrict__ ndst, int64_t FP, const T* __restrict__ Shat,
                             const int32_t* __restrict__ fi, const int32_t* __restrict__ fj,
                             const int32_t* __restrict__ fdst, T* __restrict__ Apar) {
  const int R = D - K, Dp = 2 * K;
  const int64_t q = blockIdx.y + (int64_t)blockIdx.z * gridDim.y;
  if (q >= NP + FP) return;
  const bool nr = q < NP;
  const int64_t qq = nr ? q : q - NP;
  const int i = nr ? ni[qq] : fi[qq], j = nr ? nj[qq] : fj[qq];
  const int64_t dst = nr ? ndst[qq] : fdst[qq];
  T* out = Apar + dst * Dp * Dp + (int64_t)(i & 1) * K * Dp + (j & 1) * K;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < K * K; e += gridDim.x * blockDim.x) {
    int a = e / K, b = e - a * K;
    T v = nr ? Ahat[qq * D * D + (int64_t)(R + a) * D + R + b] : Shat[qq * K * K + e];
    out[(int64_t)a * Dp + b] = v;
  }
}

template <typename T>
void launch_merge(int D, int K, int64_t NP, const T* Ahat, const int32_t* ni, const int32_t* nj,
                  const int32_t* ndst, int64_t FP, const T* Shat, const int32_t* fi, const int32_t* fj,
                  const int32_t* fdst, T* Apar, cudaStream_t st) {
  int64_t n = NP + FP;
  if (n == 0 || K == 0) return;
  int gx = std::min(64, (K * K + 255) / 256);
  int64_t gy = std::min<int64_t>(n, 65535), gz = (n + gy - 1) / gy;
  ++g_launches;
  merge_kernel<T><<<dim3(gx, (unsigned)gy, (unsigned)gz), 256, 0, st>>>(D, K, NP, Ahat, ni, nj, ndst, FP, Shat, fi,
                                                                         fj, fdst, Apar);
}
template void launch_merge<double>(int, int, int64_t, const double*, const int32_t*, const int32_t*,
                                   const int32_t*, int64_t, const double*, const int32_t*, const int32_t*,
                                   const int32_t*, double*, cudaStream_t);
template void launch_merge<float>(int, int, int64_t, const float*, const int32_t*, const int32_t*, const int32_t*,
                                  int64_t, const float*, const int32_t*, const int32_t*, const int32_t*, float*,
                                  cudaStream_t);

}  // namespace h2
