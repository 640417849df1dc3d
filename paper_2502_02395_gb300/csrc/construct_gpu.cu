// Algorithm 1 on the GPU at a level rank K laid out beforehand (by the rank
// predictor, or the rank cap): randomized interpolative decompositions of
// every box of a level, batched, in FP64.
//
// For box i with points B_i (n_i <= 256), far samples S_F(i) and close boxes
// j != i with close samples S_C(j) (<= 64 points each), the composite matrix
// of Algorithm 1 is M_i = [G(B_i, S_F) | G(B_i, S_C(j)) G(S_C(j), S_C(j))^-1 ...].
// Its sketch Y_i = M_i Omega (n_i x m) takes Omega(p, t) = +-1 as a function
// of the sample point p (splitmix64), so the close part factors as
// G(B_i, S_C(j)) W_j with W_j = G(S_C(j), S_C(j))^-1 Omega(S_C(j)), computed
// once per box j and shared by every box that has j close:
//   cc_weights_kernel  per box j: W_j by Gauss-Jordan on [G(S_C, S_C) | Omega]
//                      (partial pivoting); cc_sweeps_kernel: by `gs`
//                      Gauss-Seidel sweeps from W = 0 (the shortcut of Section
//                      3.5 for the inverse of the close part in Algorithm 1)
//   sketch_kernel      per box, half of its rows and split of its samples:
//                      Y_i = G(B_i, S_F) Omega(S_F) + sum_j G(B_i, S_C(j))
//                      W_j, kernel entries evaluated in 32-sample chunks into
//                      shared memory
//   pivqr_id_kernel    per box, a thread-block cluster: column-pivoted
//                      Householder QR of the first ms columns of Y_i,
//                      transposed (ms x n_i; the rows of Y_i are its columns),
//                      in registers; the first K pivots are the skeleton,
//                      X_i = P [I; (R11^-1 R12)^T]; also the pivot ratio
//                      |R_K+1,K+1| / |R_11| and the interpolation error on the
//                      q probe columns.
#include <algorithm>
#include <type_traits>

#include "h2_internal.h"
#include "kernels.h"
#include "ptx_util.h"
#include "warp_sums.h"

namespace h2 {
namespace {

constexpr int GC_CHUNK = 32;   // sample points per evaluated chunk
constexpr int GC_ROWS = 128;   // box rows per sketch CTA
constexpr int GC_MAXM = 160;   // sketch + probe columns
constexpr int GC_MAXS = 64;    // close samples per box

__device__ __forceinline__ uint64_t splitmix64_d(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}
// Omega(p, t) in {-1, +1}
__device__ __forceinline__ double omega(uint64_t seed, int64_t p, int t) {
  const uint64_t bits = splitmix64_d(seed ^ ((uint64_t)p * 0x100000001B3ull + (uint64_t)(t >> 6)));
  return ((bits >> (t & 63)) & 1ull) ? 1.0 : -1.0;
}

// W_j (s x m, row-major at W + cptr[j] * m) for every box j, exact solve:
// Gauss-Jordan with partial pivoting on [G(S_C, S_C) | Omega], the augmented
// matrix in registers.  256 threads as 16 x 16: thread (ty, tx) owns rows
// ty + 16 p and columns tx + 16 b, so a step costs one FP64 multiply-add per
// entry, two barriers and one row and one column through shared memory; rows
// are not swapped (a pivot row is marked and W row k is taken from the row
// that was step k's pivot), and the finished 16-column blocks of G are
// skipped.  Bound by the FP64 pipe (about 1.75 multiply-adds per clock and
// SM): the columns of Omega are split over gridDim.y CTAs (each repeats the
// elimination of G) while a level has fewer boxes than SMs.  NB: 16-column
// blocks of Omega per CTA.
template <int NB>
__global__ void __launch_bounds__(256) cc_weights_kernel(KernelFn G, const double* __restrict__ pts,
                                                         const int64_t* __restrict__ cptr,
                                                         const int64_t* __restrict__ cidx, int m, uint64_t seed,
                                                         double* __restrict__ W) {
  constexpr int GB = GC_MAXS / 16;  // 16-row / 16-column blocks of G
  __shared__ double colb[2][GC_MAXS];
  __shared__ double rowb[2][16 * (GB + NB)];
  __shared__ int ord[GC_MAXS];  // step whose pivot a row was
  const int j = blockIdx.x, tid = threadIdx.x, ty = tid >> 4, tx = tid & 15, lane = tid & 31;
  const int64_t c0 = cptr[j];
  const int s = (int)(cptr[j + 1] - c0);
  if (s == 0) return;
  const int t0 = blockIdx.y * NB * 16;  // first column of Omega of this CTA
  double a[GB][GB + NB];
#pragma unroll
  for (int p = 0; p < GB; ++p)
#pragma unroll
    for (int b = 0; b < GB + NB; ++b) {
      const int r = ty + 16 * p, c = tx + 16 * (b < GB ? b : b - GB);
      a[p][b] = 0.0;
      if (r < s) {
        if (b < GB) {
          if (c < s) a[p][b] = G.entry(pts, cidx[c0 + r], cidx[c0 + c], r == c);
        } else if (t0 + c < m) {
          a[p][b] = omega(seed, cidx[c0 + r], t0 + c);
        }
      }
    }
  if (tid < GC_MAXS) ord[tid] = -1;
  unsigned long long used = 0;  // rows that have been pivots (the same in every thread)
  // (a function of the column block, so that a's indices are constants)
  auto block_steps = [&](auto kb_c) {
    constexpr int kb = decltype(kb_c)::value;
    for (int kk = 0; kk < 16; ++kk) {
      const int k = 16 * kb + kk, buf = k & 1;
      if (k >= s) return;
      if (tx == kk)
#pragma unroll
        for (int p = 0; p < GB; ++p) colb[buf][ty + 16 * p] = a[p][kb];
      __syncthreads();
      // the largest |entry| among the rows that were no pivot yet (first on
      // ties), found by every warp; non-negative doubles order as integers
      long long best = -1;
      int bp = 0;
      for (int r = lane; r < s; r += 32)
        if (!((used >> r) & 1ull)) {
          const long long v = __double_as_longlong(fabs(colb[buf][r]));
          if (v > best) best = v, bp = r;
        }
      for (int o = 16; o; o >>= 1) {
        const long long ov = __shfl_xor_sync(0xffffffffu, best, o);
        const int op = __shfl_xor_sync(0xffffffffu, bp, o);
        if (ov > best || (ov == best && op < bp)) best = ov, bp = op;
      }
      used |= 1ull << bp;
      if (ty == (bp & 15)) {
        const double d = colb[buf][bp];
        const double inv = d != 0.0 ? 1.0 / d : 0.0;
        const int pb = bp >> 4;
#pragma unroll
        for (int b = kb; b < GB + NB; ++b) {
          double v = a[0][b];
#pragma unroll
          for (int p = 1; p < GB; ++p) v = pb == p ? a[p][b] : v;
          rowb[buf][tx + 16 * b] = v * inv;
        }
        if (tx == 0) ord[bp] = k;
      }
      __syncthreads();
      double f[GB];
#pragma unroll
      for (int p = 0; p < GB; ++p) f[p] = colb[buf][ty + 16 * p];
#pragma unroll
      for (int b = kb; b < GB + NB; ++b) {
        const double x = rowb[buf][tx + 16 * b];
#pragma unroll
        for (int p = 0; p < GB; ++p) a[p][b] = (ty + 16 * p == bp) ? x : fma(-f[p], x, a[p][b]);
      }
    }
  };
  static_assert(GB == 4, "four column blocks");
  block_steps(std::integral_constant<int, 0>());
  block_steps(std::integral_constant<int, 1>());
  block_steps(std::integral_constant<int, 2>());
  block_steps(std::integral_constant<int, 3>());
  __syncthreads();
  double* Wj = W + c0 * m;
#pragma unroll
  for (int p = 0; p < GB; ++p) {
    const int r = ty + 16 * p;
    if (r >= s || ord[r] < 0) continue;
#pragma unroll
    for (int b = 0; b < NB; ++b) {
      const int t = t0 + tx + 16 * b;
      if (t < m) Wj[(int64_t)ord[r] * m + t] = a[p][GB + b];
    }
  }
}

// The Gauss-Seidel shortcut: W = 0, then sweeps r = 0 .. s-1 of
// W[r] = (Omega[r] - sum_{c != r} A[r][c] W[c]) / A[r][r]; thread t owns column t
__global__ void __launch_bounds__(256) cc_sweeps_kernel(KernelFn G, const double* __restrict__ pts,
                                                        const int64_t* __restrict__ cptr,
                                                        const int64_t* __restrict__ cidx, int m, uint64_t seed,
                                                        int gs, double* __restrict__ W) {
  extern __shared__ __align__(16) double smd[];
  const int j = blockIdx.x, tid = threadIdx.x;
  const int64_t c0 = cptr[j];
  const int s = (int)(cptr[j + 1] - c0);
  if (s == 0) return;
  const int ld = s + m;  // row [A_cc | Omega]
  double* Aug = smd;     // s x ld
  for (int e = tid; e < s * ld; e += blockDim.x) {
    const int r = e / ld, c = e - r * ld;
    Aug[e] = (c < s) ? G.entry(pts, cidx[c0 + r], cidx[c0 + c], r == c) : omega(seed, cidx[c0 + r], c - s);
  }
  __syncthreads();
  double* Wj = W + c0 * m;
  for (int t = tid; t < m; t += blockDim.x) {
    for (int r = 0; r < s; ++r) Wj[r * m + t] = 0.0;
    for (int it = 0; it < gs; ++it)
      for (int r = 0; r < s; ++r) {
        double a = Aug[r * ld + s + t];
        for (int c = 0; c < s; ++c)
          if (c != r) a = fma(-Aug[r * ld + c], Wj[c * m + t], a);
        Wj[r * m + t] = a / Aug[r * ld + r];
      }
  }
}

// Y_i (D x m row-major at Y + i * D * m), rows [128 h, 128 h + 128) of box i.
// Bound by the FP64 pipe: 160 multiply-adds and one kernel evaluation per
// (row, sample), about 2700 samples a box.  A CTA's share takes the same time
// on every level, so a level of few boxes spreads its sample chunks over
// gridDim.y CTAs (chunk index modulo gridDim.y); split z's partial Y lies z *
// ystride further, and the pivoted QR adds the splits as it loads them.  The
// six levels of N = 16384 (leaf 256) take 22 ms; with one CTA per box half
// each level took 15 ms.
__global__ void __launch_bounds__(256) sketch_kernel(KernelFn G, const double* __restrict__ pts, int D, int m,
                                                     const int* __restrict__ nbox, const int64_t* __restrict__ bpts,
                                                     const int64_t* __restrict__ fptr,
                                                     const int64_t* __restrict__ fidx,
                                                     const int64_t* __restrict__ nptr,
                                                     const int32_t* __restrict__ nidx,
                                                     const int64_t* __restrict__ cptr,
                                                     const int64_t* __restrict__ cidx,
                                                     const double* __restrict__ W, uint64_t seed,
                                                     double* __restrict__ Y, int64_t ystride, int halves) {
  extern __shared__ __align__(16) double sks[];
  double(*Gs)[GC_CHUNK + 1] = reinterpret_cast<double(*)[GC_CHUNK + 1]>(sks);   // GC_ROWS rows
  double* Om = sks + GC_ROWS * (GC_CHUNK + 1);                                   // GC_CHUNK x m
  double(*Xa)[3] = reinterpret_cast<double(*)[3]>(Om + GC_CHUNK * m);            // GC_ROWS rows
  int64_t* pid = reinterpret_cast<int64_t*>(Xa + GC_ROWS);                       // GC_CHUNK
  const int i = blockIdx.x / halves, h = blockIdx.x % halves, tid = threadIdx.x;
  const int nz = gridDim.y;
  int turn = nz - 1 - (int)blockIdx.y;  // chunks to pass over before this CTA's next one, counted up to nz
  const int n = nbox[i];
  const int a0 = h * GC_ROWS;
  if (a0 >= n) return;
  const int rows = min(GC_ROWS, n - a0);
  const int la = tid & (GC_ROWS - 1), half = tid >> 7;
  const int mh = m / 2;  // columns of this thread: [half * mh, half * mh + mh)
  double acc[GC_MAXM / 2];
#pragma unroll
  for (int t = 0; t < GC_MAXM / 2; ++t) acc[t] = 0.0;
  for (int r = tid; r < rows; r += blockDim.x) {
    const int64_t p = bpts[(int64_t)i * D + a0 + r];
    Xa[r][0] = pts[3 * p], Xa[r][1] = pts[3 * p + 1], Xa[r][2] = pts[3 * p + 2];
  }
  // one chunk of sample points q[0 .. cnt): entries G(B_i rows, q) and the
  // chunk's right factor (Omega rows, or W rows when Wsrc is given)
  auto chunk = [&](const int64_t* q, int cnt, const double* Wsrc) {
    __syncthreads();
    if (tid < cnt) pid[tid] = q[tid];
    __syncthreads();
    for (int e = tid; e < GC_ROWS * GC_CHUNK; e += blockDim.x) {
      const int r = e / GC_CHUNK, c = e - r * GC_CHUNK;
      double g = 0.0;
      if (r < rows && c < cnt) {
        const double* y = pts + 3 * pid[c];
        g = G.off(Xa[r], y);
      }
      Gs[r][c] = g;
    }
    for (int e = tid; e < GC_CHUNK * m; e += blockDim.x) {
      const int c = e / m, t = e - c * m;
      Om[e] = (c < cnt) ? (Wsrc ? Wsrc[(int64_t)c * m + t] : omega(seed, pid[c], t)) : 0.0;
    }
    __syncthreads();
    if (la < rows) {
      for (int c = 0; c < cnt; ++c) {
        const double g = Gs[la][c];
        const double* o = Om + c * m + half * mh;
#pragma unroll
        for (int t = 0; t < GC_MAXM / 2; ++t)
          if (t < mh) acc[t] = fma(g, o[t], acc[t]);
      }
    }
  };
  auto mine = [&] {
    if (++turn == nz) turn = 0;
    return turn == 0;
  };
  for (int64_t f = fptr[i]; f < fptr[i + 1]; f += GC_CHUNK)
    if (mine()) chunk(fidx + f, (int)(fptr[i + 1] - f < GC_CHUNK ? fptr[i + 1] - f : GC_CHUNK), nullptr);
  for (int64_t e = nptr[i]; e < nptr[i + 1]; ++e) {
    const int j = nidx[e];
    if (j == i) continue;
    for (int64_t f = cptr[j]; f < cptr[j + 1]; f += GC_CHUNK)
      if (mine()) chunk(cidx + f, (int)(cptr[j + 1] - f < GC_CHUNK ? cptr[j + 1] - f : GC_CHUNK), W + f * m);
  }
  if (la < rows) {
    double* yr = Y + blockIdx.y * ystride + ((int64_t)i * D + a0 + la) * m + half * mh;
#pragma unroll
    for (int t = 0; t < GC_MAXM / 2; ++t)
      if (t < mh) yr[t] = acc[t];
  }
}

// Column-pivoted QR of Z = Y_i^T[0 .. ms) (column a of Z = row a of Y_i, ld
// m, the nz splits of Y added), K steps, then X_i, the skeleton, the pivot
// ratio and probe error.
// A cluster of C CTAs (16 warps each) holds box i: warp g of the cluster owns
// columns g + 16 C c (c < CW), lane l rows l + 32 r (r < NR) of each in
// registers, so Z is read once and a step touches no global memory but the
// finished column of R.  Step k: every warp offers its best column (the norms
// over rows k.. were formed by the previous update), a cluster barrier, the
// owner of the winner forms the Householder vector and stores it into every
// CTA's shared memory, a second cluster barrier, all warps update their
// columns and take the next norms.  Columns are not swapped: a pivot leaves
// the set (ord = its step), ties take the lower column.  The norms are
// recomputed from the updated columns at every step.  Bound by the FP64 pipe
// (three multiply-adds per entry of the shrinking (n - k) x (ms - k) part,
// 7.2 M for n = 256, K = 128), so a level with few boxes takes clusters of up
// to 8 CTAs.  One level of 64 boxes of 256 takes 3.1 ms, one of 2 to 16 boxes
// 1.7 ms (13 us a step: the owner's square root and divisions and the two
// barriers in line); in global memory, one CTA a box, all levels of N = 16384
// took about 15 ms.
// R's column k (rows <= k) and its probe rows go to row k of Y's first split
// (read no more by then); R12 -> T = R11^-1 R12 by column-oriented back
// substitution in registers with R11 in shared memory.
template <int CW, int NR>
__global__ void __launch_bounds__(512, 1)
    pivqr_id_kernel(int D, int m, int ms, int q, int K, int C, int nz, int64_t ystride, const int* __restrict__ nbox,
                    const int64_t* __restrict__ bpts, double* __restrict__ Y, double* __restrict__ X,
                    int64_t* __restrict__ SK, double* __restrict__ rho_out, double* __restrict__ err_out) {
  extern __shared__ __align__(16) double RS[];  // K x K: column t of R11 (rows < t, zeros below)
  __shared__ long long ckey[128];               // candidates of the cluster's warps
  __shared__ int ccol[128];
  __shared__ __align__(16) double vb[32 * NR];
  __shared__ double taub;
  __shared__ double rd[128], rinv[128];
  __shared__ double prb[128 * 8];               // probe rows of the skeleton columns
  __shared__ double e2s[128], y2s[128];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rank = (int)cluster_rank(), i = blockIdx.x / C, g = rank * 16 + warp, G = 16 * C;
  const int n = nbox[i];
  double* Z = Y + (int64_t)i * D * m;
  double z[CW][NR];
  int ord[CW];
#pragma unroll
  for (int c = 0; c < CW; ++c) {
    const int a = g + G * c;
    ord[c] = a < n ? -1 : -2;  // -1: in play, k >= 0: pivot of step k, -2: no column
#pragma unroll
    for (int r = 0; r < NR; ++r) {
      const int t = lane + 32 * r;
      double v = 0.0;
      if (a < n && t < m)
        for (int y = 0; y < nz; ++y) v += Z[y * ystride + (int64_t)a * m + t];
      z[c][r] = v;
    }
  }
  // squared norms over rows k0 .. ms - 1: lane l ends with column
  // tsum_index<CW, 32>(l)'s
  double nrm = 0.0;
  auto norms = [&](int k0) {
    double s[CW];
#pragma unroll
    for (int c = 0; c < CW; ++c) {
      s[c] = 0.0;
      if (ord[c] == -1) {
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (32 * r + 31 >= k0) {
            const int t = lane + 32 * r;
            const double v = (t >= k0 && t < ms) ? z[c][r] : 0.0;
            s[c] = fma(v, v, s[c]);
          }
      }
    }
    nrm = tsum<CW, 32, double>(s);
  };
  norms(0);
  cluster_sync();  // every CTA of the cluster runs (its shared memory may be written) and has read its columns
  const int steps = min(K + 1, min(ms, n));
  double rho2 = 0.0;
  for (int k = 0; k < steps; ++k) {
    // this warp's candidate, to every CTA of the cluster
    {
      const int cm = tsum_index<CW, 32>(lane);
      long long key = -1;
      int col = g + G * cm;
#pragma unroll
      for (int c = 0; c < CW; ++c)
        if (c == cm && ord[c] == -1) key = __double_as_longlong(fabs(nrm));
      for (int o = 16; o; o >>= 1) {
        const long long ok = __shfl_xor_sync(0xffffffffu, key, o);
        const int oc = __shfl_xor_sync(0xffffffffu, col, o);
        if (ok > key || (ok == key && oc < col)) key = ok, col = oc;
      }
      if (lane < C) {
        st_cluster(cluster_map(&ckey[g], lane), key);
        st_cluster(cluster_map(&ccol[g], lane), col);
      }
    }
    cluster_sync();
    long long best = -1;
    int pc = 0;
    for (int e = lane; e < G; e += 32) {
      const long long v = ckey[e];
      const int cc = ccol[e];
      if (v > best || (v == best && cc < pc)) best = v, pc = cc;
    }
    for (int o = 16; o; o >>= 1) {
      const long long ov = __shfl_xor_sync(0xffffffffu, best, o);
      const int oc = __shfl_xor_sync(0xffffffffu, pc, o);
      if (ov > best || (ov == best && oc < pc)) best = ov, pc = oc;
    }
    if (k == K) {  // the first pivot beyond K: only its size is asked for
      rho2 = __longlong_as_double(best);
      break;
    }
    if (pc % G == g) {
      const int cs = pc / G;
      double zc[NR];
#pragma unroll
      for (int c = 0; c < CW; ++c)
        if (c == cs) {
          ord[c] = k;
#pragma unroll
          for (int r = 0; r < NR; ++r) zc[r] = z[c][r];
        }
      double part = 0.0, alpha = 0.0;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int t = lane + 32 * r;
        if (t > k && t < ms) part = fma(zc[r], zc[r], part);
        if (t == k) alpha = zc[r];
      }
      for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
      alpha = __shfl_sync(0xffffffffu, alpha, k & 31);
      double tau = 0.0, beta = alpha, scal = 0.0;
      if (part != 0.0) {
        beta = -copysign(sqrt(alpha * alpha + part), alpha);
        tau = (beta - alpha) / beta;
        scal = 1.0 / (alpha - beta);
      }
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int t = lane + 32 * r;
        const double v = (t > k && t < ms) ? zc[r] * scal : (t == k ? 1.0 : 0.0);
        for (int cta = 0; cta < C; ++cta) st_cluster(cluster_map(&vb[t], cta), v);
        if (t < k || (t >= ms && t < m)) Z[(int64_t)k * m + t] = zc[r];
        if (t == k) Z[(int64_t)k * m + t] = beta;
      }
      if (lane < C) st_cluster(cluster_map(&taub, lane), tau);
    }
    cluster_sync();
    const double tau = taub;
    double v[NR], s[CW];
#pragma unroll
    for (int r = 0; r < NR; ++r) v[r] = vb[lane + 32 * r];
#pragma unroll
    for (int c = 0; c < CW; ++c) {
      s[c] = 0.0;
      if (ord[c] == -1) {
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (32 * r + 31 >= k) s[c] = fma(v[r], z[c][r], s[c]);
      }
    }
    const double dot = tau * tsum<CW, 32, double>(s);
#pragma unroll
    for (int c = 0; c < CW; ++c) {
      // (any lane whose tsum_index is c)
      const double w = __shfl_sync(0xffffffffu, dot, tsum_lane<CW, 32>(c));
      if (ord[c] == -1) {
#pragma unroll
        for (int r = 0; r < NR; ++r)
          if (32 * r + 31 >= k) z[c][r] = fma(-w, v[r], z[c][r]);
      }
    }
    norms(k + 1);
  }
  // (the barriers of the last step order the R columns before these reads:
  // with steps == K that step's update has none after it)
  cluster_sync();
  const double rr0 = fabs(Z[0]);
  if (rank == 0 && tid == 0) rho_out[i] = (steps > K && rr0 > 0.0) ? sqrt(rho2) / rr0 : 0.0;
  for (int e = tid; e < K * K; e += blockDim.x) {
    const int t = e / K, r = e - t * K;
    RS[e] = r < t ? Z[(int64_t)t * m + r] : 0.0;
  }
  for (int t = tid; t < K; t += blockDim.x) {
    const double d = Z[(int64_t)t * m + t];
    const bool ok = fabs(d) > 1e-15 * rr0 && d != 0.0;
    rd[t] = d;
    rinv[t] = ok ? 1.0 / d : 0.0;
  }
  for (int e = tid; e < K * 8; e += blockDim.x) {
    const int u = e >> 3, c = e & 7;
    prb[e] = c < q ? Z[(int64_t)u * m + ms + c] : 0.0;
  }
  __syncthreads();
#pragma unroll
  for (int rb = 3; rb >= 0; --rb) {
    if (rb >= NR) continue;
    for (int tt = 31; tt >= 0; --tt) {
      const int t = 32 * rb + tt;
      if (t >= K) continue;
      const double d = rd[t], inv = rinv[t];
      double rc[4];
#pragma unroll
      for (int r = 0; r <= rb; ++r) rc[r] = (lane + 32 * r < K) ? RS[t * K + lane + 32 * r] : 0.0;
#pragma unroll
      for (int c = 0; c < CW; ++c) {
        if (ord[c] != -1) continue;
        const double sv = __shfl_sync(0xffffffffu, z[c][rb], tt);
        // quotient by the reciprocal and one correction
        double x = sv * inv;
        x = fma(fma(-x, d, sv), inv, x);
#pragma unroll
        for (int r = 0; r <= rb; ++r) z[c][r] = fma(-x, rc[r], z[c][r]);
        if (lane == tt) z[c][rb] = x;
      }
    }
  }
  // X (D x K row-major; rows n .. D - 1 are padding), skeleton, probe error
  double e2 = 0.0, y2 = 0.0;
#pragma unroll
  for (int c = 0; c < CW; ++c) {
    const int a = g + G * c;
    if (a < D) {
      double* xr = X + ((int64_t)i * D + a) * K;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int u = lane + 32 * r;
        if (u < K) xr[u] = ord[c] == -1 ? z[c][r] : (ord[c] == u ? 1.0 : 0.0);
      }
      if (ord[c] >= 0 && lane == 0) SK[(int64_t)i * K + ord[c]] = bpts[(int64_t)i * D + a];
    }
    if (ord[c] != -2) {
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const int t = lane + 32 * r;
        if (t >= ms && t < ms + q) y2 = fma(z[c][r], z[c][r], y2);
      }
    }
    if (ord[c] == -1) {
      double s[8];
#pragma unroll
      for (int p = 0; p < 8; ++p) s[p] = 0.0;
#pragma unroll
      for (int r = 0; r < (NR < 4 ? NR : 4); ++r) {
        const int u = lane + 32 * r;
        if (u < K)
#pragma unroll
          for (int p = 0; p < 8; ++p) s[p] = fma(z[c][r], prb[u * 8 + p], s[p]);
      }
      const double sp = tsum<8, 32, double>(s);
      const int p = tsum_index<8, 32>(lane);
      // the column's own probe entry, row ms + p
      const int t = ms + min(p, q - 1);
      double own = 0.0;
#pragma unroll
      for (int r = 0; r < NR; ++r) {
        const double o = __shfl_sync(0xffffffffu, z[c][r], t & 31);
        if ((t >> 5) == r) own = o;
      }
      if (p < q && tsum_leader<8, 32>(lane)) e2 = fma(own - sp, own - sp, e2);
    }
  }
  for (int o = 16; o; o >>= 1) {
    e2 += __shfl_xor_sync(0xffffffffu, e2, o);
    y2 += __shfl_xor_sync(0xffffffffu, y2, o);
  }
  if (lane == 0) {
    st_cluster(cluster_map(&e2s[g], 0), __double_as_longlong(e2));
    st_cluster(cluster_map(&y2s[g], 0), __double_as_longlong(y2));
  }
  cluster_sync();
  if (rank == 0 && tid == 0) {
    double a = 0.0, b = 0.0;
    for (int w = 0; w < G; ++w) a += e2s[w], b += y2s[w];
    err_out[i] = sqrt(a / fmax(b, 1e-300));
  }
}

}  // namespace

namespace {
void launch_cc_weights(const KernelFn& G, const double* pts, int nb, const int64_t* cptr, const int64_t* cidx, int m,
                       uint64_t seed, int gs, double* W, cudaStream_t st) {
  ++g_launches;
  if (gs > 0) {
    const size_t sm = sizeof(double) * (size_t)GC_MAXS * (GC_MAXS + m);
    allow_smem((const void*)cc_sweeps_kernel);
    cc_sweeps_kernel<<<nb, 256, sm, st>>>(G, pts, cptr, cidx, m, seed, gs, W);
    return;
  }
  // one CTA per box when the boxes fill the SMs, else Omega's columns over
  // two or four (a CTA's time goes with 64 x (40 + its columns))
  const int nsm = num_sms();
  if (nb >= nsm || m <= 48) cc_weights_kernel<10><<<dim3(nb, (m + 159) / 160), 256, 0, st>>>(G, pts, cptr, cidx, m, seed, W);
  else if (nb > nsm / 2) cc_weights_kernel<5><<<dim3(nb, (m + 79) / 80), 256, 0, st>>>(G, pts, cptr, cidx, m, seed, W);
  else cc_weights_kernel<3><<<dim3(nb, (m + 47) / 48), 256, 0, st>>>(G, pts, cptr, cidx, m, seed, W);
}

// CTAs a box's sample chunks are split over: about four per SM in all (one is
// resident: 200 registers a thread), so that the last wave weighs little; at
// most 16 (every split writes its own Y_i, 0.3 MB)
int sketch_splits(int nb, int halves) {
  const int base = std::max(1, nb * halves);
  return std::max(1, std::min(16, (4 * num_sms() + base - 1) / base));
}

void launch_sketch(const KernelFn& G, const double* pts, int nb, int D, int m, int nz, const int* nbox,
                   const int64_t* bpts, const int64_t* fptr, const int64_t* fidx, const int64_t* nptr,
                   const int32_t* nidx, const int64_t* cptr, const int64_t* cidx, const double* W, uint64_t seed,
                   double* Y, cudaStream_t st) {
  const size_t sm = sizeof(double) * ((size_t)GC_ROWS * (GC_CHUNK + 1) + (size_t)GC_CHUNK * m + GC_ROWS * 3) +
                    sizeof(int64_t) * GC_CHUNK;
  allow_smem((const void*)sketch_kernel);
  const int halves = (D + GC_ROWS - 1) / GC_ROWS;
  ++g_launches;
  sketch_kernel<<<dim3(halves * nb, nz), 256, sm, st>>>(G, pts, D, m, nbox, bpts, fptr, fidx, nptr, nidx, cptr, cidx,
                                                        W, seed, Y, (int64_t)nb * D * m, halves);
}

template <int CW, int NR>
cudaError_t launch_pivqr_t(int C, int nb, int D, int m, int ms, int q, int K, int nz, const int* nbox,
                           const int64_t* bpts, double* Y, double* X, int64_t* SK, double* rho, double* err,
                           cudaStream_t st) {
  const size_t sm = sizeof(double) * (size_t)K * K;
  allow_smem((const void*)pivqr_id_kernel<CW, NR>);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nb * C));
  cfg.blockDim = dim3(512);
  cfg.dynamicSmemBytes = sm;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)C;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  ++g_launches;
  return cudaLaunchKernelEx(&cfg, pivqr_id_kernel<CW, NR>, D, m, ms, q, K, C, nz, (int64_t)nb * D * m, nbox, bpts, Y,
                            X, SK, rho, err);
}

// cluster size: the fewest CTAs whose 16 warps hold the box at 8 columns a
// warp (128 columns a CTA), doubled while the level still leaves SMs idle
cudaError_t launch_pivqr_id(int nb, int D, int m, int ms, int q, int K, int nz, const int* nbox, const int64_t* bpts,
                            double* Y, double* X, int64_t* SK, double* rho, double* err, cudaStream_t st) {
  int C = D > 128 ? 2 : 1;
  while (C < 8 && nb * C * 2 <= num_sms() && 16 * C < D) C *= 2;
  const int cw = (D + 16 * C - 1) / (16 * C);
#define GC_QR(CW)                                                                                         \
  return m <= 96 ? launch_pivqr_t<CW, 3>(C, nb, D, m, ms, q, K, nz, nbox, bpts, Y, X, SK, rho, err, st) \
                 : launch_pivqr_t<CW, 5>(C, nb, D, m, ms, q, K, nz, nbox, bpts, Y, X, SK, rho, err, st)
  if (cw <= 1) GC_QR(1);
  if (cw <= 2) GC_QR(2);
  if (cw <= 4) GC_QR(4);
  GC_QR(8);
#undef GC_QR
}
}  // namespace

// ---------------------------------------------------------------------------
// host side: one level at a time; device buffers grow as needed
// ---------------------------------------------------------------------------
namespace {

struct DeviceGpuCompressor : GpuCompressor {
  KernelFn G;
  int gs = 0;
  double* pts = nullptr;
  std::vector<void*> bufs;  // freed at destruction
  ~DeviceGpuCompressor() override {
    for (void* b : bufs) cudaFree(b);
    cudaFree(pts);
  }
  bool supported(int D, int K) const override { return D <= 2 * GC_ROWS && K >= 1 && K + 32 <= GC_MAXM; }
  template <typename V>
  cudaError_t put(V** d, const std::vector<V>& h) {
    *d = nullptr;
    cudaError_t e = cudaMalloc(d, sizeof(V) * std::max<size_t>(h.size(), 1));
    if (e != cudaSuccess) return e;
    bufs.push_back(*d);
    if (!h.empty()) e = cudaMemcpy(*d, h.data(), sizeof(V) * h.size(), cudaMemcpyHostToDevice);
    return e;
  }
  template <typename V>
  cudaError_t make(V** d, size_t n) {
    cudaError_t e = cudaMalloc(d, sizeof(V) * std::max<size_t>(n, 1));
    if (e == cudaSuccess) bufs.push_back(*d);
    return e;
  }
  std::string run(GpuLevelJob& j) override {
    j.gs = gs;
    const size_t nb = j.nb, D = j.D, K = j.K, m = j.m;
    int* d_nbox;
    int64_t *d_bpts, *d_fptr, *d_fidx, *d_nptr, *d_cptr, *d_cidx, *d_SK;
    int32_t* d_nidx;
    double *d_W, *d_Y, *d_X, *d_rho, *d_err;
    cudaError_t e = cudaSuccess;
#define GC_TRY(x) \
  if ((e = (x)) != cudaSuccess) return std::string(#x) + ": " + cudaGetErrorString(e)
    const size_t nbufs = bufs.size();
    GC_TRY(put(&d_nbox, j.nbox));
    GC_TRY(put(&d_bpts, j.bpts));
    GC_TRY(put(&d_fptr, j.fptr));
    GC_TRY(put(&d_fidx, j.fidx));
    GC_TRY(put(&d_nptr, j.nptr));
    GC_TRY(put(&d_nidx, j.nidx));
    GC_TRY(put(&d_cptr, j.cptr));
    GC_TRY(put(&d_cidx, j.cidx));
    GC_TRY(make(&d_W, j.cidx.size() * m));
    GC_TRY(make(&d_X, nb * D * K));
    GC_TRY(make(&d_SK, nb * K));
    GC_TRY(make(&d_rho, nb));
    GC_TRY(make(&d_err, nb));
    // (the splits' partial sums last: fewer splits where they do not fit)
    int nz = sketch_splits(j.nb, (j.D + GC_ROWS - 1) / GC_ROWS);
    while ((e = make(&d_Y, nz * nb * D * m)) == cudaErrorMemoryAllocation && nz > 1) {
      cudaGetLastError();
      nz /= 2;
    }
    if (e != cudaSuccess) return std::string("the sketch's sums: ") + cudaGetErrorString(e);
    launch_cc_weights(G, pts, j.nb, d_cptr, d_cidx, j.m, j.seed, j.gs, d_W, 0);
    launch_sketch(G, pts, j.nb, j.D, j.m, nz, d_nbox, d_bpts, d_fptr, d_fidx, d_nptr, d_nidx, d_cptr, d_cidx, d_W,
                  j.seed, d_Y, 0);
    GC_TRY(launch_pivqr_id(j.nb, j.D, j.m, j.ms, j.q, j.K, nz, d_nbox, d_bpts, d_Y, d_X, d_SK, d_rho, d_err, 0));
    GC_TRY(take_launch_error());
    j.X.resize(nb * D * K);
    j.SK.resize(nb * K);
    j.rho.resize(nb);
    j.err.resize(nb);
    GC_TRY(cudaMemcpy(j.X.data(), d_X, sizeof(double) * j.X.size(), cudaMemcpyDeviceToHost));
    GC_TRY(cudaMemcpy(j.SK.data(), d_SK, sizeof(int64_t) * j.SK.size(), cudaMemcpyDeviceToHost));
    GC_TRY(cudaMemcpy(j.rho.data(), d_rho, sizeof(double) * nb, cudaMemcpyDeviceToHost));
    GC_TRY(cudaMemcpy(j.err.data(), d_err, sizeof(double) * nb, cudaMemcpyDeviceToHost));
#undef GC_TRY
    for (size_t b = nbufs; b < bufs.size(); ++b) cudaFree(bufs[b]);
    bufs.resize(nbufs);
    // flops (2 per multiply-add; kernel evaluations not counted): the
    // close-field part (W_j and the close sketch terms) and the far part
    for (size_t jb = 0; jb < nb; ++jb) {
      const double sj = (double)(j.cptr[jb + 1] - j.cptr[jb]);
      j.flops_prefactor += 2.0 * sj * sj * (sj + (double)m);
    }
    for (size_t i = 0; i < nb; ++i) {
      const double ni = j.nbox[i];
      j.flops_far += 2.0 * ni * (double)(j.fptr[i + 1] - j.fptr[i]) * (double)m;
      for (int64_t e2 = j.nptr[i]; e2 < j.nptr[i + 1]; ++e2) {
        const int jj = j.nidx[e2];
        if ((size_t)jj == i) continue;
        j.flops_prefactor += 2.0 * ni * (double)(j.cptr[jj + 1] - j.cptr[jj]) * (double)m;
      }
    }
    return "";
  }
};

}  // namespace

GpuCompressor* make_gpu_compressor(const KernelFn& G, const double* pts, int64_t N, int gs_sweeps) {
  DeviceGpuCompressor* c = new DeviceGpuCompressor();
  c->G = G;
  c->gs = gs_sweeps;
  if (cudaMalloc(&c->pts, sizeof(double) * 3 * (size_t)N) != cudaSuccess ||
      cudaMemcpy(c->pts, pts, sizeof(double) * 3 * (size_t)N, cudaMemcpyHostToDevice) != cudaSuccess) {
    cudaGetLastError();
    delete c;
    return nullptr;
  }
  return c;
}

}  // namespace h2
