// Blocked FP64 Cholesky factor and triangular inverse of the small matrices of the subspace calls
// (the Gram matrix of Cholesky-QR, the projected overlap of Rayleigh-Ritz), spread over the GPU.
//
// Bound: a chain of n / CB block columns, each a few dependent FP64 operations of CB steps; the
// FP64 pipe issues two multiply-adds a clock per SM, so the trailing updates are spread over one
// CTA per CB x CB block and CB is small (16: one output per thread of a 256-thread CTA, 1 us per
// block product; at 32 each product alone takes 8 us on its SM). One launch per block column: the
// CTA of the next diagonal block factors and inverts it right after its update, so the chain has
// no launch of its own for it. The one-CTA right-looking factor and the one-thread-per-column
// inverse that this replaces took 4.78 + 6.45 ms at n = 360 (real), and 16.7 + 20.1 ms in complex
// arithmetic.
#include "oefe_internal.h"

namespace {

constexpr int CB = 16;   // block size

__device__ __forceinline__ double c_zero(double) { return 0.0; }
__device__ __forceinline__ cd c_zero(cd) { return mkc(0, 0); }
__device__ __forceinline__ double c_one(double) { return 1.0; }
__device__ __forceinline__ cd c_one(cd) { return mkc(1, 0); }
__device__ __forceinline__ double c_re(double a) { return a; }
__device__ __forceinline__ double c_re(cd a) { return a.x; }
__device__ __forceinline__ double c_real(double a, double) { return a; }
__device__ __forceinline__ cd c_real(double a, cd) { return mkc(a, 0.0); }
__device__ __forceinline__ double c_scale(double a, double s) { return a * s; }
__device__ __forceinline__ cd c_scale(cd a, double s) { return a * s; }
// acc + a b and acc + a conj(b)
__device__ __forceinline__ double c_fma(double a, double b, double acc) { return fma(a, b, acc); }
__device__ __forceinline__ cd c_fma(cd a, cd b, cd acc) { return cfma(a, b, acc); }
__device__ __forceinline__ double c_fmac(double a, double b, double acc) { return fma(a, b, acc); }
__device__ __forceinline__ cd c_fmac(cd a, cd b, cd acc) { return cfmac(b, a, acc); }
__device__ __forceinline__ double c_neg(double a) { return -a; }
__device__ __forceinline__ cd c_neg(cd a) { return -a; }

// The diagonal block d (rows j0 .. j0 + nb) in shared memory: its lower Cholesky factor into L, the
// inverse of the factor into Dinv (CB x CB, zero outside the lower triangle). Returns the failing
// pivot + 1 (0: none). All 256 threads.
template <typename S>
__device__ int factor_block(S (*d)[CB + 1], S (*y)[CB + 1], int nb) {
  __shared__ double inv_[CB];
  __shared__ int bad;
  const int i = threadIdx.x / CB, k = threadIdx.x % CB;
  if (threadIdx.x == 0) bad = 0;
  __syncthreads();
  for (int j = 0; j < nb; ++j) {
    if (threadIdx.x == 0) {
      const double p = c_re(d[j][j]);
      if (!(p > 0.0) || !isfinite(p)) bad = j + 1;
      const double s = sqrt(p);
      d[j][j] = c_real(s, S{});
      inv_[j] = 1.0 / s;
    }
    __syncthreads();
    if (bad) return bad;
    if (k == j && i > j && i < nb) d[i][j] = c_scale(d[i][j], inv_[j]);
    __syncthreads();
    if (k > j && k <= i && i < nb) d[i][k] = c_fmac(c_neg(d[i][j]), d[k][j], d[i][k]);
    __syncthreads();
  }
  // inverse by rows: y_ic = (delta_ic - sum_{c <= m < i} L_im y_mc) / L_ii, a thread per column
  if (threadIdx.x < CB) {
    const int c = threadIdx.x;
    for (int r = 0; r < CB; ++r) {
      S s = r == c && r < nb ? c_one(S{}) : c_zero(S{});
      if (r < nb && c < nb && r >= c) {
        for (int m = c; m < r; ++m) s = c_fma(c_neg(d[r][m]), y[m][c], s);
        s = c_scale(s, inv_[r]);
      } else {
        s = c_zero(S{});
      }
      y[r][c] = s;
    }
  }
  __syncthreads();
  return 0;
}

// Step p of the right-looking factor of A (lower triangle used): the CTA (i, k), i >= k > p, takes
// A_ik -= L_ip L_kp^+ with L_ip = A_ip Dinv_p^+ formed here; the CTAs of column p + 1 store L_ip and
// the CTA of the diagonal block p + 1 factors it. p = -1 factors block 0 only.
template <typename S>
__global__ void __launch_bounds__(CB * CB) k_chol_step(S* __restrict__ A, S* __restrict__ L, S* __restrict__ Dinv, int n,
                                                       int p, int* info) {
  __shared__ S ai[CB][CB + 1], ak[CB][CB + 1], dp[CB][CB + 1], li[CB][CB + 1], lk[CB][CB + 1];
  if (*info) return;
  const int r = threadIdx.x / CB, c = threadIdx.x % CB;
  // blockIdx.x enumerates the pairs (i, k), i >= k, of the trailing blocks row by row
  int bi = 0, t = blockIdx.x;
  while (t > bi) { t -= bi + 1; ++bi; }
  const int i = p + 1 + bi, k = p + 1 + t;
  const int ri = i * CB + r, ck = k * CB + c;
  auto at = [&](int row, int col) { return row < n && col < n ? A[(size_t)row * n + col] : c_zero(S{}); };
  S v = at(ri, ck);
  if (p >= 0) {
    const int pc = p * CB + c;
    ai[r][c] = at(ri, pc);
    ak[r][c] = at(k * CB + r, pc);
    dp[r][c] = Dinv[(size_t)p * CB * CB + threadIdx.x];
    __syncthreads();
    S a = c_zero(S{}), b = c_zero(S{});
#pragma unroll
    for (int m = 0; m < CB; ++m) {   // L_ip[r][c] = sum_m A_ip[r][m] conj(Dinv_p[c][m])
      a = c_fmac(ai[r][m], dp[c][m], a);
      if (i != k) b = c_fmac(ak[r][m], dp[c][m], b);
    }
    li[r][c] = a;
    lk[r][c] = i != k ? b : a;
    if (k == p + 1 && ri < n && pc < n) L[(size_t)ri * n + pc] = a;
    __syncthreads();
#pragma unroll
    for (int m = 0; m < CB; ++m) v = c_fmac(c_neg(li[r][m]), lk[c][m], v);
  }
  if (i != p + 1) {
    if (ri < n && ck < n) A[(size_t)ri * n + ck] = v;
    return;
  }
  // i == k == p + 1: the next diagonal block
  __syncthreads();
  ai[r][c] = v;
  const int nb = min(CB, n - i * CB);
  const int bad = factor_block<S>(ai, ak, nb);
  if (bad) {
    if (threadIdx.x == 0) *info = i * CB + bad;
    return;
  }
  if (ri < n && ck < n && c <= r) L[(size_t)ri * n + ck] = ai[r][c];
  Dinv[(size_t)i * CB * CB + threadIdx.x] = ak[r][c];
}

// Y = L^{-1}: a CTA per CC columns, down the row blocks: Y_i = Dinv_i (E_i - sum_{k < i} L_ik Y_k),
// CB rows x CC columns per block, the sum split over KS threads per entry. Zeros above the diagonal
// blocks of the columns come from the caller.
constexpr int CC = 4;
constexpr int KS = 4;
template <typename S>
__global__ void __launch_bounds__(CB * CC * KS) k_tri_inv(const S* __restrict__ L, const S* __restrict__ Dinv, S* Y,
                                                          int n) {
  __shared__ S part[KS][CB][CC];
  __shared__ S rhs[CB][CC];
  const int c0 = blockIdx.x * CC;
  const int b0 = c0 / CB, nblk = (n + CB - 1) / CB;
  const int c = threadIdx.x % CC, s = (threadIdx.x / CC) % KS, r = threadIdx.x / (CC * KS);
  for (int i = b0; i < nblk; ++i) {
    const int row = i * CB + r;
    S acc = c_zero(S{});
    if (row < n && c0 + c < n)
      for (int k = b0 * CB + s; k < i * CB; k += KS) acc = c_fma(L[(size_t)row * n + k], Y[(size_t)k * n + c0 + c], acc);
    part[s][r][c] = acc;
    __syncthreads();
    if (s == 0) {
      S t = row == c0 + c ? c_one(S{}) : c_zero(S{});
#pragma unroll
      for (int u = 0; u < KS; ++u) t = t + c_neg(part[u][r][c]);
      rhs[r][c] = t;
    }
    __syncthreads();
    if (s == 0 && row < n && c0 + c < n) {
      S y = c_zero(S{});
      for (int m = 0; m <= r; ++m) y = c_fma(Dinv[(size_t)i * CB * CB + r * CB + m], rhs[m][c], y);
      Y[(size_t)row * n + c0 + c] = y;
    }
    __syncthreads();   // the block's rows of Y are visible to the whole CTA (the only reader)
  }
}

}  // namespace

size_t chol_scratch(int n, size_t scalar) { return (size_t)((n + CB - 1) / CB) * CB * CB * scalar; }

// L = lower Cholesky factor of A (overwritten), Y = L^{-1}, both full n x n with zero upper parts;
// scratch: chol_scratch() bytes; *info_host: 0, or the failing pivot + 1 (then L and Y are partial).
// d_info: a device word.
template <typename S>
int chol_factor_inverse(oefe_ctx* c, S* A, S* L, S* Y, int n, void* scratch, int* d_info, int* info_host) {
  S* Dinv = (S*)scratch;
  const int nblk = (n + CB - 1) / CB;
  const size_t nn = (size_t)n * n * sizeof(S);
  OEFE_CUDA_TRY(c, cudaMemsetAsync(d_info, 0, sizeof(int), c->stream));
  OEFE_CUDA_TRY(c, cudaMemsetAsync(L, 0, nn, c->stream));
  OEFE_CUDA_TRY(c, cudaMemsetAsync(Y, 0, nn, c->stream));
  for (int p = -1; p + 1 < nblk; ++p) {
    const int m = nblk - p - 1;   // trailing block rows
    OEFE_COUNTED k_chol_step<S><<<p < 0 ? 1 : m * (m + 1) / 2, CB * CB, 0, c->stream>>>(A, L, Dinv, n, p, d_info);
  }
  // (on a failed factor the inverse below works on partial data; the caller discards it)
  OEFE_COUNTED k_tri_inv<S><<<(n + CC - 1) / CC, CB * CC * KS, 0, c->stream>>>(L, Dinv, Y, n);
  OEFE_CUDA_TRY(c, cudaGetLastError());
  OEFE_CUDA_TRY(c, cudaMemcpyAsync(info_host, d_info, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  OEFE_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return OEFE_OK;
}

template int chol_factor_inverse<double>(oefe_ctx*, double*, double*, double*, int, void*, int*, int*);
template int chol_factor_inverse<cd>(oefe_ctx*, cd*, cd*, cd*, int, void*, int*, int*);
