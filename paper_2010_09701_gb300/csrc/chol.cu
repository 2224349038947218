// Blocked FP64 Cholesky factor and triangular inverse of the small matrices of the subspace calls
// (the Gram matrix of Cholesky-QR, the projected overlap of Rayleigh-Ritz), spread over the GPU.
//
// Bound: a chain of n / CB block columns, each a few dependent FP64 operations of CB steps; the
// FP64 pipe issues two multiply-adds a clock per SM, so the trailing updates are spread over one
// CTA per CB x CB block and CB is small (16: one output per thread of a 256-thread CTA). One launch per
// block column: the CTA of the next diagonal block factors it right after its update, so the chain has
// no launch of its own for it.
//
// Every entry takes the operations of the unblocked right-looking factor in its order (a_ik - l_i0 l_k0^*
// - l_i1 l_k1^* ..., then times 1 / l_kk), and the inverse those of the unblocked substitution: the
// signs of Ritz vectors follow the last bits of the projected matrix, so another order would return other
// vectors. The one-CTA right-looking factor and the one-thread-per-column inverse that this replaces took
// 4.78 + 6.45 ms at n = 360 (real), and 16.7 + 20.1 ms in complex arithmetic; these take 1.1 + 1.1 ms there.
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
// v - a conj(b) and v - a b
__device__ __forceinline__ double c_subc(double v, double a, double b) { return v - a * b; }
__device__ __forceinline__ cd c_subc(cd v, cd a, cd b) { return v - a * cconj(b); }
__device__ __forceinline__ double c_sub(double v, double a, double b) { return v - a * b; }
__device__ __forceinline__ cd c_sub(cd v, cd a, cd b) { return v - a * b; }

// The diagonal block d (nb rows) in shared memory: its lower Cholesky factor in place, 1 / l_jj into inv.
// Returns the failing pivot + 1 (0: none). All 256 threads.
template <typename S>
__device__ int factor_block(S (*d)[CB + 1], double* inv, int nb) {
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
      inv[j] = 1.0 / s;
    }
    __syncthreads();
    if (bad) return bad;
    if (k == j && i > j && i < nb) d[i][j] = c_scale(d[i][j], inv[j]);
    __syncthreads();
    if (k > j && k <= i && i < nb) d[i][k] = c_subc(d[i][k], d[i][j], d[k][j]);
    __syncthreads();
  }
  return 0;
}

// Step p of the right-looking factor of A (lower triangle used): the CTA (i, k), i >= k > p, takes
// A_ik -= L_ip L_kp^+ with L_ip = A_ip L_pp^{-+} by substitution here; the CTAs of column p + 1 store L_ip
// and the CTA of the diagonal block p + 1 factors it. p = -1 factors block 0 only. inv: 1 / l_jj.
template <typename S>
__global__ void __launch_bounds__(CB * CB) k_chol_step(S* __restrict__ A, S* __restrict__ L, double* __restrict__ inv, int n,
                                                       int p, int* info) {
  __shared__ S li[CB][CB + 1], lk[CB][CB + 1], lp[CB][CB + 1];
  __shared__ double iv[CB];
  // only a failure of an earlier launch counts (its pivot lies in the blocks up to p): the diagonal block of this
  // launch may report one while other CTAs start, and a CTA must take one decision
  const int failed = *(volatile int*)info;
  if (failed && failed <= (p + 1) * CB) return;
  const int r = threadIdx.x / CB, c = threadIdx.x % CB;
  // blockIdx.x enumerates the pairs (i, k), i >= k, of the trailing blocks row by row
  int bi = 0, t = blockIdx.x;
  while (t > bi) { t -= bi + 1; ++bi; }
  const int i = p + 1 + bi, k = p + 1 + t;
  const int ri = i * CB + r, ck = k * CB + c;
  auto at = [&](int row, int col) { return row < n && col < n ? A[(size_t)row * n + col] : c_zero(S{}); };
  S v = at(ri, ck);
  if (p >= 0) {
    const int pc = p * CB + c;   // (block p is whole: a trailing block follows it)
    li[r][c] = at(ri, pc);
    lk[r][c] = at(k * CB + r, pc);
    lp[r][c] = L[(size_t)(p * CB + r) * n + pc];
    if (threadIdx.x < CB) iv[threadIdx.x] = inv[p * CB + threadIdx.x];
    __syncthreads();
    for (int j = 0; j < CB; ++j) {   // a row is half a warp's
      if (c == j) {
        li[r][j] = c_scale(li[r][j], iv[j]);
        lk[r][j] = c_scale(lk[r][j], iv[j]);
      }
      __syncwarp();
      if (c > j) {
        li[r][c] = c_subc(li[r][c], li[r][j], lp[c][j]);
        lk[r][c] = c_subc(lk[r][c], lk[r][j], lp[c][j]);
      }
      __syncwarp();
    }
    if (k == p + 1 && ri < n) L[(size_t)ri * n + pc] = li[r][c];
    __syncthreads();
#pragma unroll
    for (int m = 0; m < CB; ++m) v = c_subc(v, li[r][m], lk[c][m]);
  }
  if (i != p + 1) {
    if (ri < n && ck < n) A[(size_t)ri * n + ck] = v;
    return;
  }
  // i == k == p + 1: the next diagonal block
  __syncthreads();
  li[r][c] = v;
  const int nb = min(CB, n - i * CB);
  const int bad = factor_block<S>(li, iv, nb);
  if (bad) {
    if (threadIdx.x == 0) *info = i * CB + bad;
    return;
  }
  if (ri < n && ck < n && c <= r) L[(size_t)ri * n + ck] = li[r][c];
  if ((int)threadIdx.x < nb) inv[i * CB + threadIdx.x] = iv[threadIdx.x];
}

// Y = L^{-1}: a CTA per CC columns, down the row blocks, a thread per entry of a block: its sum over the
// rows above the block, then the substitution within it. Zeros above the diagonal blocks of the
// columns come from the caller.
constexpr int CC = 4;
template <typename S>
__global__ void __launch_bounds__(CB * CC) k_tri_inv(const S* __restrict__ L, const double* __restrict__ inv, S* Y, int n) {
  __shared__ S y[CB][CC], lb[CB][CB + 1];
  const int c0 = blockIdx.x * CC;
  const int b0 = c0 / CB, nblk = (n + CB - 1) / CB;
  const int c = threadIdx.x % CC, r = threadIdx.x / CC;
  for (int i = b0; i < nblk; ++i) {
    const int row = i * CB + r;
    for (int t = threadIdx.x; t < CB * CB; t += CB * CC) {
      const int a = i * CB + t / CB, b = i * CB + t % CB;
      lb[t / CB][t % CB] = a < n && b < n ? L[(size_t)a * n + b] : c_zero(S{});
    }
    const bool in = row < n && c0 + c < n;
    S s = row == c0 + c ? c_one(S{}) : c_zero(S{});
    if (in) {
#pragma unroll 16
      for (int k = b0 * CB; k < i * CB; ++k) s = c_sub(s, L[(size_t)row * n + k], Y[(size_t)k * n + c0 + c]);
    }
    __syncthreads();
    for (int m = 0; m < CB; ++m) {
      if (r == m) y[m][c] = in && row >= c0 + c ? c_scale(s, inv[row]) : c_zero(S{});
      __syncthreads();
      if (r > m) s = c_sub(s, lb[r][m], y[m][c]);
    }
    if (in) Y[(size_t)row * n + c0 + c] = y[r][c];
    __syncthreads();   // the block's rows of Y are visible to the whole CTA (the only reader)
  }
}

}  // namespace

size_t chol_scratch(int n) { return (size_t)n * sizeof(double); }

// L = lower Cholesky factor of A (overwritten), Y = L^{-1}, both full n x n with zero upper parts;
// scratch: chol_scratch() bytes; *info_host: 0, or the failing pivot + 1 (then L and Y are partial).
// d_info: a device word.
template <typename S>
int chol_factor_inverse(oefe_ctx* c, S* A, S* L, S* Y, int n, void* scratch, int* d_info, int* info_host) {
  double* inv = (double*)scratch;
  const int nblk = (n + CB - 1) / CB;
  const size_t nn = (size_t)n * n * sizeof(S);
  OEFE_CUDA_TRY(c, cudaMemsetAsync(d_info, 0, sizeof(int), c->stream));
  OEFE_CUDA_TRY(c, cudaMemsetAsync(L, 0, nn, c->stream));
  OEFE_CUDA_TRY(c, cudaMemsetAsync(Y, 0, nn, c->stream));
  for (int p = -1; p + 1 < nblk; ++p) {
    const int m = nblk - p - 1;   // trailing block rows
    OEFE_COUNTED k_chol_step<S><<<p < 0 ? 1 : m * (m + 1) / 2, CB * CB, 0, c->stream>>>(A, L, inv, n, p, d_info);
  }
  // (on a failed factor the inverse below works on partial data; the caller discards it)
  OEFE_COUNTED k_tri_inv<S><<<(n + CC - 1) / CC, CB * CC, 0, c->stream>>>(L, inv, Y, n);
  OEFE_CUDA_TRY(c, cudaGetLastError());
  OEFE_CUDA_TRY(c, cudaMemcpyAsync(info_host, d_info, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  OEFE_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return OEFE_OK;
}

template int chol_factor_inverse<double>(oefe_ctx*, double*, double*, double*, int, void*, int*, int*);
template int chol_factor_inverse<cd>(oefe_ctx*, cd*, cd*, cd*, int, void*, int*, int*);
