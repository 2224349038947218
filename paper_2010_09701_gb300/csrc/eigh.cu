// Dense FP64 generalized Hermitian eigensolver for the projected problem of
// Rayleigh-Ritz (Eq. ProjKS), H^Q u = eps M^Q u, entirely on the GPU:
//   M^Q = L L^+ (chol.cu), C = L^{-1} H^Q L^{-+}, C = W diag(eps) W^+ by a
//   parallel cyclic Jacobi method (circle ordering: n/2 disjoint rotations per
//   round, n-1 rounds per sweep), U = L^{-+} W, eigenvalues ascending. Real data
//   stays real throughout.
#include <algorithm>
#include <cmath>

#include "oefe_internal.h"

namespace {

constexpr int JT = 1024;
constexpr int MAXPAIRS = 512;   // n <= 1024
// matrices up to this size take the one-CTA sweeps (the grid barrier costs more than their updates)
constexpr int ONE_CTA_N = 24;

// one scalar interface over double and cd
__device__ __forceinline__ double s_re(double a) { return a; }
__device__ __forceinline__ double s_re(cd a) { return a.x; }
__device__ __forceinline__ double s_abs2(double a) { return a * a; }
__device__ __forceinline__ double s_abs2(cd a) { return cabs2(a); }
__device__ __forceinline__ double s_abs(double a) { return fabs(a); }
__device__ __forceinline__ double s_abs(cd a) { return sqrt(cabs2(a)); }
__device__ __forceinline__ double s_conj(double a) { return a; }
__device__ __forceinline__ cd s_conj(cd a) { return cconj(a); }
__device__ __forceinline__ double s_fma(double a, double b, double acc) { return fma(a, b, acc); }
__device__ __forceinline__ cd s_fma(cd a, cd b, cd acc) { return cfma(a, b, acc); }
__device__ __forceinline__ double s_num(double a, double) { return a; }
__device__ __forceinline__ cd s_num(double a, cd) { return mkc(a, 0.0); }
// x a + g b with x real
__device__ __forceinline__ double s_rot(double x, double a, double g, double b) { return fma(x, a, g * b); }
__device__ __forceinline__ cd s_rot(double x, cd a, cd g, cd b) {
  return mkc(fma(x, a.x, fma(g.x, b.x, -g.y * b.y)), fma(x, a.y, fma(g.x, b.y, g.y * b.x)));
}

__device__ inline double block_sum(double v, double* red) {
  const int tid = threadIdx.x;
  red[tid] = v;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (tid < w) red[tid] += red[tid + w];
    __syncthreads();
  }
  const double s = red[0];
  __syncthreads();
  return s;
}

// C = op(A) op(B), n x n; op = conjugate transpose when the flag is set
template <typename S>
__global__ void k_small_gemm(const S* A, bool ca, const S* B, bool cb, S* C, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * n) return;
  const int i = t / n, j = t % n;
  S s = s_num(0.0, S{});
  for (int k = 0; k < n; ++k) {
    const S a = ca ? s_conj(A[(size_t)k * n + i]) : A[(size_t)i * n + k];
    const S b = cb ? s_conj(B[(size_t)j * n + k]) : B[(size_t)k * n + j];
    s = s_fma(a, b, s);
  }
  C[t] = s;
}

// B = the Hermitian part of A
template <typename S>
__global__ void k_hermitian_part(const S* A, S* B, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * n) return;
  const int i = t / n, j = t % n;
  if (i > j) return;
  const S v = 0.5 * (A[(size_t)i * n + j] + s_conj(A[(size_t)j * n + i]));
  B[(size_t)i * n + j] = v;
  B[(size_t)j * n + i] = s_conj(v);
}

// The rotation of pair k of round r of the circle method (m players, player n a bye when n is odd):
// its indices, cosine, sine and the phase of the entry it annihilates; identity when there is none.
template <typename S>
struct JRot {
  int p, q;   // p < q; q >= n: the bye
  double c, s;
  S g10, g11;  // G = [[c, s], [g10, g11]] = [[c, s], [-conj(u) s, conj(u) c]]
};
template <typename S, typename LD>
__device__ __forceinline__ JRot<S> jacobi_rotation(int n, int m, int r, int k, LD at) {
  // position 0 holds player m-1, position i holds (i - 1 + r) mod (m - 1)
  const int a = k == 0 ? m - 1 : (k - 1 + r) % (m - 1);
  const int b = (m - 1 - k - 1 + r) % (m - 1);
  JRot<S> o;
  o.p = min(a, b);
  o.q = max(a, b);
  o.c = 1.0;
  o.s = 0.0;
  o.g10 = s_num(0.0, S{});
  o.g11 = s_num(1.0, S{});
  if (o.q < n) {
    const S bpq = at(o.p, o.q);
    const double beta = s_abs(bpq);
    if (beta >= 1e-300) {
      const S u = (1.0 / beta) * bpq;
      const double tau = (s_re(at(o.q, o.q)) - s_re(at(o.p, o.p))) / (2.0 * beta);
      const double tt = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
      o.c = 1.0 / sqrt(1.0 + tt * tt);
      o.s = tt * o.c;
      const S ub = s_conj(u);
      o.g10 = (-o.s) * ub;
      o.g11 = o.c * ub;
    }
  }
  return o;
}

// Jacobi sweeps of a small matrix by one CTA, A and V (from the identity) in shared memory.
template <typename S>
__global__ void __launch_bounds__(JT) k_jacobi(S* Ag, S* Vg, int n, int max_sweeps, double tol) {
  extern __shared__ double jsm[];
  S* A = reinterpret_cast<S*>(jsm);
  S* V = A + (size_t)n * n;
  __shared__ double red[JT];
  __shared__ JRot<S> rot[ONE_CTA_N / 2];
  const int tid = threadIdx.x;
  const int m = n + (n & 1), np = m / 2;
  double fro = 0;
  for (int t = tid; t < n * n; t += JT) {
    A[t] = Ag[t];
    V[t] = s_num(t / n == t % n ? 1.0 : 0.0, S{});
    fro += s_abs2(A[t]);
  }
  fro = block_sum(fro, red);
  for (int sweep = 0; sweep < max_sweeps; ++sweep) {
    double off = 0;
    for (int t = tid; t < n * n; t += JT)
      if (t / n != t % n) off += s_abs2(A[t]);
    off = block_sum(off, red);
    if (off <= tol * tol * fro || off == 0.0) break;
    for (int r = 0; r < m - 1; ++r) {
      for (int k = tid; k < np; k += JT)
        rot[k] = jacobi_rotation<S>(n, m, r, k, [&](int i, int j) { return A[(size_t)i * n + j]; });
      __syncthreads();
      for (int t = tid; t < np * n; t += JT) {   // rows: A <- G^+ A (disjoint rows)
        const JRot<S>& g = rot[t / n];
        const int j = t % n;
        if (g.q >= n) continue;
        const S ap = A[(size_t)g.p * n + j], aq = A[(size_t)g.q * n + j];
        A[(size_t)g.p * n + j] = s_rot(g.c, ap, s_conj(g.g10), aq);
        A[(size_t)g.q * n + j] = s_rot(g.s, ap, s_conj(g.g11), aq);
      }
      __syncthreads();
      for (int t = tid; t < np * n; t += JT) {   // columns: A <- A G, V <- V G
        const JRot<S>& g = rot[t / n];
        const int i = t % n;
        if (g.q >= n) continue;
        const S ap = A[(size_t)i * n + g.p], aq = A[(size_t)i * n + g.q];
        const bool own = g.s != 0.0;             // the annihilated entries are exactly zero
        A[(size_t)i * n + g.p] = own && i == g.q ? s_num(0.0, S{}) : s_rot(g.c, ap, g.g10, aq);
        A[(size_t)i * n + g.q] = own && i == g.p ? s_num(0.0, S{}) : s_rot(g.s, ap, g.g11, aq);
        const S vp = V[(size_t)i * n + g.p], vq = V[(size_t)i * n + g.q];
        V[(size_t)i * n + g.p] = s_rot(g.c, vp, g.g10, vq);
        V[(size_t)i * n + g.q] = s_rot(g.s, vp, g.g11, vq);
      }
      __syncthreads();
    }
  }
  for (int t = tid; t < n * n; t += JT) {
    Ag[t] = A[t];
    Vg[t] = V[t];
  }
}

// ---- the same method for larger matrices, spread over the GPU by one cooperative launch.
// Bound: (n - 1) rounds a sweep, each a chain of an L2 round trip, a rotation (three divisions and
// two square roots on the FP64 pipe) and a grid barrier; the arithmetic itself is small. So one
// launch runs every sweep, every CTA forms all of a round's rotations itself (no barrier between
// parameters and updates), A ping-pongs between two buffers (no barrier between readers and writers
// of a round: one per round), and each CTA keeps its rows of V in shared memory (they depend on no
// other CTA). Three launches per round took 20 us a round (71 ms for the 360 real columns of the
// 62-atom cell), and one CTA 13 us a round at 64 complex columns (7.6 ms).
constexpr int GJ = 256;              // threads per CTA
constexpr long long GJ_SPIN = 1ll << 24;

struct GridBar {
  unsigned* count;     // zeroed before the launch
  int* fail;
};
// all CTAs of the cooperative launch; false (in every thread of the CTA) when the wait gave up
__device__ inline bool grid_barrier(const GridBar& b, unsigned target) {
  __shared__ int ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(b.count, 1u);
    int good = 0;
    for (long long i = 0; i < GJ_SPIN; ++i) {
      unsigned v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(b.count) : "memory");
      if (v >= target) { good = 1; break; }
      if ((i & 1023) == 1023 && *(volatile int*)b.fail) break;
    }
    if (!good) atomicExch(b.fail, 1);
    __threadfence();
    ok = good;
  }
  __syncthreads();
  return ok != 0;
}

__device__ __forceinline__ double ld_l2(const double* p) { return __ldcg(p); }
__device__ __forceinline__ cd ld_l2(const cd* p) {
  const double2 v = __ldcg(reinterpret_cast<const double2*>(p));
  return mkc(v.x, v.y);
}

template <typename S>
__global__ void __launch_bounds__(GJ) k_jacobi_grid(S* A0, S* A1, S* Vg, int n, int max_sweeps, double tol2,
                                                    double* part, GridBar bar) {
  extern __shared__ double jsm[];
  const int m = n + (n & 1), np = m / 2, G = gridDim.x, tid = threadIdx.x;
  JRot<S>* rot = reinterpret_cast<JRot<S>*>(jsm);
  S* V = reinterpret_cast<S*>(rot + np);
  const int nrow = (n - (int)blockIdx.x + G - 1) / G;   // rows blockIdx.x, blockIdx.x + G, ..
  __shared__ double red[GJ];
  for (int t = tid; t < nrow * n; t += GJ)
    V[t] = s_num((int)blockIdx.x + (t / n) * G == t % n ? 1.0 : 0.0, S{});
  unsigned arrivals = 0;
  double fro = -1.0;
  S *A = A0, *B = A1;
  bool ok = true;
  for (int sweep = 0; sweep < max_sweeps && ok; ++sweep) {
    double off = 0, all = 0;
    for (int i = blockIdx.x; i < n; i += G)
      for (int j = tid; j < n; j += GJ) {
        const double v = s_abs2(ld_l2(A + (size_t)i * n + j));
        all += v;
        if (i != j) off += v;
      }
    off = block_sum(off, red);
    all = block_sum(all, red);
    double* ps = part + (size_t)(sweep & 1) * 2 * G;
    if (tid == 0) {
      ps[2 * blockIdx.x] = off;
      ps[2 * blockIdx.x + 1] = all;
    }
    if (!(ok = grid_barrier(bar, arrivals += G))) break;
    off = all = 0;
    for (int b = tid; b < G; b += GJ) {   // the same sums in every CTA, so all take the same decision
      off += __ldcg(ps + 2 * b);
      all += __ldcg(ps + 2 * b + 1);
    }
    off = block_sum(off, red);
    all = block_sum(all, red);
    if (fro < 0) fro = all;
    if (off <= tol2 * fro || off == 0.0) break;
    for (int r = 0; r < m - 1 && ok; ++r) {
      for (int k = tid; k < np; k += GJ)
        rot[k] = jacobi_rotation<S>(n, m, r, k, [&](int i, int j) { return ld_l2(A + (size_t)i * n + j); });
      __syncthreads();
      // 2x2 blocks of A (rows of pair kr, columns of pair kc): rows, then columns
      for (int t = blockIdx.x + G * tid; t < np * np; t += G * GJ) {
        const int kr = t / np, kc = t % np;
        const JRot<S>&gr = rot[kr], &gc = rot[kc];
        const int ri[2] = {gr.p, gr.q}, ci[2] = {gc.p, gc.q};
        S x[2][2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j)
            x[i][j] = ri[i] < n && ci[j] < n ? ld_l2(A + (size_t)ri[i] * n + ci[j]) : s_num(0.0, S{});
        if (ri[1] < n) {
          const S h10 = s_conj(gr.g10), h11 = s_conj(gr.g11);
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const S xp = x[0][j], xq = x[1][j];
            x[0][j] = s_rot(gr.c, xp, h10, xq);
            x[1][j] = s_rot(gr.s, xp, h11, xq);
          }
        }
        if (ci[1] < n) {
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const S yp = x[i][0], yq = x[i][1];
            x[i][0] = s_rot(gc.c, yp, gc.g10, yq);
            x[i][1] = s_rot(gc.s, yp, gc.g11, yq);
          }
        }
        if (kr == kc && gr.s != 0.0) x[0][1] = x[1][0] = s_num(0.0, S{});
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (ri[i] < n && ci[j] < n) B[(size_t)ri[i] * n + ci[j]] = x[i][j];
      }
      for (int t = tid; t < nrow * np; t += GJ) {   // this CTA's rows of V
        const JRot<S>& g = rot[t % np];
        if (g.q >= n) continue;
        S* v = V + (size_t)(t / np) * n;
        const S vp = v[g.p], vq = v[g.q];
        v[g.p] = s_rot(g.c, vp, g.g10, vq);
        v[g.q] = s_rot(g.s, vp, g.g11, vq);
      }
      ok = grid_barrier(bar, arrivals += G);
      S* t = A;
      A = B;
      B = t;
    }
  }
  __syncthreads();
  for (int t = tid; t < nrow * n; t += GJ) Vg[((size_t)blockIdx.x + (size_t)(t / n) * G) * n + t % n] = V[t];
  // the diagonal form into A0 (this CTA's rows; the last barrier ordered them)
  if (A != A0)
    for (int i = blockIdx.x; i < n; i += G)
      for (int j = tid; j < n; j += GJ) A0[(size_t)i * n + j] = ld_l2(A + (size_t)i * n + j);
}

// ascending order: rank of each diagonal entry (ties by index), then permute
template <typename S>
__global__ void k_sort_eig(const S* A, const S* W, int n, double* eps, S* Wsorted) {
  const int i = blockIdx.x;
  const double wi = s_re(A[(size_t)i * n + i]);
  __shared__ int rank;
  if (threadIdx.x == 0) rank = 0;
  __syncthreads();
  int mine = 0;
  for (int j = threadIdx.x; j < n; j += blockDim.x) {
    const double wj = s_re(A[(size_t)j * n + j]);
    if (wj < wi || (wj == wi && j < i)) ++mine;
  }
  if (mine) atomicAdd(&rank, mine);
  __syncthreads();
  if (threadIdx.x == 0) eps[rank] = wi;
  for (int r = threadIdx.x; r < n; r += blockDim.x) Wsorted[(size_t)r * n + rank] = W[(size_t)r * n + i];
}

}  // namespace

// H, M: device n x n (double or cd). eps: host n. U: device n x n (same type).
// Returns OEFE_ERR_CHOLESKY if M is not positive definite. Scratch: the context's ws.
template <typename S>
int gpu_geneig(oefe_ctx* c, const S* H, const S* M, int n, double* eps_host, S* U) {
  if (n > 2 * MAXPAIRS) { c->err = "eigensolver: n too large"; return OEFE_ERR_ARG; }
  auto a256 = [](size_t x) { return ((x + 255) / 256) * 256; };
  const size_t nn = (size_t)n * n, nb = a256(nn * sizeof(S));
  const size_t sb = a256(chol_scratch(n, sizeof(S))), eb = a256((size_t)n * sizeof(double));
  const size_t pb = a256((size_t)4 * c->num_sms * sizeof(double));
  OEFE_TRY(ensure_ws(c, 6 * nb + sb + eb + pb + 256));
  char* p = (char*)c->ws;
  S *Hc = (S*)p, *Mc = (S*)(p + nb), *Y = (S*)(p + 2 * nb), *T = (S*)(p + 3 * nb), *W = (S*)(p + 4 * nb),
    *Ws = (S*)(p + 5 * nb);
  void* scr = p + 6 * nb;
  double* d_eps = (double*)(p + 6 * nb + sb);
  double* d_part = (double*)(p + 6 * nb + sb + eb);
  GridBar bar{(unsigned*)(p + 6 * nb + sb + eb + pb), (int*)(p + 6 * nb + sb + eb + pb) + 1};
  const int b = 256, g = (int)((nn + b - 1) / b);
  OEFE_COUNTED k_hermitian_part<S><<<g, b, 0, c->stream>>>(H, Hc, n);
  OEFE_COUNTED k_hermitian_part<S><<<g, b, 0, c->stream>>>(M, Mc, n);
  int info = 0;
  OEFE_TRY(chol_factor_inverse<S>(c, Mc, T, Y, n, scr, c->d_status + 3, &info));   // Y = L^{-1}
  if (info != 0) {
    c->err = "rayleigh_ritz: projected overlap not positive definite";
    return OEFE_ERR_CHOLESKY;
  }
  OEFE_COUNTED k_small_gemm<S><<<g, b, 0, c->stream>>>(Y, false, Hc, false, T, n);  // T = L^{-1} H
  OEFE_COUNTED k_small_gemm<S><<<g, b, 0, c->stream>>>(T, false, Y, true, Mc, n);   // C = T L^{-+}
  OEFE_COUNTED k_hermitian_part<S><<<g, b, 0, c->stream>>>(Mc, Hc, n);
  OEFE_CUDA_TRY(c, cudaGetLastError());
  int fail = 0;
  if (n <= ONE_CTA_N) {
    OEFE_COUNTED k_jacobi<S><<<1, JT, 2 * nn * sizeof(S), c->stream>>>(Hc, W, n, 40, 1e-15);
  } else {
    const int m = n + (n & 1), np = m / 2;
    // 16 blocks of A per CTA: enough CTAs that the FP64 updates take less than the barrier
    const int grid = std::max(1, std::min(c->num_sms, np * np / 16));
    const size_t smem = (size_t)np * sizeof(JRot<S>) + (size_t)((n + grid - 1) / grid) * n * sizeof(S);
    OEFE_CUDA_TRY(c, cudaFuncSetAttribute(k_jacobi_grid<S>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    OEFE_CUDA_TRY(c, cudaMemsetAsync(bar.count, 0, 8, c->stream));
    int sweeps = 40;
    double tol2 = 1e-30;
    S *A1 = Mc, *A0 = Hc, *Vp = W;
    void* args[] = {&A0, &A1, &Vp, (void*)&n, &sweeps, &tol2, &d_part, &bar};
    OEFE_CUDA_TRY(c, cudaLaunchCooperativeKernel((const void*)k_jacobi_grid<S>, dim3(grid), dim3(GJ), args, smem, c->stream));
    oefe_launch_add(1);
    OEFE_CUDA_TRY(c, cudaMemcpyAsync(&fail, bar.fail, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  }
  OEFE_COUNTED k_sort_eig<S><<<n, 128, 0, c->stream>>>(Hc, W, n, d_eps, Ws);
  OEFE_COUNTED k_small_gemm<S><<<g, b, 0, c->stream>>>(Y, true, Ws, false, U, n);   // U = L^{-+} W
  OEFE_CUDA_TRY(c, cudaGetLastError());
  OEFE_CUDA_TRY(c, cudaMemcpyAsync(eps_host, d_eps, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream));
  OEFE_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  if (fail) { c->err = "eigensolver: a grid barrier timed out"; return OEFE_ERR_TIMEOUT; }
  return OEFE_OK;
}

template int gpu_geneig<double>(oefe_ctx*, const double*, const double*, int, double*, double*);
template int gpu_geneig<cd>(oefe_ctx*, const cd*, const cd*, int, double*, cd*);

// eigenvalues of a real symmetric tridiagonal (Lanczos) matrix, ascending
int gpu_tridiag_eig(oefe_ctx* c, const std::vector<double>& al, const std::vector<double>& be, std::vector<double>& w) {
  const int m = (int)al.size();
  std::vector<double> T((size_t)m * m, 0.0), I((size_t)m * m, 0.0);
  for (int i = 0; i < m; ++i) {
    T[(size_t)i * m + i] = al[i];
    I[(size_t)i * m + i] = 1.0;
    if (i + 1 < m) T[(size_t)i * m + i + 1] = T[(size_t)(i + 1) * m + i] = be[i];
  }
  double *dT = nullptr;
  OEFE_TRY(dev_alloc(c, (void**)&dT, 3 * (size_t)m * m * sizeof(double)));
  cudaMemcpyAsync(dT, T.data(), T.size() * sizeof(double), cudaMemcpyHostToDevice, c->stream);
  cudaMemcpyAsync(dT + (size_t)m * m, I.data(), I.size() * sizeof(double), cudaMemcpyHostToDevice, c->stream);
  w.assign(m, 0.0);
  const int st = gpu_geneig<double>(c, dT, dT + (size_t)m * m, m, w.data(), dT + 2 * (size_t)m * m);
  cudaStreamSynchronize(c->stream);
  dev_free(dT);
  return st;
}
