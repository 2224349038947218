// Dense FP64 generalized Hermitian eigensolver for the projected problem of
// Rayleigh-Ritz (Eq. ProjKS), H^Q u = eps M^Q u, entirely on the GPU:
//   M^Q = L L^+ (Cholesky), C = L^{-1} H^Q L^{-+}, C = W diag(eps) W^+ by a
//   parallel cyclic Jacobi method (circle ordering: n/2 disjoint rotations per
//   round, n-1 rounds per sweep), U = L^{-+} W, eigenvalues ascending.
#include <algorithm>
#include <cmath>

#include "oefe_internal.h"
#include "pair_dev.cuh"

namespace {

constexpr int JT = 1024;
constexpr int MAXN = 1024;
// one CTA takes matrices up to this size: A and V in its shared memory (204800 bytes) beside the rotations and
// the reduction (9792)
constexpr int CTA_N = 80;

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

// C = op(A) op(B), n x n complex; op = conjugate transpose when the flag is set
__global__ void k_small_gemm(const cd* A, bool ca, const cd* B, bool cb, cd* C, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * n) return;
  const int i = t / n, j = t % n;
  cd s = mkc(0, 0);
  for (int k = 0; k < n; ++k) {
    const cd a = ca ? cconj(A[(size_t)k * n + i]) : A[(size_t)i * n + k];
    const cd b = cb ? cconj(B[(size_t)j * n + k]) : B[(size_t)k * n + j];
    s += a * b;
  }
  C[t] = s;
}

__global__ void k_hermitian_part(cd* A, int n) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n * n) return;
  const int i = t / n, j = t % n;
  if (i > j) return;
  const cd v = 0.5 * (A[(size_t)i * n + j] + cconj(A[(size_t)j * n + i]));
  A[(size_t)i * n + j] = v;
  A[(size_t)j * n + i] = cconj(v);
}

// Jacobi sweeps on A (n x n Hermitian, overwritten by its diagonal form), V <- eigenvectors.
// One CTA, A and V in shared memory.
// init_v: start from V = I; otherwise from the V given (the sweeps continue an earlier phase).
__global__ void __launch_bounds__(JT) k_jacobi(cd* Ag, cd* Vg, int n, int max_sweeps, double tol, int* sweeps_out,
                                               bool init_v) {
  extern __shared__ cd jsm[];
  cd* A = jsm;
  cd* V = jsm + (size_t)n * n;
  {
    for (int t = threadIdx.x; t < n * n; t += JT) {
      A[t] = Ag[t];
      if (!init_v) V[t] = Vg[t];
    }
    __syncthreads();
  }
  __shared__ double red[JT];
  __shared__ double cs_[CTA_N / 2], sn_[CTA_N / 2];
  __shared__ cd u_[CTA_N / 2];
  __shared__ int p_[CTA_N / 2], q_[CTA_N / 2];
  const int tid = threadIdx.x;
  const int m = n + (n & 1);  // even number of players; player n is a bye when n is odd
  const int np = m / 2;
  if (init_v)
    for (int t = tid; t < n * n; t += JT) V[t] = (t / n == t % n) ? mkc(1, 0) : mkc(0, 0);
  double fro = 0;
  for (int t = tid; t < n * n; t += JT) fro += cabs2(A[t]);
  fro = block_sum(fro, red);
  int sweep = 0;
  for (; sweep < max_sweeps; ++sweep) {
    double off = 0;
    for (int t = tid; t < n * n; t += JT)
      if (t / n != t % n) off += cabs2(A[t]);
    off = block_sum(off, red);
    if (off <= tol * tol * fro || off == 0.0) break;
    for (int r = 0; r < m - 1; ++r) {
      for (int k = tid; k < np; k += JT) {
        // circle method: position 0 holds player m-1, position i holds (i - 1 + r) mod (m - 1)
        const int a = k == 0 ? m - 1 : (k - 1 + r) % (m - 1);
        const int b = (m - 1 - k - 1 + r) % (m - 1);
        int p = min(a, b), q = max(a, b);
        if (q >= n) { p_[k] = -1; continue; }
        const cd bpq = A[(size_t)p * n + q];
        const double beta = sqrt(cabs2(bpq));
        if (beta < 1e-300) { p_[k] = -1; continue; }
        const cd u = (1.0 / beta) * bpq;
        const double tau = (A[(size_t)q * n + q].x - A[(size_t)p * n + p].x) / (2.0 * beta);
        const double tt = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
        const double c = 1.0 / sqrt(1.0 + tt * tt);
        p_[k] = p;
        q_[k] = q;
        cs_[k] = c;
        sn_[k] = tt * c;
        u_[k] = u;
      }
      __syncthreads();
      // rows: A <- G^+ A for every pair (disjoint rows)
      for (int t = tid; t < np * n; t += JT) {
        const int k = t / n, j = t % n;
        const int p = p_[k];
        if (p < 0) continue;
        const int q = q_[k];
        const double c = cs_[k], s = sn_[k];
        const cd ub = cconj(u_[k]);
        // G = [[c, s], [-conj(u) s, conj(u) c]]
        const cd g10 = -s * ub, g11 = c * ub;
        const cd apj = A[(size_t)p * n + j], aqj = A[(size_t)q * n + j];
        A[(size_t)p * n + j] = c * apj + cmulc(g10, aqj);
        A[(size_t)q * n + j] = s * apj + cmulc(g11, aqj);
      }
      __syncthreads();
      // columns: A <- A G, V <- V G
      for (int t = tid; t < np * n; t += JT) {
        const int k = t / n, i = t % n;
        const int p = p_[k];
        if (p < 0) continue;
        const int q = q_[k];
        const double c = cs_[k], s = sn_[k];
        const cd ub = cconj(u_[k]);
        const cd g10 = -s * ub, g11 = c * ub;
        const cd aip = A[(size_t)i * n + p], aiq = A[(size_t)i * n + q];
        A[(size_t)i * n + p] = c * aip + aiq * g10;
        A[(size_t)i * n + q] = s * aip + aiq * g11;
        const cd vip = V[(size_t)i * n + p], viq = V[(size_t)i * n + q];
        V[(size_t)i * n + p] = c * vip + viq * g10;
        V[(size_t)i * n + q] = s * vip + viq * g11;
      }
      __syncthreads();
      for (int k = tid; k < np; k += JT) {
        const int p = p_[k];
        if (p < 0) continue;
        A[(size_t)p * n + q_[k]] = mkc(0, 0);
        A[(size_t)q_[k] * n + p] = mkc(0, 0);
      }
      __syncthreads();
    }
  }
  if (tid == 0) *sweeps_out = sweep;
  {
    __syncthreads();
    for (int t = threadIdx.x; t < n * n; t += JT) {
      Ag[t] = A[t];
      Vg[t] = V[t];
    }
  }
}


// ---- FP32-pair elements (pair_dev.cuh): the sweeps of pair mode on the FP32 pipe
struct alignas(16) c2j {
  f2 r, i;
};
__device__ __forceinline__ c2j c2j_from(cd a) { return c2j{f2_from(a.x), f2_from(a.y)}; }
__device__ __forceinline__ cd c2j_to(c2j a) { return mkc(f2_to(a.r), f2_to(a.i)); }
// x a + conj(g) b
__device__ __forceinline__ c2j rot_c(f2 x, c2j a, c2j g, c2j b) {
  f2acc r{0.0f, 0.0f}, i{0.0f, 0.0f};
  f2_mac(r, x, a.r);
  f2_mac(r, g.r, b.r);
  f2_mac(r, g.i, b.i);
  f2_mac(i, x, a.i);
  f2_mac(i, g.r, b.i);
  f2_mac(i, f2_neg(g.i), b.r);
  return c2j{f2_fin(r), f2_fin(i)};
}
// x a + b g
__device__ __forceinline__ c2j rot_n(f2 x, c2j a, c2j b, c2j g) {
  f2acc r{0.0f, 0.0f}, i{0.0f, 0.0f};
  f2_mac(r, x, a.r);
  f2_mac(r, b.r, g.r);
  f2_mac(r, f2_neg(b.i), g.i);
  f2_mac(i, x, a.i);
  f2_mac(i, b.r, g.i);
  f2_mac(i, b.i, g.r);
  return c2j{f2_fin(r), f2_fin(i)};
}
__device__ __forceinline__ cd rot_c(double x, cd a, cd g, cd b) { return x * a + cmulc(g, b); }
__device__ __forceinline__ cd rot_n(double x, cd a, cd b, cd g) { return x * a + b * g; }

__device__ __forceinline__ cd e_to(cd a) { return a; }
__device__ __forceinline__ cd e_to(c2j a) { return c2j_to(a); }
template <typename E>
__device__ __forceinline__ E e_from(cd a);
template <>
__device__ __forceinline__ cd e_from<cd>(cd a) { return a; }
template <>
__device__ __forceinline__ c2j e_from<c2j>(cd a) { return c2j_from(a); }
template <typename E>
struct Real;
template <>
struct Real<cd> {
  using type = double;
  static __device__ __forceinline__ double from(double x) { return x; }
};
template <>
struct Real<c2j> {
  using type = f2;
  static __device__ __forceinline__ f2 from(double x) { return f2_from(x); }
};

// ---- the same cyclic Jacobi method spread over the GPU by one cooperative launch, in FP64 (E = cd) or in
// pairs (E = c2j, rotations taken in FP64 from the current entries).
// Bound: (n - 1) rounds a sweep, each a chain of an L2 round trip, a rotation (divisions and square roots
// on the FP64 pipe), the updates and a grid barrier. So one launch runs every sweep, A ping-pongs between
// two buffers (no barrier between readers and writers of a round), each CTA keeps its rows of V in shared
// memory (they depend on no other CTA), and each thread takes a 2x2 block of A (rows of one pair,
// columns of another: they commute with every other block's). Same rotations and same arithmetic per entry
// as k_jacobi (rows first, then columns, the rotated pair's off-diagonal entries set to zero).
// Three launches per round took 20 us a round (71 ms for the 360 real columns of the 62-atom cell), and
// one CTA 13 us a round at 64 complex columns (7.6 ms); this takes 46 and 3.6 ms.
constexpr int GJ = 256;              // threads per CTA
constexpr long long GJ_SPIN = 1ll << 24;
// pairs up to which every CTA forms all rotations of a round itself; above, they are shared out and a second
// barrier publishes them (100 FP64 operations each, two a clock per SM: 180 of them take 5 us, a
// barrier 2 us)
constexpr int GJ_OWN = 64;
// matrices up to this size take the one-CTA sweeps (the grid barrier costs more than their updates)
constexpr int ONE_CTA_N = 24;

template <typename E>
struct JRot {
  int p, q;     // the pair's indices p < q (q >= n: the bye of an odd n)
  int rot;      // 1 when the pair rotates
  typename Real<E>::type c, s;
  E g10, g11;   // G = [[c, s], [g10, g11]] = [[c, s], [-conj(u) s, conj(u) c]]
};

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

// 16 bytes through L2 (other CTAs' writes of an earlier round)
template <typename E>
__device__ __forceinline__ E ld_l2(const E* p) {
  static_assert(sizeof(E) == 16, "16-byte elements");
  const int4 v = __ldcg(reinterpret_cast<const int4*>(p));
  return *reinterpret_cast<const E*>(&v);
}

template <typename E>
__device__ JRot<E> jacobi_rotation(const E* A, int n, int r, int k) {
  const int m = n + (n & 1);
  const int a = k == 0 ? m - 1 : (k - 1 + r) % (m - 1);
  const int b = (m - 1 - k - 1 + r) % (m - 1);
  JRot<E> o;
  o.p = min(a, b);
  o.q = max(a, b);
  o.rot = 0;
  if (o.q < n) {
    const int p = o.p, q = o.q;
    const E epq = ld_l2(A + (size_t)p * n + q), epp = ld_l2(A + (size_t)p * n + p), eqq = ld_l2(A + (size_t)q * n + q);
    const cd bpq = e_to(epq);
    const double beta = sqrt(cabs2(bpq));
    if (beta >= 1e-300) {
      const cd u = (1.0 / beta) * bpq;
      const double tau = (e_to(eqq).x - e_to(epp).x) / (2.0 * beta);
      const double tt = (tau >= 0 ? 1.0 : -1.0) / (fabs(tau) + sqrt(1.0 + tau * tau));
      const double c = 1.0 / sqrt(1.0 + tt * tt), s = tt * c;
      const cd ub = cconj(u);
      o.c = Real<E>::from(c);
      o.s = Real<E>::from(s);
      o.g10 = e_from<E>(-s * ub);
      o.g11 = e_from<E>(c * ub);
      o.rot = 1;
    }
  }
  return o;
}

template <typename E>
__global__ void __launch_bounds__(GJ) k_jacobi_grid(E* A0, E* A1, E* Vg, int n, int max_sweeps, double tol2, double* part,
                                                    JRot<E>* rot_g, GridBar bar) {
  extern __shared__ __align__(16) unsigned char jg_raw[];
  const int m = n + (n & 1), np = m / 2, G = gridDim.x, tid = threadIdx.x;
  E* V = reinterpret_cast<E*>(jg_raw);
  const int nrow = (n - (int)blockIdx.x + G - 1) / G;   // rows blockIdx.x, blockIdx.x + G, ..
  JRot<E>* rot = reinterpret_cast<JRot<E>*>(V + (size_t)((n + G - 1) / G) * n);
  __shared__ double red[GJ];
  for (int t = tid; t < nrow * n; t += GJ) V[t] = e_from<E>(mkc((int)blockIdx.x + (t / n) * G == t % n ? 1.0 : 0.0, 0.0));
  unsigned arrivals = 0;
  double fro = -1.0;
  E *A = A0, *B = A1;
  bool ok = true;
  auto sum = [&](double v) {   // over the CTA, in every thread
    red[tid] = v;
    __syncthreads();
    for (int w = GJ / 2; w > 0; w >>= 1) {
      if (tid < w) red[tid] += red[tid + w];
      __syncthreads();
    }
    const double s = red[0];
    __syncthreads();
    return s;
  };
  for (int sweep = 0; sweep < max_sweeps && ok; ++sweep) {
    double off = 0, all = 0;
    for (int i = blockIdx.x; i < n; i += G)
      for (int j = tid; j < n; j += GJ) {
        const double v = cabs2(e_to(ld_l2(A + (size_t)i * n + j)));
        all += v;
        if (i != j) off += v;
      }
    off = sum(off);
    all = sum(all);
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
    off = sum(off);
    all = sum(all);
    if (fro < 0) fro = all;
    if (off <= tol2 * fro || off == 0.0) break;
    for (int r = 0; r < m - 1 && ok; ++r) {
      if (np <= GJ_OWN) {
        for (int k = tid; k < np; k += GJ) rot[k] = jacobi_rotation<E>(A, n, r, k);
      } else {
        // (the readers of the last round's rotations passed the barrier at its end)
        if (tid < 2 && (int)blockIdx.x + tid * G < np) {
          const int k = blockIdx.x + tid * G;
          const JRot<E> o = jacobi_rotation<E>(A, n, r, k);
          rot_g[k] = o;
        }
        for (int k = blockIdx.x + (2 + tid) * G; k < np; k += GJ * G) rot_g[k] = jacobi_rotation<E>(A, n, r, k);
        if (!(ok = grid_barrier(bar, arrivals += G))) break;
        const int4* src = reinterpret_cast<const int4*>(rot_g);
        for (int t = tid; t < np * (int)(sizeof(JRot<E>) / 16); t += GJ) reinterpret_cast<int4*>(rot)[t] = __ldcg(src + t);
      }
      __syncthreads();
      for (int t = blockIdx.x + G * tid; t < np * np; t += G * GJ) {
        const int kr = t / np, kc = t % np;
        const JRot<E>&gr = rot[kr], &gc = rot[kc];
        const int ri[2] = {gr.p, gr.q}, ci[2] = {gc.p, gc.q};
        E x[2][2];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j)
            x[i][j] = ri[i] < n && ci[j] < n ? ld_l2(A + (size_t)ri[i] * n + ci[j]) : e_from<E>(mkc(0, 0));
        if (gr.rot) {   // rows
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const E xp = x[0][j], xq = x[1][j];
            x[0][j] = rot_c(gr.c, xp, gr.g10, xq);
            x[1][j] = rot_c(gr.s, xp, gr.g11, xq);
          }
        }
        if (gc.rot) {   // columns
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const E yp = x[i][0], yq = x[i][1];
            x[i][0] = rot_n(gc.c, yp, yq, gc.g10);
            x[i][1] = rot_n(gc.s, yp, yq, gc.g11);
          }
        }
        if (kr == kc && gr.rot) x[0][1] = x[1][0] = e_from<E>(mkc(0, 0));
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int j = 0; j < 2; ++j)
            if (ri[i] < n && ci[j] < n) B[(size_t)ri[i] * n + ci[j]] = x[i][j];
      }
      for (int t = tid; t < nrow * np; t += GJ) {   // this CTA's rows of V
        const JRot<E>& g = rot[t % np];
        if (!g.rot) continue;
        E* v = V + (size_t)(t / np) * n;
        const E vp = v[g.p], vq = v[g.q];
        v[g.p] = rot_n(g.c, vp, vq, g.g10);
        v[g.q] = rot_n(g.s, vp, vq, g.g11);
      }
      ok = grid_barrier(bar, arrivals += G);
      E* t = A;
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

// to pairs and back, in place (16 bytes either way)
__global__ void k_to_pairs(cd* A, int n2) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t < n2) reinterpret_cast<c2j*>(A)[t] = c2j_from(A[t]);
}
__global__ void k_from_pairs(cd* A, cd* B, int n2) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n2) return;
  A[t] = c2j_to(reinterpret_cast<const c2j*>(A)[t]);
  B[t] = c2j_to(reinterpret_cast<const c2j*>(B)[t]);
}

// ascending order: rank of each diagonal entry (ties by index), then permute
__global__ void k_sort_eig(const cd* A, const cd* W, int n, double* eps, cd* Wsorted) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double wi = A[(size_t)i * n + i].x;
  int rank = 0;
  for (int j = 0; j < n; ++j) {
    const double wj = A[(size_t)j * n + j].x;
    if (wj < wi || (wj == wi && j < i)) ++rank;
  }
  eps[rank] = wi;
  for (int r = 0; r < n; ++r) Wsorted[(size_t)r * n + rank] = W[(size_t)r * n + i];
}

template <typename S>
__global__ void k_to_cd(const S* A, cd* B, int n2) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n2) return;
  if constexpr (sizeof(S) == sizeof(cd)) B[t] = reinterpret_cast<const cd*>(A)[t];
  else B[t] = mkc(reinterpret_cast<const double*>(A)[t], 0.0);
}

template <typename S>
__global__ void k_from_cd(const cd* B, S* A, int n2) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= n2) return;
  if constexpr (sizeof(S) == sizeof(cd)) reinterpret_cast<cd*>(A)[t] = B[t];
  else reinterpret_cast<double*>(A)[t] = B[t].x;
}

}  // namespace

// H, M: device n x n (double or cd). eps: host n. U: device n x n (same type).
// Returns OEFE_ERR_CHOLESKY if M is not positive definite.
template <typename S>
int gpu_geneig(oefe_ctx* c, const S* H, const S* M, int n, double* eps_host, S* U) {
  if (n > MAXN) { c->err = "eigensolver: n too large"; return OEFE_ERR_ARG; }
  const size_t nn = (size_t)n * n;
  auto a256 = [](size_t x) { return ((x + 255) / 256) * 256; };
  const size_t nb = a256(nn * sizeof(cd)), eb = a256((size_t)n * sizeof(double)), cb = a256(chol_scratch(n));
  const size_t pb = a256((size_t)4 * c->num_sms * sizeof(double));
  OEFE_TRY(ensure_ws(c, 6 * nb + eb + cb + pb + 256));
  char* w = (char*)c->ws;
  cd *Hc = (cd*)w, *Mc = (cd*)(w + nb), *Y = (cd*)(w + 2 * nb), *T = (cd*)(w + 3 * nb), *W = (cd*)(w + 4 * nb),
     *Ws = (cd*)(w + 5 * nb);
  double* d_eps = (double*)(w + 6 * nb);
  void* cscr = w + 6 * nb + eb;
  double* d_part = (double*)(w + 6 * nb + eb + cb);
  GridBar bar{(unsigned*)(w + 6 * nb + eb + cb + pb), (int*)(w + 6 * nb + eb + cb + pb) + 1};
  int* d_int = bar.fail + 1;
  const int b = 256, g = (int)((nn + b - 1) / b);
  int st = OEFE_OK, fail = 0;
  OEFE_COUNTED k_to_cd<S><<<g, b, 0, c->stream>>>(H, Hc, (int)nn);
  OEFE_COUNTED k_to_cd<S><<<g, b, 0, c->stream>>>(M, Mc, (int)nn);
  OEFE_COUNTED k_hermitian_part<<<g, b, 0, c->stream>>>(Hc, n);
  OEFE_COUNTED k_hermitian_part<<<g, b, 0, c->stream>>>(Mc, n);
  int info = 0;
  OEFE_TRY(chol_factor_inverse<cd>(c, Mc, T, Y, n, cscr, c->d_status + 3, &info));   // Y = L^{-1}
  if (info != 0) {
    c->err = "rayleigh_ritz: projected overlap not positive definite";
    st = OEFE_ERR_CHOLESKY;
  } else {
    OEFE_COUNTED k_small_gemm<<<g, b, 0, c->stream>>>(Y, false, Hc, false, T, n);  // T = L^{-1} H
    OEFE_COUNTED k_small_gemm<<<g, b, 0, c->stream>>>(T, false, Y, true, Hc, n);   // C = T L^{-+}
    OEFE_COUNTED k_hermitian_part<<<g, b, 0, c->stream>>>(Hc, n);
    const size_t jsm = 2 * nn * sizeof(cd);
    const int np = (n + (n & 1)) / 2;
    auto one_cta = [&](bool init_v) -> int {
      OEFE_CUDA_TRY(c, cudaFuncSetAttribute(k_jacobi, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)jsm));
      OEFE_COUNTED k_jacobi<<<1, JT, jsm, c->stream>>>(Hc, W, n, 40, 1e-15, d_int, init_v);
      return OEFE_OK;
    };
    auto sweeps = [&](auto elem, double tol) -> int {   // the cooperative launch
      using E = decltype(elem);
      // 16 blocks of A per CTA: enough CTAs that the updates take less than the barrier
      const int grid = std::max(1, std::min(c->num_sms, np * np / 16));
      const size_t smem = (size_t)((n + grid - 1) / grid) * n * sizeof(E) + (size_t)np * sizeof(JRot<E>);
      OEFE_CUDA_TRY(c, cudaFuncSetAttribute(k_jacobi_grid<E>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      OEFE_CUDA_TRY(c, cudaMemsetAsync(bar.count, 0, 8, c->stream));
      int most = 40;
      double tol2 = tol * tol;
      E *A1 = (E*)Mc, *A0 = (E*)Hc, *Vp = (E*)W;
      JRot<E>* rot = (JRot<E>*)Ws;   // Ws is free until the sort below (n^2 cd >= n / 2 JRot)
      void* args[] = {&A0, &A1, &Vp, (void*)&n, &most, &tol2, &d_part, &rot, &bar};
      OEFE_CUDA_TRY(c, cudaLaunchCooperativeKernel((const void*)k_jacobi_grid<E>, dim3(grid), dim3(GJ), args, smem, c->stream));
      oefe_launch_add(1);
      OEFE_CUDA_TRY(c, cudaMemcpyAsync(&fail, bar.fail, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
      return OEFE_OK;
    };
    if (c->f64_products == OEFE_F64_PAIRS && n <= CTA_N) {
      // the sweeps down to about the pair precision on the FP32 pipe, the rest (usually none: Jacobi
      // converges quadratically) in FP64; the result carries the pair arithmetic's backward error,
      // about 2^-48 ||A||
      OEFE_COUNTED k_to_pairs<<<g, b, 0, c->stream>>>(Hc, (int)nn);
      OEFE_TRY(sweeps(c2j{}, 1e-12));
      OEFE_COUNTED k_from_pairs<<<g, b, 0, c->stream>>>(Hc, W, (int)nn);
      OEFE_TRY(one_cta(false));
    } else if (n <= ONE_CTA_N) {
      OEFE_TRY(one_cta(true));
    } else {
      OEFE_TRY(sweeps(cd{}, 1e-15));
    }
    OEFE_COUNTED k_sort_eig<<<(n + 127) / 128, 128, 0, c->stream>>>(Hc, W, n, d_eps, Ws);
    OEFE_COUNTED k_small_gemm<<<g, b, 0, c->stream>>>(Y, true, Ws, false, T, n);   // U = L^{-+} W
    OEFE_COUNTED k_from_cd<S><<<g, b, 0, c->stream>>>(T, U, (int)nn);
    cudaMemcpyAsync(eps_host, d_eps, n * sizeof(double), cudaMemcpyDeviceToHost, c->stream);
    if (cudaGetLastError() != cudaSuccess) { c->err = "eigensolver launch failed"; st = OEFE_ERR_CUDA; }
    cudaStreamSynchronize(c->stream);
    if (fail && st == OEFE_OK) { c->err = "eigensolver: a grid barrier timed out"; st = OEFE_ERR_TIMEOUT; }
  }
  return st;
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
