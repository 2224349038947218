// CFE-CFE block of the single-leaf cells' FP64-class products (Eq. HOEFEelelements), sum factorized
// with register tiles: the pair-mode counterpart of sf_cc (sumfac_dev.cuh) for the orders and rules in
// use (P = p + 1 = 4 .. 7 nodes, N1 = P or P + 2 points per axis).
//
// Bound: the FP32 pipe (12 instructions per pair multiply-add; about 41 k of them per real column and
// cell at p = 6). One output per thread, as in sf_cc, needs two shared-memory operands per
// multiply-add, address arithmetic and 13 barriers, and reached a third of the pipe's rate. Here a
// thread owns a line (a 1D contraction) of two columns: every output of the line is an accumulator in
// registers, each line entry is read once (16 bytes, two columns) and each table entry once for both
// columns, packed instructions (pair2_dev.cuh) take the two columns together, and 7 to 18 independent
// chains hide the latency of the two-sums. The z contraction to the
// points, the point weights and the contraction back run on one line without leaving registers, the
// kinetic contractions share the barriers of the potential's: 5 barriers. A CTA takes 4 real columns
// (complex data interleaved: two vectors), small enough for three CTAs per SM, whose barriers overlap.
// Pairs enter and leave through integer conversions: the FP64 pipe, at two results a clock, took
// a sixth of the old kernel's time converting.
#include <algorithm>

#include "oefe_internal.h"
#include "pair2_dev.cuh"
#include "sumfac_dev.cuh"

namespace {

constexpr int CJ = 4;       // real columns per CTA
constexpr int CT = 128;     // threads per CTA

struct CcArgs {
  const double* sf;          // per listed cell: SF_STRIDE doubles
  const int* cells;
  const double* X;           // real view
  long long ldx;
  int nvr;                   // real columns
  const int* cell_nodes;
  const int* act_off;
  int nloc, npad;
  const double* qw;
  const double* veff;
  const int64_t* q_off;
  double k[3];
  double* Z;                 // real view (ncells x npad x nvr): enrichment part in, product out
};

template <int P, int N1>
struct CcPlan {
  static constexpr int P2 = P * P, P3 = P2 * P, N2 = N1 * N1, N3 = N2 * N1;
  static constexpr int NB = (P3 > P * N2 ? P3 : P * N2);        // X, later the (c, qy, qx) lines
  static constexpr int NA = P2 * N1;                            // the (c, b, qx) lines
  static constexpr int TAB = 3 * N1 * P + 9 * P2;               // L, M, K/2, -(k/2) A
  static constexpr size_t SMEM = ((size_t)TAB + (size_t)(NB + NA + 2 * P3) * (CJ / 2)) * sizeof(p2) + (size_t)N3 * sizeof(f2);
};

template <bool CPLX, int P, int N1>
__global__ void __launch_bounds__(CT, 3) k_sf_cc(const CcArgs A) {
  using C = CcPlan<P, N1>;
  constexpr int P2 = C::P2, P3 = C::P3, N2 = C::N2, N3 = C::N3;
  extern __shared__ __align__(16) unsigned char cc_raw[];
  constexpr int JP = CJ / 2;
  p2* L = reinterpret_cast<p2*>(cc_raw);          // [3][N1][P], both halves the same value
  p2* M = L + 3 * N1 * P;                         // [3][P][P]
  p2* Kh = M + 3 * P2;                            // [3][P][P]  K / 2
  p2* Ai = Kh + 3 * P2;                           // [3][P][P]  -(k / 2) A
  p2* B = Ai + 3 * P2;                            // X, then the (c, qy, qx) lines; [entry][JP]
  p2* Ab = B + (size_t)C::NB * JP;                // (c, b, qx) lines
  p2* C0 = Ab + (size_t)C::NA * JP;               // M x, then M M x
  p2* C1 = C0 + (size_t)P3 * JP;                  // G x, then G M x + M G x
  f2* Ws = reinterpret_cast<f2*>(C1 + (size_t)P3 * JP);   // [N3]
  const int e = A.cells[blockIdx.y];
  const int j0 = blockIdx.x * CJ;
  const double* src = A.sf + (size_t)blockIdx.y * SF_STRIDE;
  for (int t = threadIdx.x; t < 3 * N1 * P; t += CT) {
    const int a = t % P, q = (t / P) % N1, d = t / (P * N1);
    L[t] = p2_dup(f2_from_int(src[SF_L + (d * SF_MAXN1 + q) * SF_MAXP + a]));
  }
  for (int t = threadIdx.x; t < 3 * P2; t += CT) {
    const int a = t % P, r = (t / P) % P, d = t / P2;
    const int o = (d * SF_MAXP + r) * SF_MAXP + a;
    M[t] = p2_dup(f2_from_int(src[SF_M + o]));
    Kh[t] = p2_dup(f2_from_int(0.5 * src[SF_K + o]));
    if (CPLX) Ai[t] = p2_dup(f2_from_int(-0.5 * A.k[d] * src[SF_A + o]));
  }
  {
    const double kk2 = 0.5 * (A.k[0] * A.k[0] + A.k[1] * A.k[1] + A.k[2] * A.k[2]);
    const int64_t q0 = A.q_off[e];
    for (int q = threadIdx.x; q < N3; q += CT) Ws[q] = f2_from_int(A.qw[q0 + q] * (CPLX ? A.veff[q0 + q] + kk2 : A.veff[q0 + q]));
  }
  for (int t = threadIdx.x; t < P3 * JP; t += CT) {
    const int r = t / JP, j = j0 + 2 * (t % JP);
    const double* x = A.X + (long long)A.cell_nodes[(size_t)e * A.nloc + r] * A.ldx + j;
    B[t] = p2_join(j < A.nvr ? f2_from_int(x[0]) : f2{0.f, 0.f}, j + 1 < A.nvr ? f2_from_int(x[1]) : f2{0.f, 0.f});
  }
  __syncthreads();
  // x lines to the points; z lines through M and G
  for (int t = threadIdx.x; t < 2 * P2 * JP; t += CT) {
    const int jp = t % JP, ln = (t / JP) % P2;
    if (t < P2 * JP) {
      p2 y[N1];
#pragma unroll
      for (int q = 0; q < N1; ++q) y[q] = p2_zero();
#pragma unroll 1
      for (int a = 0; a < P; ++a) {
        const p2 x = B[(a + P * ln) * JP + jp];
#pragma unroll
        for (int q = 0; q < N1; ++q) p2_mac(y[q], L[q * P + a], x);
      }
#pragma unroll
      for (int q = 0; q < N1; ++q) Ab[(ln * N1 + q) * JP + jp] = p2_fin(y[q]);
    } else {
      p2 ym[P], yg[P];
#pragma unroll
      for (int c = 0; c < P; ++c) ym[c] = yg[c] = p2_zero();
#pragma unroll 1
      for (int c2 = 0; c2 < P; ++c2) {
        const p2 x = B[(ln + P2 * c2) * JP + jp];
        const p2 ix = CPLX ? p2_times_i(x) : x;
#pragma unroll
        for (int c = 0; c < P; ++c) {
          p2_mac(ym[c], M[(2 * P + c) * P + c2], x);
          p2_mac(yg[c], Kh[(2 * P + c) * P + c2], x);
          if (CPLX) p2_mac(yg[c], Ai[(2 * P + c) * P + c2], ix);
        }
      }
#pragma unroll
      for (int c = 0; c < P; ++c) {
        C0[(ln + P2 * c) * JP + jp] = p2_fin(ym[c]);
        C1[(ln + P2 * c) * JP + jp] = p2_fin(yg[c]);
      }
    }
  }
  __syncthreads();
  // y lines to the points; y lines of the kinetic term, in place
  for (int t = threadIdx.x; t < (P2 + P * N1) * JP; t += CT) {
    const int jp = t % JP;
    if (t < P * N1 * JP) {
      const int ln = t / JP, qx = ln % N1, c = ln / N1;
      p2 y[N1];
#pragma unroll
      for (int q = 0; q < N1; ++q) y[q] = p2_zero();
#pragma unroll 1
      for (int b = 0; b < P; ++b) {
        const p2 x = Ab[((c * P + b) * N1 + qx) * JP + jp];
#pragma unroll
        for (int q = 0; q < N1; ++q) p2_mac(y[q], L[(N1 + q) * P + b], x);
      }
#pragma unroll
      for (int q = 0; q < N1; ++q) B[((c * N1 + q) * N1 + qx) * JP + jp] = p2_fin(y[q]);
    } else {
      const int ln = t / JP - P * N1, a = ln % P, c = ln / P;
      p2 w1[P], w2[P];
#pragma unroll
      for (int b = 0; b < P; ++b) w1[b] = w2[b] = p2_zero();
#pragma unroll 1
      for (int b2 = 0; b2 < P; ++b2) {
        const int o = (a + P * b2 + P2 * c) * JP + jp;
        const p2 zm = C0[o], zg = C1[o];
        const p2 iz = CPLX ? p2_times_i(zm) : zm;
#pragma unroll
        for (int b = 0; b < P; ++b) {
          const p2 m = M[(P + b) * P + b2];
          p2_mac(w1[b], m, zm);
          p2_mac(w2[b], Kh[(P + b) * P + b2], zm);
          p2_mac(w2[b], m, zg);
          if (CPLX) p2_mac(w2[b], Ai[(P + b) * P + b2], iz);
        }
      }
#pragma unroll
      for (int b = 0; b < P; ++b) {
        C0[(a + P * b + P2 * c) * JP + jp] = p2_fin(w1[b]);
        C1[(a + P * b + P2 * c) * JP + jp] = p2_fin(w2[b]);
      }
    }
  }
  __syncthreads();
  // z lines: to the points, weights, back, in place
  for (int t = threadIdx.x; t < N2 * JP; t += CT) {
    const int jp = t % JP, ln = t / JP;
    p2 u[N1];
#pragma unroll
    for (int q = 0; q < N1; ++q) u[q] = p2_zero();
#pragma unroll 1
    for (int c = 0; c < P; ++c) {
      const p2 x = B[(c * N2 + ln) * JP + jp];
#pragma unroll
      for (int q = 0; q < N1; ++q) p2_mac(u[q], L[(2 * N1 + q) * P + c], x);
    }
#pragma unroll
    for (int q = 0; q < N1; ++q) u[q] = p2_mul(p2_fin(u[q]), p2_dup(Ws[q * N2 + ln]));
    p2 y[P];
#pragma unroll
    for (int c = 0; c < P; ++c) y[c] = p2_zero();
#pragma unroll
    for (int q = 0; q < N1; ++q)
#pragma unroll
      for (int c = 0; c < P; ++c) p2_mac(y[c], L[(2 * N1 + q) * P + c], u[q]);
#pragma unroll
    for (int c = 0; c < P; ++c) B[(c * N2 + ln) * JP + jp] = p2_fin(y[c]);
  }
  __syncthreads();
  // back along y
  for (int t = threadIdx.x; t < P * N1 * JP; t += CT) {
    const int jp = t % JP, ln = t / JP, qx = ln % N1, c = ln / N1;
    p2 y[P];
#pragma unroll
    for (int b = 0; b < P; ++b) y[b] = p2_zero();
#pragma unroll 1
    for (int q = 0; q < N1; ++q) {
      const p2 x = B[((c * N1 + q) * N1 + qx) * JP + jp];
#pragma unroll
      for (int b = 0; b < P; ++b) p2_mac(y[b], L[(N1 + q) * P + b], x);
    }
#pragma unroll
    for (int b = 0; b < P; ++b) Ab[((c * P + b) * N1 + qx) * JP + jp] = p2_fin(y[b]);
  }
  __syncthreads();
  // back along x, the kinetic term's x lines, the enrichment part, out
  const bool enr = A.act_off[e + 1] > A.act_off[e];
  for (int t = threadIdx.x; t < P2 * JP; t += CT) {
    const int jp = t % JP, ln = t / JP, j = j0 + 2 * jp;
    p2 y[P];
#pragma unroll
    for (int a = 0; a < P; ++a) y[a] = p2_zero();
#pragma unroll 1
    for (int q = 0; q < N1; ++q) {
      const p2 x = Ab[(ln * N1 + q) * JP + jp];
#pragma unroll
      for (int a = 0; a < P; ++a) p2_mac(y[a], L[q * P + a], x);
    }
#pragma unroll 1
    for (int a2 = 0; a2 < P; ++a2) {
      const int o = (a2 + P * ln) * JP + jp;
      const p2 w1 = C0[o], w2 = C1[o];
      const p2 iw = CPLX ? p2_times_i(w1) : w1;
#pragma unroll
      for (int a = 0; a < P; ++a) {
        p2_mac(y[a], Kh[a * P + a2], w1);
        p2_mac(y[a], M[a * P + a2], w2);
        if (CPLX) p2_mac(y[a], Ai[a * P + a2], iw);
      }
    }
#pragma unroll
    for (int a = 0; a < P; ++a) {
      f2 s0, s1;
      p2_halves(p2_fin(y[a]), s0, s1);
      double* z = A.Z + ((size_t)e * A.npad + a + P * ln) * A.nvr + j;
      if (j < A.nvr) z[0] = enr ? z[0] + f2_to_int(s0) : f2_to_int(s0);
      if (j + 1 < A.nvr) z[1] = enr ? z[1] + f2_to_int(s1) : f2_to_int(s1);
    }
  }
}

}  // namespace

// The CFE-CFE products of `count` cells of the list from `first` (all with N1 = n1 points per axis), added
// to the enrichment part in Z; *done false when this order and rule have no instance.
int launch_sf_cc(oefe_ctx* c, const KData& K, const void* X, int ldx, int nv, bool cplx, void* Z, int first, int count,
                 int n1, bool* done, cudaStream_t st) {
  *done = false;
  if (count == 0) { *done = true; return OEFE_OK; }
  const int R = cplx ? 2 : 1;
  CcArgs A;
  A.sf = c->d_sf + (size_t)first * SF_STRIDE;
  A.cells = c->d_sf_cells + first;
  A.X = (const double*)X;
  A.ldx = (long long)ldx * R;
  A.nvr = nv * R;
  A.cell_nodes = c->d_cell_nodes;
  A.act_off = c->d_act_off;
  A.nloc = c->nloc;
  A.npad = c->npad;
  A.qw = c->d_qw;
  A.veff = c->d_veff;
  A.q_off = c->d_q_off;
  for (int d = 0; d < 3; ++d) A.k[d] = K.k[d];
  A.Z = (double*)Z;
  auto go = [&](auto kern, size_t smem) -> int {
    OEFE_CUDA_TRY(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    // (65535 rows of CTAs at most per launch)
    for (int y = 0; y < count; y += 65535) {
      CcArgs a = A;
      a.sf += (size_t)y * SF_STRIDE;
      a.cells += y;
      OEFE_COUNTED kern<<<dim3((A.nvr + CJ - 1) / CJ, std::min(65535, count - y)), CT, smem, st>>>(a);
    }
    OEFE_CUDA_TRY(c, cudaGetLastError());
    *done = true;
    return OEFE_OK;
  };
#define OEFE_CC(p, q) \
  if (c->P == p && n1 == q) return cplx ? go(k_sf_cc<true, p, q>, CcPlan<p, q>::SMEM) : go(k_sf_cc<false, p, q>, CcPlan<p, q>::SMEM);
  OEFE_CC(4, 4) OEFE_CC(4, 6) OEFE_CC(5, 5) OEFE_CC(5, 7) OEFE_CC(6, 6) OEFE_CC(6, 8) OEFE_CC(7, 7) OEFE_CC(7, 9)
#undef OEFE_CC
  return OEFE_OK;
}
