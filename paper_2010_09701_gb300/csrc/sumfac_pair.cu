// FP64-class products of the single-leaf cells in pair mode (Eq. HOEFEelelements), for the orders and rules
// in use (P = p + 1 = 4 .. 7 nodes, N1 = P or P + 2 points per axis), in two kernels: the CFE-CFE block sum
// factorized with register tiles (k_sf_cc), then the blocks with enrichment rows from the stored matrix
// (k_sf_strips). Every value takes the operations of sf_cc and k_cell_apply_sf (sumfac_dev.cuh, sumfac.cu)
// in their order: the two partial sums of v_dot, the interleaving of the kinetic terms. The defect
// filter's degrees round in FP32 on this product and the signs of Ritz vectors follow its last bits, so
// another order of sums would change both by far more than the order's own rounding.
//
// Bound: the FP32 pipe (12 instructions per pair multiply-add; about 41 k of them per real column and
// cell at p = 6, and 27 k in the strips). One output per thread, as in sf_cc, needs two shared-memory
// operands per multiply-add, address arithmetic and 13 barriers, and reached a third of the pipe's rate.
// Here a thread owns a line (a 1D contraction) of two columns: every output of the line is an accumulator
// in registers, each line entry is read once (16 bytes, two columns) and each table entry once for both
// columns, packed instructions (pair2_dev.cuh) take the two columns together. The z contraction to the
// points, the point weights and the contraction back run on one line without leaving registers, the
// kinetic contractions share the barriers of the potential's: 5 barriers. A CTA takes 4 real columns
// (complex data interleaved: two vectors), small enough for three CTAs per SM, whose barriers overlap.
// Pairs enter and leave through integer conversions: the FP64 pipe, at two results a clock, took
// a sixth of the old kernel's time converting. The strips run by themselves on more columns per CTA, each
// matrix entry loaded once for 8 real columns. 64 real columns of the 62-atom cell at 16^3: 15.6 ms in one
// kernel, 6.0 + 6.7 ms in these.
#include <algorithm>
#include <type_traits>

#include "oefe_internal.h"
#include "pair2_dev.cuh"
#include "sumfac_dev.cuh"

namespace {

constexpr int CJ = 4;       // real columns per pass
constexpr int CP = 4;       // passes per CTA at most: the cell's tables and weights are set up once for them
constexpr int CT = 128;     // threads per CTA

struct CcArgs {
  const double* sf;          // per listed cell: SF_STRIDE doubles
  const int* cells;
  const double* X;           // real view
  long long ldx;
  int nvr;                   // real columns
  int passes;                // per CTA
  const int* cell_nodes;
  const int* act_off;
  int nloc, npad;
  const double* qw;
  const double* veff;
  const int64_t* q_off;
  double k[3];
  f2* Z;                     // real view (ncells x npad x nvr): the CFE-CFE part as pairs, then the product
};

template <int P, int N1>
struct CcPlan {
  static constexpr int P2 = P * P, P3 = P2 * P, N2 = N1 * N1, N3 = N2 * N1;
  static constexpr int NB = (P3 > P * N2 ? P3 : P * N2);        // X, later the (c, qy, qx) lines
  static constexpr int NA = P2 * N1;                            // the (c, b, qx) lines
  static constexpr int TAB = 3 * N1 * P + 13 * P2;              // L, M, K/2, -(k/2) A, the joined ones
  static constexpr size_t SMEM = ((size_t)TAB + (size_t)(NB + NA + 2 * P3) * (CJ / 2)) * sizeof(p2) + (size_t)N3 * sizeof(f2);
};

// y[o] = sum_{i < N} t(o, i) x(i), as v_dot: the even and the odd terms summed apart
template <int N, int NOUT, typename FX, typename FT>
__device__ __forceinline__ void line(p2 (&y)[NOUT], FX x, FT t) {
  p2 y1[NOUT];
#pragma unroll
  for (int o = 0; o < NOUT; ++o) y[o] = y1[o] = p2_zero();
#pragma unroll 1
  for (int i = 0; i + 1 < N; i += 2) {
    const p2 xa = x(i), xb = x(i + 1);
#pragma unroll
    for (int o = 0; o < NOUT; ++o) {
      p2_mac(y[o], t(o, i), xa);
      p2_mac(y1[o], t(o, i + 1), xb);
    }
  }
  if (N & 1) {
    const p2 xa = x(N - 1);
#pragma unroll
    for (int o = 0; o < NOUT; ++o) p2_mac(y[o], t(o, N - 1), xa);
  }
#pragma unroll
  for (int o = 0; o < NOUT; ++o) y[o] = p2_add(p2_fin(y[o]), p2_fin(y1[o]));
}

// operands of the tables (M, A) and (A, M): (g.re, m.re), (-m.im, g.im)
__device__ __forceinline__ void cross(p2 g, p2 m, p2& a, p2& b) {
  f2 gr, gi, mr, mi;
  p2_halves(g, gr, gi);
  p2_halves(m, mr, mi);
  a = p2_join(gr, mr);
  b = p2_join(f2_neg(mi), gi);
}

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
  p2* MA = Ai + 3 * P2;                           // [2][P][P]  (M, -(k / 2) A) of x and y: the real and imaginary parts
  p2* AM = MA + 2 * P2;                           //            take these two terms in opposite order
  p2* B = AM + 2 * P2;                            // X, then the (c, qy, qx) lines; [entry][JP]
  p2* Ab = B + (size_t)C::NB * JP;                // (c, b, qx) lines
  p2* C0 = Ab + (size_t)C::NA * JP;               // M x, then M M x
  p2* C1 = C0 + (size_t)P3 * JP;                  // G x, then G M x + M G x
  f2* Ws = reinterpret_cast<f2*>(C1 + (size_t)P3 * JP);   // [N3]
  const int e = A.cells[blockIdx.y];
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
    if (CPLX) {
      const f2 m = f2_from_int(src[SF_M + o]), av = f2_from_int(-0.5 * (d == 0 ? A.k[0] : d == 1 ? A.k[1] : A.k[2]) * src[SF_A + o]);
      Ai[t] = p2_dup(av);
      if (d < 2) {
        MA[t] = p2_join(m, av);
        AM[t] = p2_join(av, m);
      }
    }
  }
  {
    const double kk = A.k[0] * A.k[0] + A.k[1] * A.k[1] + A.k[2] * A.k[2];
    const int64_t q0 = A.q_off[e];
    for (int q = threadIdx.x; q < N3; q += CT) Ws[q] = f2_from_int(A.qw[q0 + q] * (A.veff[q0 + q] + 0.5 * kk));
  }
  for (int pass = 0; pass < A.passes; ++pass) {
  const int j0 = (blockIdx.x * A.passes + pass) * CJ;
  if (j0 >= A.nvr) break;
  __syncthreads();
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
      line<P, N1>(y, [&](int a) { return B[(a + P * ln) * JP + jp]; }, [&](int q, int a) { return L[q * P + a]; });
#pragma unroll
      for (int q = 0; q < N1; ++q) Ab[(ln * N1 + q) * JP + jp] = y[q];
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
      line<P, N1>(y, [&](int b) { return Ab[((c * P + b) * N1 + qx) * JP + jp]; },
                  [&](int q, int b) { return L[(N1 + q) * P + b]; });
#pragma unroll
      for (int q = 0; q < N1; ++q) B[((c * N1 + q) * N1 + qx) * JP + jp] = y[q];
    } else {
      const int ln = t / JP - P * N1, a = ln % P, c = ln / P;
      p2 w1[P], w2[P];
#pragma unroll
      for (int b = 0; b < P; ++b) w1[b] = w2[b] = p2_zero();
#pragma unroll 1
      for (int b2 = 0; b2 < P; ++b2) {
        const int o = (a + P * b2 + P2 * c) * JP + jp;
        const p2 zm = C0[o], zg = C1[o];
        p2 za = zg, zb = zg;
        if (CPLX) cross(zg, zm, za, zb);
#pragma unroll
        for (int b = 0; b < P; ++b) {
          const int o1 = (P + b) * P + b2;
          p2_mac(w1[b], M[o1], zm);
          p2_mac(w2[b], Kh[o1], zm);
          if (CPLX) {
            p2_mac(w2[b], MA[o1], za);
            p2_mac(w2[b], AM[o1], zb);
          } else {
            p2_mac(w2[b], M[o1], zg);
          }
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
    line<P, N1>(u, [&](int c) { return B[(c * N2 + ln) * JP + jp]; }, [&](int q, int c) { return L[(2 * N1 + q) * P + c]; });
#pragma unroll
    for (int q = 0; q < N1; ++q) u[q] = p2_mul(u[q], p2_dup(Ws[q * N2 + ln]));
    p2 y[P], y1[P];
#pragma unroll
    for (int c = 0; c < P; ++c) y[c] = y1[c] = p2_zero();
#pragma unroll
    for (int q = 0; q < N1; ++q)
#pragma unroll
      for (int c = 0; c < P; ++c) p2_mac(q & 1 ? y1[c] : y[c], L[(2 * N1 + q) * P + c], u[q]);
#pragma unroll
    for (int c = 0; c < P; ++c) B[(c * N2 + ln) * JP + jp] = p2_add(p2_fin(y[c]), p2_fin(y1[c]));
  }
  __syncthreads();
  // back along y
  for (int t = threadIdx.x; t < P * N1 * JP; t += CT) {
    const int jp = t % JP, ln = t / JP, qx = ln % N1, c = ln / N1;
    p2 y[P];
    line<N1, P>(y, [&](int q) { return B[((c * N1 + q) * N1 + qx) * JP + jp]; },
                [&](int b, int q) { return L[(N1 + q) * P + b]; });
#pragma unroll
    for (int b = 0; b < P; ++b) Ab[((c * P + b) * N1 + qx) * JP + jp] = y[b];
  }
  __syncthreads();
  // back along x, the kinetic term's x lines, out
  for (int t = threadIdx.x; t < P2 * JP; t += CT) {
    const int jp = t % JP, ln = t / JP, j = j0 + 2 * jp;
    p2 y[P], w[P];
    line<N1, P>(y, [&](int q) { return Ab[(ln * N1 + q) * JP + jp]; }, [&](int a, int q) { return L[q * P + a]; });
#pragma unroll
    for (int a = 0; a < P; ++a) {
      y[a] = p2_add(p2_zero(), y[a]);
      w[a] = p2_zero();
    }
#pragma unroll 1
    for (int a2 = 0; a2 < P; ++a2) {
      const int o = (a2 + P * ln) * JP + jp;
      const p2 w1 = C0[o], w2 = C1[o];
      p2 wa = w2, wb = w2;
      if (CPLX) cross(w2, w1, wa, wb);
#pragma unroll
      for (int a = 0; a < P; ++a) {
        p2_mac(w[a], Kh[a * P + a2], w1);
        if (CPLX) {
          p2_mac(w[a], MA[a * P + a2], wa);
          p2_mac(w[a], AM[a * P + a2], wb);
        } else {
          p2_mac(w[a], M[a * P + a2], w2);
        }
      }
    }
#pragma unroll
    for (int a = 0; a < P; ++a) {
      f2 s0, s1;
      p2_halves(p2_add(y[a], p2_fin(w[a])), s0, s1);
      f2* z = A.Z + ((size_t)e * A.npad + a + P * ln) * A.nvr + j;
      if (j < A.nvr) z[0] = s0;
      if (j + 1 < A.nvr) z[1] = s1;
    }
  }
  }
}

// ------------------------------------------------------------------ blocks with enrichment rows
constexpr int SJ = 8;       // real columns per CTA
constexpr int ST = 256;     // threads per CTA

struct StripArgs {
  const int* cells;
  const float* Hp;           // the stored matrix as pairs
  int compact, ne_max;       // compact layout: the listed cell's strip starts at base + slot * strip
  long long base, strip;
  const double* X;           // real view
  long long ldx;
  int nvr;
  const int* cell_nodes;
  const int* act_off;
  const int* act_idx;
  int nloc, npad, nbuf, rows;   // rows: the largest cell's
  int64_t nh;
  void* Z;                   // real view: the CFE-CFE part as pairs in, FP64 out
};

// One item per thread, 8 real columns: a node row over the ne enrichment columns on top of its CFE-CFE part, or a
// chunk of about 48 columns of an enrichment row (the partial sums meet in shared memory), so that the
// items have about the same length. A warp's lanes take the same columns of different rows: one row of the
// vectors per column, a broadcast. L1 is what bounds it (90% of its rate), by the 32 lines that a load of
// 32 rows touches: so 16 bytes a lane, four columns in flight (8 bytes: 9.9 ms for 64 real columns of the
// 62-atom cell at 16^3, 6.7 with 16; tiles of 64 bytes a row staged through shared memory: 12.8).
template <bool CPLX>
__global__ void __launch_bounds__(ST, 3) k_sf_strips(const StripArgs A) {
  using E = typename std::conditional<CPLX, float4, float2>::type;   // a matrix entry: (h, l) per real part
  constexpr int JP = SJ / 2, CW = 4;
  extern __shared__ __align__(16) unsigned char st_raw[];
  const int e = A.cells[blockIdx.y], j0 = blockIdx.x * SJ;
  const int nloc = A.nloc, npad = A.npad, ne = A.act_off[e + 1] - A.act_off[e], naug = nloc + ne;
  p2* Xs = reinterpret_cast<p2*>(st_raw);          // [rows][JP]
  p2* part = Xs + (size_t)A.rows * JP;               // [ne * nch][JP]
  for (int t = threadIdx.x; t < naug * JP; t += ST) {
    const int r = t / JP, j = j0 + 2 * (t % JP);
    const int64_t row = r < nloc ? (int64_t)A.cell_nodes[(size_t)e * nloc + r] : A.nh + A.act_idx[A.act_off[e] + r - nloc];
    const double* x = A.X + row * A.ldx + j;
    Xs[t] = p2_join(j < A.nvr ? f2_from_int(x[0]) : f2{0.f, 0.f}, j + 1 < A.nvr ? f2_from_int(x[1]) : f2{0.f, 0.f});
  }
  __syncthreads();
  const bool pairs16 = A.nvr % 2 == 0 && ((uintptr_t)A.Z & 15) == 0;   // two columns of a row in 16-byte accesses
  int nch = min((naug + 47) / 48, A.nbuf / max(ne, 1));
  nch = max(nch, 1);
  const int EC = (naug + nch - 1) / nch;
  for (int it = threadIdx.x; it < nloc + ne * nch; it += ST) {
    int r, ca, cb, pidx = 0;
    if (it < nloc) {
      r = it;
      ca = nloc;
      cb = naug;
    } else {
      const int q = it - nloc, ch = q / ne, i = q % ne;
      r = nloc + i;
      ca = ch * EC;
      cb = min(naug, ca + EC);
      pidx = i * nch + ch;
    }
    f2* z = reinterpret_cast<f2*>(A.Z) + ((size_t)e * npad + r) * A.nvr + j0;
    p2 y[JP];
#pragma unroll
    for (int j = 0; j < JP; ++j) {
      y[j] = p2_zero();
      if (it >= nloc) continue;
      if (pairs16) {
        if (j0 + 2 * j < A.nvr) {
          const float4 v = *reinterpret_cast<const float4*>(z + 2 * j);
          y[j] = p2_join(f2{v.x, v.y}, f2{v.z, v.w});
        }
      } else {
        y[j] = p2_join(j0 + 2 * j < A.nvr ? z[2 * j] : f2{0.f, 0.f}, j0 + 2 * j + 1 < A.nvr ? z[2 * j + 1] : f2{0.f, 0.f});
      }
    }
    long long ro;   // entry (r, c) at ro + c, for the columns this row holds
    if (!A.compact) {
      ro = ((long long)e * npad + r) * npad;
    } else {
      const long long b = A.base + (long long)blockIdx.y * A.strip;
      ro = r < nloc ? b + (long long)r * A.ne_max - nloc : b + (long long)nloc * A.ne_max + (long long)(r - nloc) * npad;
    }
    const E* hr = reinterpret_cast<const E*>(A.Hp) + ro;
    auto column = [&](int c, const E& h) {
      const p2* x = Xs + (size_t)c * JP;
      const p2 hre = p2_dup(f2{h.x, h.y});
      if constexpr (CPLX) {
        const p2 him = p2_dup(f2{h.z, h.w});
#pragma unroll
        for (int j = 0; j < JP; ++j) {
          const p2 xv = x[j];
          p2_mac(y[j], hre, xv);
          p2_mac(y[j], him, p2_times_i(xv));
        }
      } else {
#pragma unroll
        for (int j = 0; j < JP; ++j) p2_mac(y[j], hre, x[j]);
      }
    };
    int c0 = ca;
    if constexpr (!CPLX)   // to a 16-byte boundary of the row
      if (c0 < cb && ((ro + c0) & 1)) {
        column(c0, hr[c0]);
        ++c0;
      }
    for (; c0 + CW <= cb; c0 += CW) {
      E h[CW];
      if constexpr (CPLX) {
#pragma unroll
        for (int u = 0; u < CW; ++u) h[u] = hr[c0 + u];
      } else {
#pragma unroll
        for (int u = 0; u < CW; u += 2) {
          const float4 v = *reinterpret_cast<const float4*>(hr + c0 + u);
          h[u] = make_float2(v.x, v.y);
          h[u + 1] = make_float2(v.z, v.w);
        }
      }
#pragma unroll
      for (int u = 0; u < CW; ++u) column(c0 + u, h[u]);
    }
    for (; c0 < cb; ++c0) column(c0, hr[c0]);
    if (it < nloc) {
      double* zo = reinterpret_cast<double*>(z);
#pragma unroll
      for (int j = 0; j < JP; ++j) {
        f2 s0, s1;
        p2_halves(p2_fin(y[j]), s0, s1);
        if (pairs16) {
          if (j0 + 2 * j < A.nvr) *reinterpret_cast<double2*>(zo + 2 * j) = make_double2(f2_to_int(s0), f2_to_int(s1));
        } else {
          if (j0 + 2 * j < A.nvr) zo[2 * j] = f2_to_int(s0);
          if (j0 + 2 * j + 1 < A.nvr) zo[2 * j + 1] = f2_to_int(s1);
        }
      }
    } else {
#pragma unroll
      for (int j = 0; j < JP; ++j) part[(size_t)pidx * JP + j] = p2_fin(y[j]);
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < ne * JP; t += ST) {   // enrichment rows: sum of the chunks
    const int i = t / JP, j = t % JP;
    p2 s = p2_zero();
    for (int ch = 0; ch < nch; ++ch) s = p2_add(s, part[(size_t)(i * nch + ch) * JP + j]);
    f2 s0, s1;
    p2_halves(s, s0, s1);
    double* zo = reinterpret_cast<double*>(A.Z) + ((size_t)e * npad + nloc + i) * A.nvr + j0 + 2 * j;
    if (j0 + 2 * j < A.nvr) zo[0] = f2_to_int(s0);
    if (j0 + 2 * j + 1 < A.nvr) zo[1] = f2_to_int(s1);
  }
}

}  // namespace

// The pair products of the listed single-leaf cells into Z; *done false when an order or rule has no instance.
int launch_sf_pair(oefe_ctx* c, const KData& K, const void* X, int ldx, int nv, bool cplx, void* Z, bool* done, cudaStream_t st) {
  *done = false;
  const int count = c->n_sf, R = cplx ? 2 : 1, P = c->P;
  if (count == 0) { *done = true; return OEFE_OK; }
  StripArgs S;
  S.nbuf = c->sf_nbuf;
  S.npad = c->npad;
  // shared memory of the strips: a cell's vectors, and the partial sums of its enrichment rows' chunks
  S.rows = c->nloc + c->ne_max;
  const int most = std::max(c->ne_max, std::min(c->sf_nbuf, c->ne_max * ((S.rows + 47) / 48)));
  const size_t ssm = ((size_t)S.rows + most) * (SJ / 2) * sizeof(p2);
  if (P < 4 || P > 7 || ssm > 227 * 1024) return OEFE_OK;
  for (int n1 : c->sf_n1_h)
    if (n1 != P && n1 != P + 2) return OEFE_OK;
  CcArgs A;
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
  A.Z = (f2*)Z;
  const int groups = (A.nvr + CJ - 1) / CJ;
  for (int i = 0; i < count;) {   // per class of points per axis (the list is sorted by it)
    const int n1 = c->sf_n1_h[i];
    int m = i;
    while (m < count && c->sf_n1_h[m] == n1) ++m;
    // as many passes as leave the GPU four waves of its three CTAs per SM
    A.passes = (int)std::max(1LL, std::min<long long>(CP, (long long)groups * (m - i) / (12LL * c->num_sms)));
    auto go = [&](auto kern, size_t smem) -> int {
      OEFE_CUDA_TRY(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      for (int y = i; y < m; y += 65535) {   // (65535 rows of CTAs at most per launch)
        A.sf = c->d_sf + (size_t)y * SF_STRIDE;
        A.cells = c->d_sf_cells + y;
        OEFE_COUNTED kern<<<dim3((groups + A.passes - 1) / A.passes, std::min(65535, m - y)), CT, smem, st>>>(A);
      }
      return OEFE_OK;
    };
    int s = OEFE_OK;
#define OEFE_CC(p, q) \
  if (P == p && n1 == q) s = cplx ? go(k_sf_cc<true, p, q>, CcPlan<p, q>::SMEM) : go(k_sf_cc<false, p, q>, CcPlan<p, q>::SMEM);
    OEFE_CC(4, 4) OEFE_CC(4, 6) OEFE_CC(5, 5) OEFE_CC(5, 7) OEFE_CC(6, 6) OEFE_CC(6, 8) OEFE_CC(7, 7) OEFE_CC(7, 9)
#undef OEFE_CC
    OEFE_TRY(s);
    i = m;
  }
  S.Hp = K.Hp;
  S.compact = K.compact ? 1 : 0;
  S.ne_max = c->ne_max;
  S.strip = (long long)compact_strip(c);
  S.X = A.X;
  S.ldx = A.ldx;
  S.nvr = A.nvr;
  S.cell_nodes = c->d_cell_nodes;
  S.act_off = c->d_act_off;
  S.act_idx = c->d_act_idx;
  S.nloc = c->nloc;
  S.nh = c->nh;
  S.Z = Z;
  auto strips = [&](auto kern) -> int {
    OEFE_CUDA_TRY(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)ssm));
    for (int y = 0; y < count; y += 65535) {
      S.cells = c->d_sf_cells + y;
      S.base = (long long)c->n_dense * c->npad * c->npad + (long long)y * S.strip;
      OEFE_COUNTED kern<<<dim3((A.nvr + SJ - 1) / SJ, std::min(65535, count - y)), ST, ssm, st>>>(S);
    }
    return OEFE_OK;
  };
  OEFE_TRY(cplx ? strips(k_sf_strips<true>) : strips(k_sf_strips<false>));
  OEFE_CUDA_TRY(c, cudaGetLastError());
  *done = true;
  return OEFE_OK;
}
