// Fields of the density and the band-trace gradient in pair mode (Eqs. UOEFE, rho):
//   u(x_q) = sum_a N_a(x_q) X_a + sum_j N^O_j(x_q) X^o_j, then sum_v w_v |u_v|^2 per point,
// in two kernels over batches of leaves:
//   k_fields_oz  the enrichment part, a dense product of the stored N^O table with the enrichment
//                coefficients, as an exact fixed-point product on the tensor cores (oz8_dev.cuh), into a
//                workspace as FP32 pairs;
//   k_fields_cc  the CFE part by sum factorization with register tiles (as k_sf_cc, sumfac_pair.cu), added to it,
//                squared, weighted and summed over the vectors without leaving registers.
//
// Bound: per leaf of 729 points and real vector the enrichment part was 28 k of 41 k pair multiply-adds,
// on an FP32 pipe that the one-output-per-thread kernel (k_fields, density.cu) kept a third busy: 558 ms
// for 360 vectors on the 62-atom cell at 16^3. On the tensor cores that part costs the cutting and combining
// of its digits; the rest runs at the rate of k_sf_cc. The workspace round trip (16 bytes per point
// and vector) is an eighth of the time saved.
#include <algorithm>

#include <vector>

#include "oefe_internal.h"
#include "enrich_dev.cuh"
#include "oz8_dev.cuh"
#include "pair2_dev.cuh"

namespace {

// ------------------------------------------------------------------ enrichment part
constexpr int FZ = 512;      // threads per CTA of k_fields_oz

struct FieldOzArgs {
  const Leaf* leaves;
  int l0, nl;                // leaves of the batch
  const int* act_off;
  const int* act_idx;
  int ne_max, mtiles;        // M tiles of 128 points per leaf (the largest leaf's)
  int64_t nh;
  const double* NO;          // per leaf ne_max columns of its points (complex: interleaved)
  const double* X;           // real view
  long long ldx;
  int nc, vblocks;           // real columns, blocks of 64
  int64_t q0;                // first point of the batch
  float4* U;                 // [point][nc / 2]: two columns (h0, h1, l0, l1)
  int ncp;                   // nc rounded up to even, halved
  int* err;
};

template <bool CPLX>
__global__ void __launch_bounds__(FZ, 1) k_fields_oz(const FieldOzArgs A) {
  constexpr int R = CPLX ? 2 : 1;
  extern __shared__ __align__(1024) unsigned char oz_raw[];
  __shared__ int sE[128], sF[ZN];
  __shared__ uint64_t bar[2];
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const OzCta C = oz_begin(oz_raw, &tmem_slot, bar, &s_fail);
  Halves H{bar};
  const bool warp0 = __shfl_sync(0xffffffffu, (int)threadIdx.x >> 5, 0) == 0;   // (uniform)
  // A: a thread per point and 8 entries of a half; B: a thread per column and 4 entries (pair orders
  // rotated per 8 rows so that stores spread over the banks)
  const int ar = tid & 127, ag = tid >> 7, bn = tid & 63, bg = tid >> 6;
  const int ash = (ar >> 3) & 3, bsh = (bn >> 3) & 1;
  double a[8], b[4];
  const long long total = (long long)A.nl * A.mtiles;
  for (long long job = blockIdx.x; job < total && !s_fail; job += gridDim.x) {
    const Leaf L = A.leaves[A.l0 + job / A.mtiles];
    const int n3 = L.n1 * L.n1 * L.n1, p0 = (int)(job % A.mtiles) * 128;
    const int o0 = A.act_off[L.cell], ne = A.act_off[L.cell + 1] - o0;
    if (p0 >= n3 || ne == 0) continue;   // (k_fields_cc does not read the part of a leaf without active functions)
    const int nr = min(128, n3 - p0);
    const bool aok = ar < nr;
    const double* no = A.NO + R * ((size_t)L.q0 * A.ne_max + p0 + ar);
    const size_t cs = (size_t)R * n3;                  // reals between columns of the table
    const int steps = R * ((ne + 31) / 32);
    if (tid < 128) sE[tid] = 0;
    __syncthreads();
    if (aok) {
      int m = 0;
      for (int k = ag; k < ne; k += 4) {
        m = max(m, bexp_of(__ldg(no + k * cs)));
        if (CPLX) m = max(m, bexp_of(__ldg(no + k * cs + R - 1)));
      }
      atomicMax(&sE[ar], m);
    }
    const bool keep = steps <= 2;                      // A digits stay in the planes for every column block
    for (int vb = 0; vb < A.vblocks && !s_fail; ++vb) {
      const int col = vb * ZN + bn;
      const bool bok = col < A.nc;
      const double* xc = A.X + A.nh * A.ldx + vb * ZN;
      if (tid < ZN) sF[tid] = 0;
      __syncthreads();
      if (bok) {
        int m = 0;
        for (int k = bg; k < ne; k += 8) {
          const double* x = xc + (long long)A.act_idx[o0 + k] * A.ldx;
          m = max(m, bexp_of(x[bn]));
          if (CPLX) m = max(m, bexp_of(x[bn ^ 1]));
        }
        if (m) atomicMax(&sF[bn], m);
      }
      auto load = [&](int st) {
        const int k0 = 32 * (CPLX ? st >> 1 : st), part = CPLX ? st & 1 : 0;
        if (!keep || vb == 0) {
#pragma unroll
          for (int q = 0; q < 4; ++q)
#pragma unroll
            for (int u = 0; u < 2; ++u) {
              const int k = k0 + 8 * ag + 2 * ((q + ash) & 3) + u;
              a[2 * q + u] = aok && k < ne ? __ldg(no + k * cs + part) : 0.0;
            }
        }
#pragma unroll
        for (int q = 0; q < 2; ++q)
#pragma unroll
          for (int u = 0; u < 2; ++u) {
            const int k = k0 + 4 * bg + 2 * (q ^ bsh) + u;
            double x = 0.0;
            if (bok && k < ne) {
              const double* xr = xc + (long long)A.act_idx[o0 + k] * A.ldx;
              x = part == 0 ? xr[bn] : (bn & 1) ? xr[bn ^ 1] : -xr[bn ^ 1];
            }
            b[2 * q + u] = x;
          }
      };
      load(0);
      __syncthreads();
      // (ne <= 256 complex or 512 real: the levels are combined once; the host checks)
      for (int st = 0; st < steps; ++st) {
        const int h = st & 1;
        const bool ok = H.wait(h, &s_fail);
        if (ok) {
          if (aok && (!keep || vb == 0)) {
            const int bm = sE[ar];
#pragma unroll
            for (int q = 0; q < 4; ++q)
              put_digits(C.sA, ZPA, ar, 32 * h + 8 * ag + 2 * ((q + ash) & 3), fixed54(a[2 * q], bm), fixed54(a[2 * q + 1], bm));
          }
          if (bok) {
            const int bm = sF[bn];
#pragma unroll
            for (int q = 0; q < 2; ++q)
              put_digits(C.sB, ZPB, bn, 32 * h + 4 * bg + 2 * (q ^ bsh), fixed54(b[2 * q], bm), fixed54(b[2 * q + 1], bm));
          }
          if (st + 1 < steps) load(st + 1);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        if (__syncthreads_or(!ok)) { s_fail = 1; break; }
        if (warp0)
          issue_half(C.taddr, C.sA, C.sB, h, st == 0, &bar[h], min(2, (ne - 32 * (CPLX ? st >> 1 : st) + 15) / 16));
        H.out[h] = true;
      }
      if (s_fail) break;
      bool ok = H.wait(0, &s_fail);
      ok = H.wait(1, &s_fail) && ok;
      if (__syncthreads_or(!ok)) { s_fail = 1; break; }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (32 * (warp & 3) < nr) {   // (uniform over the warp)
        const int r = 32 * (warp & 3) + lane, cc = 16 * (warp >> 2);
        const uint32_t tl = C.taddr + ((uint32_t)(32 * (warp & 3)) << 16) + cc;
        float4* u = A.U + (size_t)(L.q0 - A.q0 + p0 + r) * A.ncp + (vb * ZN + cc) / 2;
#pragma unroll 1
        for (int g = 0; g < 2; ++g) {
          float xh[8], xl[8];
          drain8_pairs(tl + 8 * g, sE[r], sF + cc + 8 * g, xh, xl);
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            const int col = vb * ZN + cc + 8 * g + j;
            if (r < nr && col < A.nc)
              u[4 * g + j / 2] = col + 1 < A.nc ? make_float4(xh[j], xh[j + 1], xl[j], xl[j + 1]) : make_float4(xh[j], 0.f, xl[j], 0.f);
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
    }
  }
  oz_end(C, H, &s_fail, A.err);
}

// ------------------------------------------------------------------ CFE part and the sums
constexpr int FJP = 2;       // column pairs per pass
constexpr int FT = 192;      // threads per CTA

struct FieldCcArgs {
  const Leaf* leaves;
  int l0, nl;
  const double* qxyz;
  const double* cellbox;
  const double* gll;
  const int* cell_nodes;
  const int* act_off;
  const double* X;           // real view
  long long ldx;
  int nc;                    // real columns
  int nloc;
  int64_t q0;                // first point of the batch
  const float4* U;           // enrichment part, [point][ncp]
  int ncp;
  const double* occ;         // weight per vector (density), or null: 1
  const double* qw;
  double* out;               // density: out += sum; gradient: out = scale w_q sum
  double* out2;              // with the density: w_q sum |u|^2 unweighted, or null
  double scale;
  bool density;
};

template <int P, int N1>
struct FcPlan {
  static constexpr int P2 = P * P, P3 = P2 * P, N2 = N1 * N1, N3 = N2 * N1;
  static constexpr int NB = P3 > P * N2 ? P3 : P * N2;
  static constexpr size_t SMEM = ((size_t)3 * N1 * P + (size_t)(NB + P2 * N1) * FJP) * sizeof(p2);
};

template <bool CPLX, bool DUAL, int P, int N1>
__global__ void __launch_bounds__(FT, N1 >= 8 ? 2 : 3) k_fields_cc(const FieldCcArgs A) {
  using F = FcPlan<P, N1>;
  constexpr int P2 = F::P2, P3 = F::P3, N2 = F::N2, R = CPLX ? 2 : 1;
  static_assert(N2 * FJP <= FT, "a z line per thread");
  extern __shared__ __align__(16) unsigned char fc_raw[];
  p2* L = reinterpret_cast<p2*>(fc_raw);       // [3][N1][P], both halves the same value
  p2* B = L + 3 * N1 * P;                      // X, then the (c, qy, qx) lines; [entry][FJP]
  p2* T = B + (size_t)F::NB * FJP;             // (c, b, qx) lines
  __shared__ double xn[8];
  if (threadIdx.x < P) xn[threadIdx.x] = A.gll[threadIdx.x];
  const int tz = threadIdx.x, jz = tz % FJP, lz = tz / FJP;   // this thread's z line
  for (int li = blockIdx.x; li < A.nl; li += gridDim.x) {
    const Leaf lf = A.leaves[A.l0 + li];
    if (lf.n1 != N1) continue;                 // (another instance takes it)
    const int e = lf.cell;
    const bool enr = A.act_off[e + 1] > A.act_off[e];
    const double* box = A.cellbox + 6 * e;
    __syncthreads();
    if (tz < 3 * N1) {
      const int d = tz / N1, i = tz % N1;
      const int64_t qi = lf.q0 + (d == 0 ? i : d == 1 ? i * N1 : i * N2);
      const double xi = 2.0 * (A.qxyz[3 * qi + d] - box[d]) / box[3 + d] - 1.0;
      double Lv[8], Dv[8];
      lagrange_eval(xn, P, xi, Lv, Dv);
      for (int a = 0; a < P; ++a) L[tz * P + a] = p2_dup(f2_from_int(Lv[a]));
    }
    p2 sw[N1], s1[DUAL ? N1 : 1];
#pragma unroll
    for (int q = 0; q < N1; ++q) {
      sw[q] = p2_zero();
      if (DUAL) s1[DUAL ? q : 0] = p2_zero();
    }
    for (int c0 = 0; c0 < A.nc; c0 += 2 * FJP) {
      __syncthreads();
      for (int t = tz; t < P3 * FJP; t += FT) {
        const int r = t / FJP, j = c0 + 2 * (t % FJP);
        const double* x = A.X + (long long)A.cell_nodes[(size_t)e * A.nloc + r] * A.ldx + j;
        B[t] = p2_join(j < A.nc ? f2_from_int(x[0]) : f2{0.f, 0.f}, j + 1 < A.nc ? f2_from_int(x[1]) : f2{0.f, 0.f});
      }
      __syncthreads();
      for (int t = tz; t < P2 * FJP; t += FT) {           // x lines
        const int jp = t % FJP, ln = t / FJP;
        p2 y[N1];
#pragma unroll
        for (int q = 0; q < N1; ++q) y[q] = p2_zero();
#pragma unroll 1
        for (int a = 0; a < P; ++a) {
          const p2 x = B[(a + P * ln) * FJP + jp];
#pragma unroll
          for (int q = 0; q < N1; ++q) p2_mac(y[q], L[q * P + a], x);
        }
#pragma unroll
        for (int q = 0; q < N1; ++q) T[(ln * N1 + q) * FJP + jp] = p2_fin(y[q]);
      }
      __syncthreads();
      for (int t = tz; t < P * N1 * FJP; t += FT) {       // y lines
        const int jp = t % FJP, ln = t / FJP, qx = ln % N1, c = ln / N1;
        p2 y[N1];
#pragma unroll
        for (int q = 0; q < N1; ++q) y[q] = p2_zero();
#pragma unroll 1
        for (int b = 0; b < P; ++b) {
          const p2 x = T[((c * P + b) * N1 + qx) * FJP + jp];
#pragma unroll
          for (int q = 0; q < N1; ++q) p2_mac(y[q], L[(N1 + q) * P + b], x);
        }
#pragma unroll
        for (int q = 0; q < N1; ++q) B[((c * N1 + q) * N1 + qx) * FJP + jp] = p2_fin(y[q]);
      }
      __syncthreads();
      const int j = c0 + 2 * jz;
      if (lz < N2 && j < A.nc) {                           // z line, added to the enrichment part
        p2 u[N1];
#pragma unroll
        for (int q = 0; q < N1; ++q) {
          if (enr) {
            const float4 v = __ldg(A.U + (size_t)(lf.q0 - A.q0 + q * N2 + lz) * A.ncp + j / 2);
            u[q] = p2{pk_make(v.x, v.y), pk_make(v.z, v.w)};
          } else {
            u[q] = p2_zero();
          }
        }
#pragma unroll 1
        for (int c = 0; c < P; ++c) {
          const p2 x = B[(c * N2 + lz) * FJP + jz];
#pragma unroll
          for (int q = 0; q < N1; ++q) p2_mac(u[q], L[(2 * N1 + q) * P + c], x);
        }
        const int v0 = j / R;
        const f2 wa = f2_from_int(A.occ ? A.occ[v0] : 1.0);
        const p2 w = CPLX ? p2_dup(wa) : p2_join(wa, j + 1 < A.nc ? f2_from_int(A.occ ? A.occ[v0 + 1] : 1.0) : f2{0.f, 0.f});
#pragma unroll
        for (int q = 0; q < N1; ++q) {
          const p2 v = p2_fin(u[q]), s = p2_mul(v, v);
          p2_mac(sw[q], w, s);
          // (the low part left to grow over the columns lost bits: 62-atom cell, 360 vectors, error of the density
          // against FP64 3.8e-13 of its largest value, 7.5e-14 so; 211.0 -> 214.4 ms)
          sw[q] = p2_fin(sw[q]);
          if (DUAL) s1[DUAL ? q : 0] = p2_add(s1[DUAL ? q : 0], s);
        }
      }
    }
    // sums over the two halves and the column pairs of a point
    __syncthreads();
    double* red = reinterpret_cast<double*>(B);            // [2][FJP][N1][N2]
    if (lz < N2) {
#pragma unroll
      for (int q = 0; q < N1; ++q) {
        f2 x, y;
        p2_halves(sw[q], x, y);
        red[(jz * N1 + q) * N2 + lz] = f2_to_int(x) + f2_to_int(y);
        if (DUAL) {
          p2_halves(s1[DUAL ? q : 0], x, y);
          red[((FJP + jz) * N1 + q) * N2 + lz] = f2_to_int(x) + f2_to_int(y);
        }
      }
    }
    __syncthreads();
    for (int q = tz; q < F::N3; q += FT) {
      double r = 0, r1 = 0;
#pragma unroll
      for (int jp = 0; jp < FJP; ++jp) {
        r += red[jp * F::N3 + q];
        if (DUAL) r1 += red[(FJP + jp) * F::N3 + q];
      }
      const int64_t qg = lf.q0 + q;
      if (A.density) {
        A.out[qg] += r;
      } else {
        A.out[qg] = A.scale * A.qw[qg] * r;
      }
      if (DUAL) A.out2[qg] = A.qw[qg] * r1;
    }
  }
}

}  // namespace

// sum_v w_v |u_v|^2 of the columns of X at the points, in pair mode; *done false when the order and rules of
// this context have no instance (the general kernel then runs).
int fields_pair(oefe_ctx* c, KData& K, const void* X, int nv, int ld, bool cplx, const double* occ, double* out,
                bool density, double scale, double* out2, bool* done) {
  *done = false;
  const int P = c->P, R = cplx ? 2 : 1;
  if (P < 4 || P > 7 || c->nq_cell != P || c->nq_enr != P + 2 || R * c->ne_max > ZMAXK) return OEFE_OK;
  const int ncr = nv * R, vblocks = (ncr + ZN - 1) / ZN, ncp = (ncr + 1) / 2;
  const int nl_all = (int)c->leaves.size();
  const size_t per_point = (size_t)ncp * sizeof(float4);
  std::vector<int> cut{0, nl_all};
  // the leaves in batches whose workspace takes at most cap bytes (or one leaf's): the workspace
  auto batches = [&](size_t cap) -> size_t {
    size_t ws = 0;
    int64_t q0 = 0;
    cut.assign(1, 0);
    for (int i = 0; i < nl_all; ++i) {
      const int64_t q1 = i + 1 < nl_all ? c->leaves[i + 1].q0 : c->nq;
      if ((size_t)(q1 - q0) * per_point > cap && i > cut.back()) {
        cut.push_back(i);
        q0 = c->leaves[i].q0;
      }
      ws = std::max(ws, (size_t)(q1 - q0) * per_point);
    }
    cut.push_back(nl_all);
    return ws;
  };
  const bool enr = c->nO > 0 && c->ne_max > 0;
  if (enr) {
    // a 32nd of the device at most, and no more than that leaves free; smaller batches when the allocation fails.
    // Batches of less than half a leaf per SM would leave this path slower than the general kernel, which
    // needs no workspace (2.6 times as long on a full GPU)
    size_t ws = batches(std::max(c->dev_bytes / 32, (size_t)64 << 20));
    if (ws + 256 > c->ws_bytes) ws = batches(std::min(ws, ws_room(c)));
    int st = OEFE_ERR_OOM;
    while ((int)cut.size() == 2 || ((long long)cut.size() - 1) * (c->num_sms / 2) <= nl_all) {
      st = ensure_ws(c, ws + 256);
      if (st != OEFE_ERR_OOM || (int)cut.size() > nl_all) break;
      ws = batches(ws / 2);
    }
    if (st == OEFE_ERR_OOM) return OEFE_OK;
    OEFE_TRY(st);
  }
  const int n1m = std::max(c->nq_cell, c->nq_enr);
  for (size_t bi = 0; bi + 1 < cut.size(); ++bi) {
    const int l0 = cut[bi], nl = cut[bi + 1] - l0;
    const int64_t q0 = c->leaves[l0].q0;
    if (enr) {
      FieldOzArgs A;
      A.leaves = c->d_leaves;
      A.l0 = l0;
      A.nl = nl;
      A.act_off = c->d_act_off;
      A.act_idx = c->d_act_idx;
      A.ne_max = c->ne_max;
      A.mtiles = (n1m * n1m * n1m + 127) / 128;
      A.nh = c->nh;
      A.NO = (const double*)K.NO;
      A.X = (const double*)X;
      A.ldx = (long long)ld * R;
      A.nc = ncr;
      A.vblocks = vblocks;
      A.q0 = q0;
      A.U = (float4*)c->ws;
      A.ncp = ncp;
      A.err = c->d_status + 2;
      const int grid = (int)std::min<long long>((long long)nl * A.mtiles, c->num_sms);
      auto go = [&](auto kern) -> int {
        OEFE_CUDA_TRY(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)OZ_SMEM));
        OEFE_COUNTED kern<<<grid, FZ, OZ_SMEM, c->stream>>>(A);
        return OEFE_OK;
      };
      OEFE_TRY(cplx ? go(k_fields_oz<true>) : go(k_fields_oz<false>));
    }
    FieldCcArgs A;
    A.leaves = c->d_leaves;
    A.l0 = l0;
    A.nl = nl;
    A.qxyz = c->d_qxyz;
    A.cellbox = c->d_cellbox;
    A.gll = c->d_gll;
    A.cell_nodes = c->d_cell_nodes;
    A.act_off = c->d_act_off;
    A.X = (const double*)X;
    A.ldx = (long long)ld * R;
    A.nc = ncr;
    A.nloc = c->nloc;
    A.q0 = q0;
    A.U = (const float4*)c->ws;
    A.ncp = ncp;
    A.occ = occ;
    A.qw = c->d_qw;
    A.out = out;
    A.out2 = out2;
    A.scale = scale;
    A.density = density;
    const int grid = std::min(nl, (n1m >= 8 ? 2 : 3) * c->num_sms);
    auto go = [&](auto kern, size_t smem) -> int {
      OEFE_CUDA_TRY(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
      OEFE_COUNTED kern<<<grid, FT, smem, c->stream>>>(A);
      return OEFE_OK;
    };
#define OEFE_FC1(p, q)                                                                                              \
  if (P == p)                                                                                                       \
    OEFE_TRY(cplx ? (out2 ? go(k_fields_cc<true, true, p, q>, FcPlan<p, q>::SMEM) : go(k_fields_cc<true, false, p, q>, FcPlan<p, q>::SMEM)) \
                  : (out2 ? go(k_fields_cc<false, true, p, q>, FcPlan<p, q>::SMEM) : go(k_fields_cc<false, false, p, q>, FcPlan<p, q>::SMEM)));
    OEFE_FC1(4, 4) OEFE_FC1(4, 6) OEFE_FC1(5, 5) OEFE_FC1(5, 7) OEFE_FC1(6, 6) OEFE_FC1(6, 8) OEFE_FC1(7, 7) OEFE_FC1(7, 9)
#undef OEFE_FC1
    OEFE_CUDA_TRY(c, cudaGetLastError());
  }
  *done = true;
  return OEFE_OK;
}
