// Dense blocks of the FP64-class cell products of pair mode (Eq. HOEFEelelements) on the tensor
// cores: the whole matrix of the refined cells, and of every single-leaf cell the blocks that
// couple the enrichment rows (H_CO X_O, added to by the sum factorization of sumfac.cu, and
// H_OC X_C + H_OO X_O).
//
// Arithmetic: fixed point under one exponent per matrix row and one per vector column of a cell.
// A value is cut into 8 balanced digits of 7 bits (each in [-64, 64), exact in bf16), 54 bits of the
// row's (column's) largest value, more than an FP64 significand; the 36 digit products of levels
// s + t <= 7 accumulate exactly in FP32 (products at most 2^12, 8 pairs a level, so 512 entries of K
// stay below 2^24), the levels combine in integers and round once to FP64. Error about 2^-53 of the
// row maximum times the column maximum per term.
//
// Layout: one job = 128 matrix rows (M) x 64 real vector columns (N; complex data interleaved, so 32
// vectors) x all of K in chunks of 64 real entries (complex: 32 columns as [Re | Im], against
// [X; i X]). The digits are cut inside the kernel straight from the stored FP64 matrix (no digit
// planes in memory, no second copy of the matrix: these planes would be 16 bytes an entry), 8 planes
// of A (128 KB) and of B (64 KB) in shared memory, 8 accumulators of 64 columns fill tensor memory.
// Bound: per chunk the cut (12288 values, about 40 integer instructions each, over 256 threads: 4.8 k
// clocks) and the 144 MMAs (128 x 64 x 16: 4.6 k clocks), which take turns on the one buffer; the
// loads of the next chunk run under the MMAs. The FP64 pipe (2 multiply-adds a clock per SM) is
// not used at all.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>
#include <vector>

#include "oefe_internal.h"
#include "tcgen05_dev.cuh"

namespace {

constexpr int ZT = 256;                 // threads per CTA
constexpr int ZS = 8;                   // digits per value
constexpr int ZK = 64;                  // real K entries per chunk
constexpr int ZN = 64;                  // real vector columns per job
constexpr int ZPA = 128 * 128;          // bytes of an A plane (128 rows x 64 bf16)
constexpr int ZPB = ZN * 128;           // bytes of a B plane
constexpr int ZMAXCH = 8;               // chunks accumulated before the levels are combined
constexpr int ZCOLS = 512;              // tensor-memory columns: 8 levels x 64
// level sums: at most ZS digit pairs of products at most 2^12 over ZMAXCH ZK entries
static_assert((long long)ZS * ZMAXCH * ZK * (1LL << 12) <= (1LL << 24), "level sums must be exact in FP32");

struct OzJob {
  long long hoff;    // first scalar of the job's rows in the stored matrix (at column k0)
  int stride;        // scalars per row
  int cell, r0, nr;  // matrix rows r0 .. r0 + nr of the cell
  int k0, K;         // matrix columns k0 .. k0 + K
};

struct OzCellArgs {
  const OzJob* jobs;
  int njobs, vblocks;
  const double* H;
  const int* rexp;          // largest biased exponent per (cell, row) over the job's columns
  const double* X;          // real view: ldx reals per row
  long long ldx;
  int nvr;                  // real columns
  const int* cell_nodes;
  const int* act_off;
  const int* act_idx;
  int nloc, npad;
  int64_t nh;
  double* Z;                // real view: nvr per row
  int* err;
};

__device__ __forceinline__ int bexp_of(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7FF); }

// trunc(|x| 2^(54-E)) with the sign of x, plus 64 in every base-128 position, where the largest
// biased exponent of the row is bm (|x| < 2^E, E = bm - 1022); zeros and subnormals count as zero.
// 54 bits: with 55 a value just below 2^E would carry out of the top digit.
__device__ __forceinline__ unsigned long long fixed56(double x, int bm) {
  constexpr unsigned long long BIAS = 0x81020408102040ull;   // 64 (1 + 2^7 + .. + 2^49)
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7FF);
  unsigned long long m = (((b << 1) & 0x1FFFFFFFFFFFFEull) | (1ull << 53)) >> min(bm - ex, 63);
  if (ex == 0) m = 0;
  return (b >> 63) ? BIAS - m : BIAS + m;
}

// the digits of two neighbouring K entries of operand row r, one packed word per plane; plane 0 holds
// the leading digits
__device__ __forceinline__ void put_digits(unsigned char* base, int plane, int r, int kk, unsigned long long y0,
                                           unsigned long long y1) {
  unsigned char* p = base + swz(r, kk);
  const __nv_bfloat162 off = __nv_bfloat162(__ushort_as_bfloat16(0x4340), __ushort_as_bfloat16(0x4340));   // 192
#pragma unroll
  for (int i = 0; i < ZS; ++i) {
    // 128 + u as bf16 bits is 0x4300 | u for a 7-bit u; minus 192: the balanced digit
    const unsigned w = (__byte_perm((unsigned)(y0 >> (7 * i)), (unsigned)(y1 >> (7 * i)), 0x5410) & 0x007F007Fu) | 0x43004300u;
    *reinterpret_cast<__nv_bfloat162*>(p + (size_t)(ZS - 1 - i) * plane) =
        __hsub2(*reinterpret_cast<const __nv_bfloat162*>(&w), off);
  }
}

// the sum of the levels of one entry, T = sum_d lev_d 128^(7-d) in units of 2^(E + F - 59), exact in
// 128 bits (|T| < 2^71) and rounded once
__device__ __forceinline__ double from_levels(const float* v, int bsum) {
  long long hi = 0, lo = 0;
#pragma unroll
  for (int d = 0; d < 4; ++d) hi = hi * 128 + __float2int_rn(v[d]);
#pragma unroll
  for (int d = 4; d < 8; ++d) lo = lo * 128 + __float2int_rn(v[d]);
  unsigned long long tl = ((unsigned long long)hi << 28) + (unsigned long long)lo;
  long long th = (hi >> 36) + (lo >> 63) + (tl < (unsigned long long)lo ? 1 : 0);
  const bool neg = th < 0;
  if (neg) {
    tl = 0ull - tl;
    th = ~th + (tl == 0 ? 1 : 0);
  }
  if ((tl | (unsigned long long)th) == 0) return 0.0;
  unsigned long long nrm;   // leading 64 bits; T = nrm 2^(64 - lz)
  int lz;
  if (th) {
    lz = __clzll(th);
    nrm = ((unsigned long long)th << lz) | (tl >> (64 - lz));       // th < 2^7, so lz > 0
  } else {
    const int z = __clzll((long long)tl);
    nrm = tl << z;
    lz = 64 + z;
  }
  const unsigned long long r = (nrm >> 11) + ((nrm >> 10) & 1);     // 53 bits, rounded
  const int f = bsum - 2044 + 1091 - lz;                            // exponent field of r 2^(E + F - 59 + 75 - lz)
  double x;
  if (f >= 1 && f <= 2045) x = __longlong_as_double((long long)(((unsigned long long)f << 52) + (r - (1ull << 52))));
  else x = ldexp((double)r, f - 1075);
  return neg ? -x : x;
}

// 8 columns of four consecutive levels (32 lanes), complete on return
__device__ __forceinline__ void tmem_ld_levels(uint32_t taddr, float (*v)[8]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%32];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%8,%9,%10,%11,%12,%13,%14,%15}, [%33];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%16,%17,%18,%19,%20,%21,%22,%23}, [%34];\n"
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%24,%25,%26,%27,%28,%29,%30,%31}, [%35];\n"
      "tcgen05.wait::ld.sync.aligned;\n"
      : "=&r"(r[0]), "=&r"(r[1]), "=&r"(r[2]), "=&r"(r[3]), "=&r"(r[4]), "=&r"(r[5]), "=&r"(r[6]), "=&r"(r[7]), "=&r"(r[8]), "=&r"(r[9]), "=&r"(r[10]), "=&r"(r[11]), "=&r"(r[12]), "=&r"(r[13]), "=&r"(r[14]), "=&r"(r[15]), "=&r"(r[16]), "=&r"(r[17]), "=&r"(r[18]), "=&r"(r[19]), "=&r"(r[20]), "=&r"(r[21]), "=&r"(r[22]), "=&r"(r[23]), "=&r"(r[24]), "=&r"(r[25]), "=&r"(r[26]), "=&r"(r[27]), "=&r"(r[28]), "=&r"(r[29]), "=&r"(r[30]), "=&r"(r[31])
      : "r"(taddr), "r"(taddr + ZN), "r"(taddr + 2 * ZN), "r"(taddr + 3 * ZN));
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i / 8][i % 8] = __uint_as_float(r[i]);
}

template <bool CPLX>
__global__ void __launch_bounds__(ZT, 1) k_cell_oz(const OzCellArgs A) {
  constexpr int CK = CPLX ? 32 : 64;     // matrix columns per chunk
  extern __shared__ __align__(1024) unsigned char oz_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)oz_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* sA = sm;
  unsigned char* sB = sm + ZS * ZPA;
  int* rows = (int*)(sB + ZS * ZPB);     // row of X of every matrix column of the job
  __shared__ int sE[128], sF[ZN];
  __shared__ uint64_t mma_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_slot)), "r"(ZCOLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    mbar_init(&mma_bar, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t taddr = tmem_slot;
  const int bn = tid & 63, bg = tid >> 6;            // B: operand column, group of 16 K entries
  const int sh = (bn >> 3) & 3;                      // rotation of the pairs: stores free of bank conflicts
  uint32_t phase = 0;
  bool mma_out = false;
  const long long total = (long long)A.njobs * A.vblocks;
  for (long long job = blockIdx.x; job < total; job += gridDim.x) {
    const OzJob J = A.jobs[job / A.vblocks];
    const int c0 = (int)(job % A.vblocks) * ZN;      // first real column
    const int e = J.cell;
    for (int k = tid; k < J.K; k += ZT) {
      const int col = J.k0 + k;
      rows[k] = col < A.nloc ? A.cell_nodes[(size_t)e * A.nloc + col] : (int)(A.nh + A.act_idx[A.act_off[e] + col - A.nloc]);
    }
    if (tid < 128) sE[tid] = tid < J.nr ? A.rexp[(size_t)e * A.npad + J.r0 + tid] : 0;
    if (tid < ZN) sF[tid] = 0;
    __syncthreads();
    const bool cok = c0 + bn < A.nvr;
    {   // exponents of the vector columns over K (complex: of both parts of a vector)
      int mex = 0;
      const int cb = CPLX ? (c0 + bn) & ~1 : c0 + bn;
      if (cok) {
        int k = bg;
        for (; k + 12 < J.K; k += 16) {
          double v[8];
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            const double* x = A.X + (long long)rows[k + 4 * u] * A.ldx + cb;
            v[2 * u] = x[0];
            v[2 * u + 1] = CPLX ? x[1] : 0.0;
          }
#pragma unroll
          for (int u = 0; u < 8; ++u) mex = max(mex, bexp_of(v[u]));
        }
        for (; k < J.K; k += 4) {
          const double* x = A.X + (long long)rows[k] * A.ldx + cb;
          mex = max(mex, bexp_of(x[0]));
          if (CPLX) mex = max(mex, bexp_of(x[1]));
        }
      }
      atomicMax(&sF[bn], mex);
    }
    __syncthreads();
    const int nch = (J.K + CK - 1) / CK;
    const int rw0 = warp * 16;                        // A: rows of this warp, lane l the entries 2 l, 2 l + 1
    const int nrw = max(0, min(16, J.nr - rw0));
    double va[32], vb[16];
    // operand values of a chunk: A entry kk of row r, B entry kk of column bn
    auto load = [&](int ch) {
      const int kb = ch * CK;
      const int kl = CPLX ? (2 * lane) & 31 : 2 * lane;   // matrix columns kb + kl, kb + kl + 1
      const bool k0ok = kb + kl < J.K, k1ok = kb + kl + 1 < J.K;
      const double* h = CPLX ? A.H + 2 * (J.hoff + (long long)rw0 * J.stride + kb + kl) + (lane >> 4)
                             : A.H + J.hoff + (long long)rw0 * J.stride + kb + kl;
      const long long st = CPLX ? 2ll * J.stride : J.stride;
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        va[2 * i] = i < nrw && k0ok ? __ldg(h + i * st) : 0.0;
        va[2 * i + 1] = i < nrw && k1ok ? __ldg(h + i * st + (CPLX ? 2 : 1)) : 0.0;
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const int kk = 16 * bg + 2 * ((q + sh) & 7);
#pragma unroll
        for (int u = 0; u < 2; ++u) {
          double x = 0.0;
          if (cok) {
            if (!CPLX) {
              if (kb + kk + u < J.K) x = A.X[(long long)rows[kb + kk + u] * A.ldx + c0 + bn];
            } else {   // entries 0 .. 31: X; 32 .. 63: i X
              const int k = kb + ((kk + u) & 31);
              if (k < J.K) {
                const double* xr = A.X + (long long)rows[k] * A.ldx + c0;
                x = kk < 32 ? xr[bn] : ((bn & 1) ? xr[bn ^ 1] : -xr[bn ^ 1]);
              }
            }
          }
          vb[2 * q + u] = x;
        }
      }
    };
    load(0);
    bool have = false;   // an earlier part of K is in Z already
    for (int ch = 0; ch < nch; ++ch) {
      if (mma_out) {   // the previous chunk's MMAs have read the planes
        const bool ok = mbar_wait(&mma_bar, phase, &s_fail);
        if (__syncthreads_or(!ok)) { s_fail = 1; break; }
        phase ^= 1;
        mma_out = false;
      }
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        if (i >= nrw) break;
        const int r = rw0 + i, bm = sE[r];
        put_digits(sA, ZPA, r, 2 * lane, fixed56(va[2 * i], bm), fixed56(va[2 * i + 1], bm));
      }
      {
        const int bm = sF[bn];
#pragma unroll
        for (int q = 0; q < 8; ++q)
          put_digits(sB, ZPB, bn, 16 * bg + 2 * ((q + sh) & 7), fixed56(vb[2 * q], bm), fixed56(vb[2 * q + 1], bm));
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncthreads();
      if (tid == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        constexpr uint32_t ID = idesc_bf16(128, ZN, false);
        const bool first = ch % ZMAXCH == 0;
        const uint32_t a0 = smem_u32(sA), b0 = smem_u32(sB);
        const int nks = CPLX ? ZK / 16 : min(ZK / 16, (J.K - ch * CK + 15) / 16);
#pragma unroll 1
        for (int d = 0; d < ZS; ++d)
#pragma unroll 1
          for (int s = 0; s <= d; ++s)
            for (int ks = 0; ks < nks; ++ks)
              mma_bf16(taddr + d * ZN, sdesc(a0 + s * ZPA + ks * 32), sdesc(b0 + (d - s) * ZPB + ks * 32), ID,
                       (first && s == 0 && ks == 0) ? 0u : 1u);
        mma_commit(&mma_bar);
      }
      mma_out = true;
      if (ch + 1 < nch) load(ch + 1);
      if (ch + 1 < nch && (ch + 1) % ZMAXCH != 0) continue;
      // the levels of this thread's row and 32 columns
      {
        const bool ok = mbar_wait(&mma_bar, phase, &s_fail);
        if (__syncthreads_or(!ok)) { s_fail = 1; break; }
        phase ^= 1;
        mma_out = false;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int r = 32 * (warp & 3) + lane, cc = 32 * (warp >> 2);
      if (32 * (warp & 3) < J.nr) {   // (uniform over the warp)
        const uint32_t tl = taddr + ((uint32_t)(32 * (warp & 3)) << 16) + cc;
        const int bE = sE[r];
        double* z = A.Z + ((size_t)e * A.npad + J.r0 + r) * A.nvr + c0 + cc;
#pragma unroll
        for (int g = 0; g < 4; ++g) {
          float v[8][8];
          tmem_ld_levels(tl + 8 * g, v);
          tmem_ld_levels(tl + 4 * ZN + 8 * g, v + 4);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const int n = cc + 8 * g + j, bF = sF[n];
            const float lv[8] = {v[0][j], v[1][j], v[2][j], v[3][j], v[4][j], v[5][j], v[6][j], v[7][j]};
            double x = from_levels(lv, bE + bF);
            if (bE == 0x7FF || bF == 0x7FF) x = __longlong_as_double(0x7FF8000000000000ll);   // an infinity or NaN
            if (r < J.nr && c0 + n < A.nvr) z[8 * g + j] = have ? z[8 * g + j] + x : x;
          }
        }
      }
      have = true;
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncthreads();
    }
    if (s_fail) break;
  }
  if (tid == 0 && mma_out) mbar_wait_drain(&mma_bar, phase);
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (s_fail && tid == 0) atomicExch(A.err, 1);
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ZCOLS) : "memory");
}

// largest biased exponent of every job row over its columns (a warp per row)
__global__ void k_oz_row_exps(const OzJob* jobs, const double* H, int R, int npad, int* rexp) {
  const OzJob J = jobs[blockIdx.x];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int r = warp; r < J.nr; r += blockDim.x / 32) {
    const double* h = H + R * (J.hoff + (long long)r * J.stride);
    int m = 0;
    for (int k = lane; k < R * J.K; k += 32) m = max(m, bexp_of(h[k]));
    m = (int)__reduce_max_sync(0xffffffffu, (unsigned)m);
    if (lane == 0) rexp[(size_t)J.cell * npad + J.r0 + r] = m;
  }
}

}  // namespace

// Job tables (for the full and the compact matrix layout) of the current cells and enrichment; the
// longest jobs first, so that the round-robin over the CTAs ends evenly.
int oz_setup_jobs(oefe_ctx* c, bool compact) {
  void** table = compact ? &c->d_oz_jobs_c : &c->d_oz_jobs;
  if (*table) return OEFE_OK;
  std::vector<OzJob> jobs;
  const size_t npad = c->npad, strip = compact_strip(c);
  const size_t base = (size_t)c->n_dense * npad * npad;
  for (int kind = 0; kind < 3; ++kind) {   // refined cells; enrichment rows; node rows of single-leaf cells
    const std::vector<int>& list = kind == 0 ? c->dense_cells_h : c->sf_cells_h;
    for (size_t i = 0; i < list.size(); ++i) {
      const int e = list[i], ne = c->act_off[e + 1] - c->act_off[e], naug = c->nloc + ne;
      const int ra = kind == 1 ? c->nloc : 0, rb = kind == 2 ? c->nloc : naug;
      if (kind && ne == 0) continue;
      for (int r = ra; r < rb; r += 128) {
        OzJob J;
        J.cell = e;
        J.r0 = r;
        J.nr = std::min(128, rb - r);
        J.k0 = kind == 2 ? c->nloc : 0;
        J.K = kind == 2 ? ne : naug;
        if (!compact) {
          J.hoff = (long long)(((size_t)e * npad + r) * npad + J.k0);
          J.stride = (int)npad;
        } else if (kind == 0) {
          J.hoff = (long long)((i * npad + r) * npad);
          J.stride = (int)npad;
        } else if (kind == 1) {
          J.hoff = (long long)(base + i * strip + (size_t)c->nloc * c->ne_max + (size_t)(r - c->nloc) * npad);
          J.stride = (int)npad;
        } else {
          J.hoff = (long long)(base + i * strip + (size_t)r * c->ne_max);
          J.stride = c->ne_max;
        }
        jobs.push_back(J);
      }
    }
  }
  c->n_oz_jobs = (int)jobs.size();
  if (jobs.empty()) return OEFE_OK;
  OEFE_TRY(dev_alloc(c, table, jobs.size() * sizeof(OzJob)));
  OEFE_CUDA_TRY(c, cudaMemcpyAsync(*table, jobs.data(), jobs.size() * sizeof(OzJob), cudaMemcpyHostToDevice, c->stream));
  OEFE_CUDA_TRY(c, cudaStreamSynchronize(c->stream));
  return OEFE_OK;
}

// Row exponents of a freshly built operator (one read of its dense blocks)
int oz_operator_ready(oefe_ctx* c, KData& K) {
  OEFE_TRY(oz_setup_jobs(c, K.compact));
  if (c->n_oz_jobs == 0) return OEFE_OK;
  if (!K.rexp) OEFE_TRY(dev_alloc(c, (void**)&K.rexp, (size_t)c->ncells * c->npad * sizeof(int)));
  OEFE_COUNTED k_oz_row_exps<<<c->n_oz_jobs, 256, 0, c->stream>>>((const OzJob*)(K.compact ? c->d_oz_jobs_c : c->d_oz_jobs),
                                                                  K.H64, K.cplx ? 2 : 1, c->npad, K.rexp);
  OEFE_CUDA_TRY(c, cudaGetLastError());
  return OEFE_OK;
}

// The dense blocks' products of nv columns of X into Z (ncells x npad x nv)
int launch_cell_oz(oefe_ctx* c, const KData& K, const void* X, int ldx, int nv, bool cplx, void* Z, cudaStream_t st) {
  if (c->n_oz_jobs == 0) return OEFE_OK;
  const int R = cplx ? 2 : 1;
  OzCellArgs A;
  A.jobs = (const OzJob*)(K.compact ? c->d_oz_jobs_c : c->d_oz_jobs);
  A.njobs = c->n_oz_jobs;
  A.nvr = nv * R;
  A.vblocks = (A.nvr + ZN - 1) / ZN;
  A.H = K.H64;
  A.rexp = K.rexp;
  A.X = (const double*)X;
  A.ldx = (long long)ldx * R;
  A.cell_nodes = c->d_cell_nodes;
  A.act_off = c->d_act_off;
  A.act_idx = c->d_act_idx;
  A.nloc = c->nloc;
  A.npad = c->npad;
  A.nh = c->nh;
  A.Z = (double*)Z;
  A.err = c->d_status;
  const size_t smem = 1024 + (size_t)ZS * (ZPA + ZPB) + (size_t)c->npad * sizeof(int);
  if (smem > 226 * 1024) { c->err = "cell products: cell matrices too large"; return OEFE_ERR_ARG; }
  const int grid = (int)std::min<long long>((long long)A.njobs * A.vblocks, c->num_sms);
  auto go = [&](auto kern) -> int {
    OEFE_CUDA_TRY(c, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    OEFE_COUNTED kern<<<grid, ZT, smem, st>>>(A);
    OEFE_CUDA_TRY(c, cudaGetLastError());
    return OEFE_OK;
  };
  return cplx ? go(k_cell_oz<true>) : go(k_cell_oz<false>);
}
