// FP64-class Gram matrices of wide vector blocks (more than the 64 vectors the plane-based kernels of
// ozaki_gram.cu take) on the tensor cores, for the projected matrices of Rayleigh-Ritz (the signs of its
// vectors follow their last bits; oz8_wide.cu is the faster kernel), with the same exact bf16 digit
// slicing (the Ozaki scheme): every operand value is cut into 7 digits of 7 bits under a common
// exponent per operand row and K chunk, the 28 digit products of levels d = s + t <= 6 are
// accumulated exactly in FP32 in tensor memory (7 accumulators of 64 columns), and the levels are
// combined in FP32 pairs, scaled by exact powers of two and summed over the chunks in pairs.
//
// Unlike the plane-based kernels, the digits are cut inside the MMA kernels into shared memory
// (nothing is staged in global memory), so wide blocks need no digit planes the size of the operands. One round = one K chunk of 64 real entries for one
// tile of 128 operand rows and 64 output columns: 112 MMAs (M 128, N 64, K 16).
//
//   Gram S = X^+ W: real form A = [Re X | Im X]^T (2 nv operand rows, nv for real data), B = [Re W |
//   Im W] (2 nv columns); K = the rows of the blocks in passes of 64. A CTA takes one (128-row,
//   64-column) tile of D = A B over a range of passes; D's partial sums are combined afterwards:
//   Re S = D[i][j] + D[nv+i][nv+j], Im S = D[i][nv+j] - D[nv+i][j].
//
// Every wait is bounded; on a timeout the CTA raises the error flag, lets its copies and MMAs in
// flight land, frees its tensor memory and returns.
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include "oefe_internal.h"
#include "pair_dev.cuh"
#include "tcgen05_dev.cuh"
#include "ozaki_dev.cuh"

namespace {

constexpr int WT = 256;                 // threads per CTA
constexpr int WK = 64;                  // real K entries per round (one 128-byte swizzle row of bf16)
constexpr int WN = 64;                  // output columns per round
constexpr int PLA = 128 * 128;          // bytes of one A digit plane: 128 operand rows x 64 bf16
constexpr int PLB = WN * 128;           // bytes of one B digit plane: 64 rows x 64 bf16
constexpr size_t WSMEM = 1024 + (size_t)OZ_S * PLA + (size_t)OZ_S * PLB;
constexpr int WTCOLS = 512;             // tensor-memory columns (7 x 64 used)
// the FP32 accumulation of a level (at most OZ_S digit pairs, products at most 2^14) over the
// WK entries of a round stays exact
static_assert((long long)OZ_S * WK * (1LL << 14) <= (1LL << 24), "level sums must be exact in FP32");

__device__ __forceinline__ int bexp(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7FF); }

// the 7 digits of two consecutive K entries (kk, kk + 1) of operand row r into the planes at base
__device__ __forceinline__ void put_pair(unsigned char* base, int plane_bytes, int r, int kk, double v0, double v1,
                                         int E) {
  float c0[OZ_S], c1[OZ_S];
  digits7((unsigned long long)__double_as_longlong(v0), E, c0);
  digits7((unsigned long long)__double_as_longlong(v1), E, c1);
#pragma unroll
  for (int s = 0; s < OZ_S; ++s)
    *reinterpret_cast<__nv_bfloat162*>(base + (size_t)s * plane_bytes + swz(r, kk)) = __floats2bfloat162_rn(c0[s], c1[s]);
}

// the levels of (row, 32 columns ch*32 ..) combined and added to the running pair sums R:
// levels 6..4 by FP32 Horner steps in units of level 4, levels 3..0 in pairs, scaled by
// 2^(E + F_col - 14) (exact powers of two)
__device__ __forceinline__ void add_levels(uint32_t taddr, uint32_t lane_base, int ch, int E, const int* Fexp,
                                           f2* R) {
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    const int c0 = ch * 32 + 16 * g;
    float lo[16];
    {
      float v[16];
      tmem_ld16(taddr + lane_base + 6 * WN + c0, v);
#pragma unroll
      for (int c = 0; c < 16; ++c) lo[c] = v[c];
#pragma unroll
      for (int d = 5; d >= 4; --d) {
        tmem_ld16(taddr + lane_base + d * WN + c0, v);
#pragma unroll
        for (int c = 0; c < 16; ++c) lo[c] = __fmaf_rn(lo[c], 0.0078125f, v[c]);
      }
    }
    f2 S[16];
#pragma unroll
    for (int c = 0; c < 16; ++c) S[c] = f2{__fmul_rn(lo[c], 3.7252902984619141e-09f), 0.0f};   // 2^-28
#pragma unroll 1
    for (int d = 3; d >= 0; --d) {
      float v[16];
      tmem_ld16(taddr + lane_base + d * WN + c0, v);
      const float w = __int_as_float((127 - 7 * d) << 23);   // 2^(-7 d)
#pragma unroll
      for (int c = 0; c < 16; ++c) S[c] = f2_add(S[c], f2{__fmul_rn(v[c], w), 0.0f});
    }
#pragma unroll
    for (int c = 0; c < 16; ++c) {
      const int sc = E + Fexp[c0 + c] - 14;
      f2 x;
      if (sc > -127 && sc < 128) {
        const float w = __int_as_float((sc + 127) << 23);
        x = f2{__fmul_rn(S[c].h, w), __fmul_rn(S[c].l, w)};
      } else {
        x = f2{ldexpf(S[c].h, sc), ldexpf(S[c].l, sc)};
      }
      R[16 * g + c] = f2_add(R[16 * g + c], x);
    }
  }
}

__device__ __forceinline__ void tmem_alloc_cta(uint32_t* slot) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(WTCOLS)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_free_cta(uint32_t taddr) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(WTCOLS) : "memory");
}

// operand value of the Gram's real form: index ra < nv the real part of column ra, nv <= ra < 2 nv
// the imaginary part of column ra - nv (complex), zero beyond
__device__ __forceinline__ double gram_op(const void* M, int ld, long long g, int ra, int nv, bool cplx) {
  if (!cplx) return ra < nv ? reinterpret_cast<const double*>(M)[g * ld + ra] : 0.0;
  if (ra < nv) return reinterpret_cast<const cd*>(M)[g * ld + ra].x;
  if (ra < 2 * nv) return reinterpret_cast<const cd*>(M)[g * ld + ra - nv].y;
  return 0.0;
}

struct WGramArgs {
  const void* X;
  int ldx;
  const void* W;
  int ldw;
  long long n;
  int nv;
  bool cplx;
  int nI, nJ;                // tiles of 128 A rows and 64 B columns of D
  bool upper;                // symmetric result: only the tiles (I, J >= 2 I) that meet the upper triangle
  long long passes, ppc;     // passes of 64 rows, passes per CTA
  double* part;              // [block][I][J][128][64]
  int* err;
};

__global__ void __launch_bounds__(WT, 1) k_gram_wide(const WGramArgs A) {
  extern __shared__ __align__(1024) unsigned char wz_raw[];
  unsigned char* sm = (unsigned char*)(((uintptr_t)wz_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* sA = sm;
  unsigned char* sB = sm + OZ_S * PLA;
  __shared__ int sE[128], Fexp[WN];
  __shared__ uint64_t mma_bar;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5;
  const bool warp0 = __shfl_sync(0xffffffffu, warp, 0) == 0;   // (uniform)
  if (warp == 0) tmem_alloc_cta(&tmem_slot);
  if (tid == 0) {
    mbar_init(&mma_bar, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t taddr = tmem_slot;
  int I = blockIdx.y / A.nJ, J = blockIdx.y % A.nJ;
  if (A.upper) {   // blockIdx.y enumerates the tiles with J >= 2 I row by row
    int y = blockIdx.y;
    I = 0;
    while (y >= A.nJ - 2 * I) {
      y -= A.nJ - 2 * I;
      ++I;
    }
    J = 2 * I + y;
  }
  const long long pb = (long long)blockIdx.x * A.ppc, pe = min(A.passes, pb + A.ppc);
  const int row = tid & 127, ch = tid >> 7;
  const uint32_t lane_base = (uint32_t)(32 * (warp & 3)) << 16;
  f2 R[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) R[j] = f2{0.0f, 0.0f};
  int it = 0;
  bool mma_out = false;
  for (long long p = pb; p < pe; ++p, ++it) {
    const long long g0 = p * 64;
    const int ng = (int)min(64ll, A.n - g0);
    // digits: threads 0..127 one A operand row each, threads 128..191 one B operand column each,
    // over the pass's 64 rows (a warp's loads of one row are consecutive columns)
    if (tid < 192) {
      const bool isA = tid < 128;
      const int r = isA ? tid : tid - 128;
      const int ra = isA ? I * 128 + r : J * WN + r;
      const void* M = isA ? A.X : A.W;
      const int ld = isA ? A.ldx : A.ldw;
      // register u holds K entry (u + 2 s) mod 64, s = (r / 8) mod 4: at the store of register pair q
      // the 32 lanes of a warp (rows with 8 values of r mod 8, 4 of s) write 32 different banks
      const int sh = 2 * ((r >> 3) & 3);
      double v[64];
      int mex = 0;
#pragma unroll
      for (int u = 0; u < 64; ++u) {
        const int kk = (u + sh) & 63;
        v[u] = kk < ng ? gram_op(M, ld, g0 + kk, ra, A.nv, A.cplx) : 0.0;
        mex = max(mex, bexp(v[u]));
      }
      const int E = mex ? mex - 1022 : 0;
      unsigned char* base = isA ? sA : sB;
      const int pbytes = isA ? PLA : PLB;
#pragma unroll
      for (int q = 0; q < 32; ++q) put_pair(base, pbytes, r, (2 * q + sh) & 63, v[2 * q], v[2 * q + 1], E);
      if (isA) sE[r] = E;
      else Fexp[r] = E;
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncthreads();
    if (warp0) {   // the digit products of levels d = s + t <= 6 into accumulator d
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t lead = elect_lane();
      issue_digit_levels<OZ_S, WK / 16, PLA, PLB, WN>(lead, taddr, smem_u32(sA), smem_u32(sB), idesc_bf16(128, WN, false), WK / 16, true);
      mma_commit_lead(lead, &mma_bar);
    }
    mma_out = true;
    const bool ok = mbar_wait(&mma_bar, (uint32_t)(it & 1), &s_fail);
    if (__syncthreads_or(!ok)) { s_fail = 1; break; }
    mma_out = false;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    add_levels(taddr, lane_base, ch, sE[row], Fexp, R);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
  }
  if (tid == 0 && s_fail && mma_out) mbar_wait_drain(&mma_bar, (uint32_t)(it & 1));
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (!s_fail) {
    double* out = A.part + ((((size_t)blockIdx.x * A.nI + I) * A.nJ + J) * 128 + row) * WN + ch * 32;
#pragma unroll
    for (int j = 0; j < 32; ++j) out[j] = f2_to(R[j]);
  }
  if (s_fail && tid == 0) atomicExch(A.err, 1);
  if (warp == 0) tmem_free_cta(taddr);
}

// S from the partial sums of all blocks (real form combined for complex data)
template <typename S>
__global__ void k_gram_wide_reduce(const double* part, int nbx, int nI, int nJ, int nv, bool upper, S* out) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= nv * nv) return;
  // upper (real symmetric result): entry (i, j) below the diagonal is entry (j, i), which lies in a
  // computed tile (column tile j / 64 >= 2 (row tile i / 128) whenever i <= j)
  const int i = upper ? min(t / nv, t % nv) : t / nv, j = upper ? max(t / nv, t % nv) : t % nv;
  auto D = [&](int ra, int rb) {
    double s = 0.0;
    for (int b = 0; b < nbx; ++b)
      s += part[((((size_t)b * nI + ra / 128) * nJ + rb / WN) * 128 + ra % 128) * WN + rb % WN];
    return s;
  };
  if constexpr (sizeof(S) == sizeof(cd)) out[t] = mkc(D(i, j) + D(nv + i, nv + j), D(i, nv + j) - D(nv + i, j));
  else out[t] = D(i, j);
}

}  // namespace

// out = X^+ W (nv x nv) on the tensor cores, any nv; herm: the result is known to be Hermitian
// (real data: only the tiles meeting the upper triangle run, the rest is mirrored)
template <typename S>
int gram_ozaki_wide(oefe_ctx* c, const S* X, int ldx, const S* W, int ldw, int64_t n, int nv, S* out, bool herm) {
  constexpr bool CPLX = sizeof(S) == sizeof(cd);
  const int NA = CPLX ? 2 * nv : nv;
  const int nI = (NA + 127) / 128, nJ = (NA + WN - 1) / WN;
  const bool upper = herm && !CPLX;
  int ntile = nI * nJ;
  if (upper) {
    ntile = 0;
    for (int I = 0; I < nI; ++I) ntile += std::max(0, nJ - 2 * I);
  }
  const long long passes = std::max<long long>(1, (n + 63) / 64);
  const int nbx = (int)std::max<long long>(1, std::min<long long>(passes, c->num_sms / std::max(1, ntile)));
  const long long ppc = (passes + nbx - 1) / nbx;
  const size_t need = (size_t)nbx * nI * nJ * 128 * WN * sizeof(double);
  OEFE_TRY(grow_ozpart(c, need));
  WGramArgs A;
  A.X = X;
  A.ldx = ldx;
  A.W = W;
  A.ldw = ldw;
  A.n = n;
  A.nv = nv;
  A.cplx = CPLX;
  A.nI = nI;
  A.nJ = nJ;
  A.upper = upper;
  A.passes = passes;
  A.ppc = ppc;
  A.part = (double*)c->d_ozpart;
  A.err = c->d_status + 2;
  OEFE_CUDA_TRY(c, cudaFuncSetAttribute(k_gram_wide, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)WSMEM));
  dim3 grid(nbx, ntile);
  OEFE_COUNTED k_gram_wide<<<grid, WT, WSMEM, c->stream>>>(A);
  OEFE_COUNTED k_gram_wide_reduce<S><<<(nv * nv + 255) / 256, 256, 0, c->stream>>>(A.part, nbx, nI, nJ, nv, upper, out);
  return oz_finish(c, "gram");
}

template int gram_ozaki_wide<double>(oefe_ctx*, const double*, int, const double*, int, int64_t, int, double*, bool);
template int gram_ozaki_wide<cd>(oefe_ctx*, const cd*, int, const cd*, int, int64_t, int, cd*, bool);
