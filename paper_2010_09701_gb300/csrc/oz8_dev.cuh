// Exact fixed-point products of FP64 operands on the tensor cores (the Ozaki scheme with bf16 digits):
// shared by the Gram matrices and rotations of wide blocks (oz8_wide.cu) and the enrichment part of the fields
// (fields_pair.cu).
//
// A value is cut into 8 balanced digits of 7 bits (each in [-64, 64), exact in bf16) under one exponent
// per operand row: 54 bits of the row's largest value, more than an FP64 significand (a value 2^-k of that
// largest one keeps 54 - k bits: the error is relative to the operand rows' maxima). The 36 digit
// products of levels s + t <= 7 accumulate exactly in FP32 (products at most 2^12, 8 pairs a level, so
// 512 entries of K stay below 2^24), the levels combine in integers and round once to FP64. Balanced
// digits (against 7 unsigned ones, products up to 2^14) are what lets 512 entries of K, not 64, go by
// between two combinations of the levels, each of which costs as much as 150 entries' products.
#pragma once
#include <cuda_bf16.h>

#include <cstdint>

#include "tcgen05_dev.cuh"

namespace {

constexpr int ZS = 8;                   // digits per value
constexpr int ZK = 64;                  // K entries per operand row in shared memory (128 bytes)
constexpr int ZN = 64;                  // operand columns (B rows)
constexpr int ZPA = 128 * 128;          // bytes of an A plane (128 rows x 64 bf16)
constexpr int ZPB = ZN * 128;           // bytes of a B plane
constexpr int ZMAXK = 512;              // K entries accumulated before the levels are combined
constexpr int ZCOLS = 512;              // tensor-memory columns: 8 levels x 64
static_assert((long long)ZS * ZMAXK * (1LL << 12) <= (1LL << 24), "level sums must be exact in FP32");

__device__ __forceinline__ int bexp_of(double v) { return (int)((__double_as_longlong(v) >> 52) & 0x7FF); }

// trunc(|x| 2^(54-E)) with the sign of x, plus 64 in every base-128 position, where the largest
// biased exponent of the row is bm (|x| < 2^E, E = bm - 1022); zeros and subnormals count as zero.
// 54 bits: with 55 a value just below 2^E would carry out of the top digit.
__device__ __forceinline__ unsigned long long fixed54(double x, int bm) {
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

// two levels in one integer (at most 2^31: lev_d <= (d + 1) 2^21)
__device__ __forceinline__ int two_levels(float a, float b) { return __float2int_rn(a) * 128 + __float2int_rn(b); }

// the sum of the levels of one entry from its four integers (levels 01, 23, 45, 67), rounded to units of
// 2^(E + F - 51), as a double; bsum: the two biased exponents' sum. An exponent of 2047 (an infinity
// or NaN in the operand row) gives NaN.
__device__ __forceinline__ double from_levels(int l01, int l23, int l45, int l67, int bE, int bF) {
  const long long hi = (long long)l01 * 16384 + l23, lo = (long long)l45 * 16384 + l67;
  const long long V = hi * (1ll << 20) + ((lo + 128) >> 8);         // |V| < 2^63
  if (bE == 0x7FF || bF == 0x7FF) return __longlong_as_double(0x7FF8000000000000ll);
  if (V == 0) return 0.0;
  const unsigned long long mag = V < 0 ? 0ull - (unsigned long long)V : (unsigned long long)V;
  const int lz = __clzll((long long)mag);
  const unsigned long long nrm = mag << lz;
  const unsigned long long r = (nrm >> 11) + ((nrm >> 10) & 1);     // 53 bits, rounded
  const int f = bE + bF - 2044 + 1035 - lz;                         // exponent field of r 2^(E + F - 40 - lz)
  double x;
  if (f >= 1 && f <= 2045) x = __longlong_as_double((long long)(((unsigned long long)f << 52) + (r - (1ull << 52))));
  else x = ldexp((double)r, f - 1075);
  return V < 0 ? -x : x;
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

// the combined levels of 8 columns
__device__ __forceinline__ void drain8(uint32_t taddr, int bE, const int* bF, double* x) {
  float v[4][8];
  int a[8], b[8];
  tmem_ld_levels(taddr, v);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    a[j] = two_levels(v[0][j], v[1][j]);
    b[j] = two_levels(v[2][j], v[3][j]);
  }
  tmem_ld_levels(taddr + 4 * ZN, v);
#pragma unroll
  for (int j = 0; j < 8; ++j) x[j] = from_levels(a[j], b[j], two_levels(v[0][j], v[1][j]), two_levels(v[2][j], v[3][j]), bE, bF[j]);
}

// The combined levels of 8 columns as FP32 pairs: levels 4 to 7 by FP32 Horner steps (they weigh 2^-28 and
// less), levels 0 to 3 by two-sums, scaled by 2^(E + F - 10). On the FP32 pipe, against the integer pipe of
// drain8, which the cutting of digits already fills; about 2^-48 of the result and of the largest product.
__device__ __forceinline__ void drain8_pairs(uint32_t taddr, int bE, const int* bF, float* h, float* l) {
  float v[4][8], lo[8];
  tmem_ld_levels(taddr + 4 * ZN, v);
#pragma unroll
  for (int j = 0; j < 8; ++j)
    lo[j] = __fmaf_rn(__fmaf_rn(__fmaf_rn(v[3][j], 0.0078125f, v[2][j]), 0.0078125f, v[1][j]), 0.0078125f, v[0][j]);
  tmem_ld_levels(taddr, v);
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    float a = v[0][j], b = 0.0f;
    const float w[4] = {__fmul_rn(v[1][j], 0.0078125f), __fmul_rn(v[2][j], 6.103515625e-05f),
                        __fmul_rn(v[3][j], 4.76837158203125e-07f), __fmul_rn(lo[j], 3.7252902984619141e-09f)};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float t = __fadd_rn(a, w[i]), bp = __fsub_rn(t, a);
      b = __fadd_rn(b, __fadd_rn(__fsub_rn(a, __fsub_rn(t, bp)), __fsub_rn(w[i], bp)));
      a = t;
    }
    const float s = __fadd_rn(a, b), r = __fsub_rn(b, __fsub_rn(s, a));
    const int sc = bE + bF[j] - 2044 - 10;
    if (bE == 0x7FF || bF[j] == 0x7FF) {
      h[j] = l[j] = __int_as_float(0x7FC00000);
    } else if (sc > -127 && sc < 128) {
      const float f = __int_as_float((sc + 127) << 23);
      h[j] = __fmul_rn(s, f);
      l[j] = __fmul_rn(r, f);
    } else {
      h[j] = ldexpf(s, sc);
      l[j] = ldexpf(r, sc);
    }
  }
}

__device__ __forceinline__ void oz_tmem_alloc(uint32_t* slot) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(ZCOLS) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void oz_tmem_free(uint32_t taddr) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ZCOLS) : "memory");
}

constexpr size_t OZ_SMEM = 1024 + (size_t)ZS * (ZPA + ZPB);   // operand planes, 1024-byte aligned

// the two halves of the operand planes: MMAs in flight on each
struct Halves {
  uint64_t* bar;
  uint32_t phase[2] = {0, 0};
  bool out[2] = {false, false};
  __device__ __forceinline__ bool wait(int h, volatile int* fail) {
    if (!out[h]) return true;
    const bool ok = mbar_wait(&bar[h], phase[h], fail);
    if (ok) {
      phase[h] ^= 1;
      out[h] = false;
    }
    return ok;
  }
};

// warp 0 (every lane): the digit products of half h
__device__ __forceinline__ void issue_half(uint32_t taddr, const unsigned char* sA, const unsigned char* sB, int h,
                                           bool fresh, uint64_t* bar, int nks = 2) {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t lead = elect_lane();
  issue_digit_levels<ZS, 2, ZPA, ZPB, ZN>(lead, taddr, smem_u32(sA) + 64 * h, smem_u32(sB) + 64 * h, idesc_bf16(128, ZN, false), nks,
                                          fresh);
  mma_commit_lead(lead, bar);
}

// prologue and epilogue shared by the two kernels
struct OzCta {
  unsigned char *sA, *sB;
  uint32_t taddr;
};
__device__ __forceinline__ OzCta oz_begin(unsigned char* raw, uint32_t* slot, uint64_t* bar, volatile int* fail) {
  OzCta c;
  c.sA = (unsigned char*)(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
  c.sB = c.sA + ZS * ZPA;
  if ((threadIdx.x >> 5) == 0) oz_tmem_alloc(slot);
  if (threadIdx.x == 0) {
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  c.taddr = *slot;
  return c;
}
__device__ __forceinline__ void oz_end(const OzCta& c, Halves& H, volatile int* fail, int* err) {
  if (threadIdx.x == 0 && *fail) {
    for (int h = 0; h < 2; ++h)
      if (H.out[h]) mbar_wait_drain(&H.bar[h], H.phase[h]);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (*fail && threadIdx.x == 0) atomicExch(err, 1);
  if ((threadIdx.x >> 5) == 0) oz_tmem_free(c.taddr);
}
}  // namespace
