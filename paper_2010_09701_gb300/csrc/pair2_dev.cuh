// Two FP32 pairs (pair_dev.cuh) side by side in packed FP32 instructions (fma.rn.f32x2 and its
// kin): the same operations in the same order on both, with half the issue slots of the scalar
// form. The FP32 pipe's own rate is the same; what the packing frees are the slots that shared-memory
// loads and addresses need: a register-tiled 1D contraction ran at 2.85 T pair multiply-adds a
// second against 2.31 T in scalar form (85% and 69% of the pipe's 3.36 T).
#pragma once
#include <cstdint>

#include "pair_int_dev.cuh"

namespace {

typedef unsigned long long pk;   // two FP32 values

__device__ __forceinline__ pk pk_fma(pk a, pk b, pk c) {
  pk d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ pk pk_add(pk a, pk b) {
  pk d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ pk pk_mul(pk a, pk b) {
  pk d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ pk pk_make(float lo, float hi) {
  pk d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ void pk_split(pk a, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(a)); }
__device__ __forceinline__ pk pk_neg(pk a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ pk pk_minus1() { return 0xBF800000BF800000ull; }
// a - b, exactly rounded like a subtraction
__device__ __forceinline__ pk pk_sub(pk a, pk b) { return pk_fma(b, pk_minus1(), a); }

struct alignas(16) p2 {   // two pairs: high parts, low parts
  pk h, l;
};

// s += t x: f2_mac on both halves
__device__ __forceinline__ void p2_mac(p2& s, p2 t, p2 x) {
  const pk np = pk_mul(pk_neg(t.h), x.h);              // -(t.h x.h), rounded
  pk e = pk_fma(t.h, x.h, np);                         // exact remainder
  e = pk_fma(t.h, x.l, e);
  e = pk_fma(t.l, x.h, e);
  const pk r = pk_sub(s.h, np);                        // two-sum of s.h and -np
  const pk bp = pk_sub(r, s.h);
  const pk er = pk_sub(pk_sub(s.h, pk_sub(r, bp)), pk_add(np, bp));
  s.h = r;
  s.l = pk_add(s.l, pk_add(er, e));
}
__device__ __forceinline__ p2 p2_fin(p2 s) {
  const pk h = pk_add(s.h, s.l);
  return p2{h, pk_sub(s.l, pk_sub(h, s.h))};
}
// f2_add on both halves
__device__ __forceinline__ p2 p2_add(p2 a, p2 b) {
  const pk t = pk_add(a.h, b.h);
  const pk bp = pk_sub(t, a.h);
  const pk er = pk_add(pk_sub(a.h, pk_sub(t, bp)), pk_sub(b.h, bp));
  return p2_fin(p2{t, pk_add(er, pk_add(a.l, b.l))});
}
__device__ __forceinline__ p2 p2_mul(p2 a, p2 b) {
  const pk np = pk_mul(pk_neg(a.h), b.h);
  pk e = pk_fma(a.h, b.h, np);
  e = pk_fma(a.h, b.l, e);
  e = pk_fma(a.l, b.h, e);
  return p2_fin(p2{pk_neg(np), e});
}
__device__ __forceinline__ p2 p2_zero() { return p2{0ull, 0ull}; }
__device__ __forceinline__ p2 p2_dup(f2 a) { return p2{pk_make(a.h, a.h), pk_make(a.l, a.l)}; }
__device__ __forceinline__ p2 p2_join(f2 a, f2 b) { return p2{pk_make(a.h, b.h), pk_make(a.l, b.l)}; }
__device__ __forceinline__ void p2_halves(p2 x, f2& a, f2& b) {
  pk_split(x.h, a.h, b.h);
  pk_split(x.l, a.l, b.l);
}
// i x for x = (real, imaginary part): (-imaginary, real)
__device__ __forceinline__ p2 p2_times_i(p2 x) {
  f2 a, b;
  p2_halves(x, a, b);
  return p2_join(f2_neg(b), a);
}

}  // namespace
