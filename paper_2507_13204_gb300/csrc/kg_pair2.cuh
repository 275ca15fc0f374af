// Float-pair arithmetic on two values at once: GB300's packed FP32 instructions
// (add, sub, mul, fma on .f32x2, an aligned register pair).
//
// They run at the lane rate of the scalar ones (measured 37 against 36 T lane
// operations a second for 8 independent chains a thread) but take one issue slot
// for two results, and a scalar pair FMA does not reach that rate: eight chains
// of acc_fma run at 25.3 T, of acc2_fma at 34.1 T lane operations a second, and
// the other instructions of a loop find the slots that are left.  Every operation
// rounds each half as the scalar one does, so acc2_* give the bits of two acc_*.
//
// Prepared copies hold the pairs of two neighbouring entries as (h0, h1, l0, l1),
// 16 bytes: one 128-bit load gives the packed operands.
#pragma once

#include "kg_pair.cuh"

namespace kg {

struct F2 {
  unsigned long long v;
};

__device__ __forceinline__ F2 f2(float x, float y) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ F2 f2_dup(float x) { return f2(x, x); }
__device__ __forceinline__ float2 f2_get(F2 a) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(a.v));
  return r;
}
__device__ __forceinline__ F2 f2_zero() { return F2{0ull}; }
__device__ __forceinline__ F2 f2_neg(F2 a) {
  const float2 q = f2_get(a);
  return f2(-q.x, -q.y);
}
__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f2_sub(F2 a, F2 b) {
  F2 r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
  return r;
}
__device__ __forceinline__ F2 f2_fma(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
  return r;
}

// Two accumulators / two pairs.
struct Acc2 {
  F2 s, l;
};
struct Pair2 {
  F2 h, l;
};

__device__ __forceinline__ Acc2 acc2_zero() { return Acc2{f2_zero(), f2_zero()}; }

// The entry pair (h0, h1, l0, l1) at p (16-byte aligned).
__device__ __forceinline__ Pair2 pair2_load(const float4* p) {
  const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(p);
  return Pair2{F2{q.x}, F2{q.y}};
}
__device__ __forceinline__ float4 pair2_entry(Pair a, Pair b) { return make_float4(a.h, b.h, a.l, b.l); }
__device__ __forceinline__ Pair2 pair2_of(Pair a, Pair b) { return Pair2{f2(a.h, b.h), f2(a.l, b.l)}; }
__device__ __forceinline__ Pair2 pair2_dup(Pair a) { return Pair2{f2_dup(a.h), f2_dup(a.l)}; }

__device__ __forceinline__ void two_sum2(F2 a, F2 b, F2& s, F2& e) {
  s = f2_add(a, b);
  const F2 bb = f2_sub(s, a);
  e = f2_add(f2_sub(a, f2_sub(s, bb)), f2_sub(b, bb));
}

// c += a * b, as acc_fma on each half.
__device__ __forceinline__ void acc2_fma(Acc2& c, Pair2 a, Pair2 b) {
  const F2 p = f2_mul(a.h, b.h);
  F2 e = f2_fma(a.h, b.h, f2_neg(p));
  e = f2_fma(a.h, b.l, e);
  e = f2_fma(a.l, b.h, e);
  F2 s, r;
  two_sum2(c.s, p, s, r);
  c.s = s;
  c.l = f2_add(c.l, f2_add(r, e));
}

// acc_prod on each half.
__device__ __forceinline__ Acc2 acc2_prod(Pair2 a, Pair2 b) {
  const F2 p = f2_mul(a.h, b.h);
  F2 e = f2_fma(a.h, b.h, f2_neg(p));
  e = f2_fma(a.h, b.l, e);
  e = f2_fma(a.l, b.h, e);
  return Acc2{p, e};
}

__device__ __forceinline__ void acc2_renorm(Acc2& c) {
  F2 s, e;
  two_sum2(c.s, c.l, s, e);
  c.s = s;
  c.l = e;
}

// The two accumulators by themselves, and their sum.
__device__ __forceinline__ Acc acc2_x(Acc2 a) { return Acc{f2_get(a.s).x, f2_get(a.l).x}; }
__device__ __forceinline__ Acc acc2_y(Acc2 a) { return Acc{f2_get(a.s).y, f2_get(a.l).y}; }
__device__ __forceinline__ Acc acc2_sum(Acc2 a) { return acc_add(acc2_x(a), acc2_y(a)); }

// acc_pair on each half.
__device__ __forceinline__ Pair2 acc2_pair(Acc2 a) {
  Pair2 p;
  two_sum2(a.s, a.l, p.h, p.l);
  return p;
}

// pair_mul on each half.
__device__ __forceinline__ Pair2 pair2_mul(Pair2 a, Pair2 b) {
  const F2 p = f2_mul(a.h, b.h);
  F2 e = f2_fma(a.h, b.h, f2_neg(p));
  e = f2_fma(a.h, b.l, e);
  e = f2_fma(a.l, b.h, e);
  const F2 s = f2_add(p, e);
  return Pair2{s, f2_sub(e, f2_sub(s, p))};
}

__device__ __forceinline__ Pair pair2_x(Pair2 a) { return Pair{f2_get(a.h).x, f2_get(a.l).x}; }
__device__ __forceinline__ Pair pair2_y(Pair2 a) { return Pair{f2_get(a.h).y, f2_get(a.l).y}; }

}  // namespace kg
