// Double-float arithmetic (df64, hmc_internal.cuh) on two values at a time
// with the paired-FP32 instructions of this architecture (add, sub, mul, fma
// .f32x2): the operations of the scalar form, lane by lane, at half the
// instruction issues.  The paired instructions run at the rate of two scalar
// ones, so the FP32 pipe bounds both forms alike; the scalar kernels stopped
// at 50-55 % of it with the issue slots 55-62 % busy.
//
// A product needs its negated high part twice; mul and fma take it from the
// negated high part of one factor (nbh), which the callers keep for factors
// used several times.
#pragma once
#include "hmc_internal.cuh"

namespace hmc {

typedef unsigned long long f32x2;

__device__ __forceinline__ f32x2 pk2(float a, float b) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ float lane0(f32x2 v) { return __uint_as_float((unsigned)v); }
__device__ __forceinline__ float lane1(f32x2 v) { return __uint_as_float((unsigned)(v >> 32)); }
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 sub2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 mul2(f32x2 a, f32x2 b) {
  f32x2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
// sign masks of the two lanes
constexpr f32x2 kNeg0 = 0x0000000080000000ull, kNeg1 = 0x8000000000000000ull;
constexpr f32x2 kNegBoth = kNeg0 | kNeg1;

// two double-floats
struct dd2 {
  f32x2 h, l;
};
__device__ __forceinline__ dd2 pack(df64 a, df64 b) { return {pk2(a.hi, b.hi), pk2(a.lo, b.lo)}; }
__device__ __forceinline__ df64 first(dd2 v) { return {lane0(v.h), lane0(v.l)}; }
__device__ __forceinline__ df64 second(dd2 v) { return {lane1(v.h), lane1(v.l)}; }
__device__ __forceinline__ dd2 flip2(dd2 v, f32x2 mask) { return {v.h ^ mask, v.l ^ mask}; }
__device__ __forceinline__ dd2 swap2(dd2 v) {
  return {pk2(lane1(v.h), lane0(v.h)), pk2(lane1(v.l), lane0(v.l))};
}
// requires |a| >= |b| per lane
__device__ __forceinline__ dd2 quick2(f32x2 a, f32x2 b) {
  const f32x2 s = add2(a, b);
  return {s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ dd2 add(dd2 a, dd2 b) {
  const f32x2 s = add2(a.h, b.h), bb = sub2(s, a.h);
  const f32x2 e = add2(sub2(a.h, sub2(s, bb)), sub2(b.h, bb));
  return quick2(s, add2(e, add2(a.l, b.l)));
}
// a b;  nbh = -b.h
__device__ __forceinline__ dd2 mul(dd2 a, dd2 b, f32x2 nbh) {
  const f32x2 pn = mul2(a.h, nbh);
  f32x2 e = fma2(a.h, b.h, pn);
  e = fma2(a.h, b.l, e);
  e = fma2(a.l, b.h, e);
  return quick2(pn ^ kNegBoth, e);
}
// a b + c;  nbh = -b.h
__device__ __forceinline__ dd2 fma(dd2 a, dd2 b, f32x2 nbh, dd2 c) {
  const f32x2 pn = mul2(a.h, nbh);  // -p
  f32x2 e = fma2(a.h, b.h, pn);
  e = fma2(a.h, b.l, e);
  e = fma2(a.l, b.h, e);
  // two-sum of p and c.h
  const f32x2 s = sub2(c.h, pn), bb = add2(s, pn);
  const f32x2 q = add2(pn, sub2(s, bb));  // -(p - (s - bb))
  const f32x2 t = sub2(sub2(c.h, bb), q);
  return quick2(s, add2(t, add2(e, c.l)));
}

// a complex factor used on the right of several products: value, negated
// value
struct cdd2 {
  dd2 re, im;
};
struct cneg2 {
  dd2 re, im;
};
__device__ __forceinline__ cneg2 negated(const cdd2 &v) {
  return {flip2(v.re, kNegBoth), flip2(v.im, kNegBoth)};
}
// u v
__device__ __forceinline__ cdd2 cmul(const cdd2 &u, const cdd2 &v, const cneg2 &n) {
  return {fma(u.re, v.re, n.re.h, mul(u.im, dd2{n.im.h, n.im.l}, v.im.h)),
          fma(u.re, v.im, n.im.h, mul(u.im, v.re, n.re.h))};
}
// acc + u v
__device__ __forceinline__ cdd2 cmac(cdd2 acc, const cdd2 &u, const cdd2 &v, const cneg2 &n) {
  acc.re = fma(u.re, v.re, n.re.h, acc.re);
  acc.re = fma(u.im, dd2{n.im.h, n.im.l}, v.im.h, acc.re);
  acc.im = fma(u.re, v.im, n.im.h, acc.im);
  acc.im = fma(u.im, v.re, n.re.h, acc.im);
  return acc;
}

// ---- asynchronous copies into a thread's own slots of shared memory -------------------
__device__ __forceinline__ void cp_async16(void *smem, const void *g) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(s), "l"(g) : "memory");
}
// the same through L1 (data that other warps of the block read too)
__device__ __forceinline__ void cp_async16_l1(void *smem, const void *g) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"(s), "l"(g) : "memory");
}
// all copies this thread has issued are in its shared memory
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
}

}  // namespace hmc
