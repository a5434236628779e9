// Two double-floats at a time on the packed FP32 instructions (add / mul / fma .rn.f32x2): the
// two values (rows or columns) side by side.  Every operation rounds like its scalar form in common.cuh,
// so results are the same bits; one instruction slot serves both (the FP32 pipes give the
// packed form no more flops, but half the issue slots, and kernels with few warps are bound by
// issue and latency).
#pragma once

#include "common.cuh"

namespace ql {

// One stored element and its biased double exponent (0 for zeros and subnormals); FP32 subnormals
// keep their value, unlike in ArithDF::load, whose sums of squares could not hold them.
QL_DEV df load_df(double x, int& E) { return df_split_double(x, E); }
QL_DEV df load_df(float x, int& E) {
  const int e = (__float_as_int(x) >> 23) & 0xff;
  E = e == 0 ? 0 : e + 896;
  return df{x, 0.0f};
}

using f2 = unsigned long long;  // two floats, the first in the low word
struct df2 {
  f2 hi, lo;
};

QL_DEV f2 f2_make(float a, float b) {
  f2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
QL_DEV void f2_split(f2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
QL_DEV f2 f2_add(f2 a, f2 b) {
  f2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
QL_DEV f2 f2_mul(f2 a, f2 b) {
  f2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
QL_DEV f2 f2_fma(f2 a, f2 b, f2 c) {
  f2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
constexpr f2 kF2MinusOne = 0xbf800000bf800000ull;
QL_DEV f2 f2_sub(f2 a, f2 b) { return f2_fma(b, kF2MinusOne, a); }  // a - b, rounded once
QL_DEV f2 f2_neg(f2 a) { return a ^ 0x8000000080000000ull; }

// A factor with its negatives: the error terms of a product are formed with them (as -e), so
// that no other sign flips are needed.
struct df2n {
  f2 hi, lo, nhi, nlo;
};
QL_DEV df2n df2_factor(df2 a) { return df2n{a.hi, a.lo, f2_neg(a.hi), f2_neg(a.lo)}; }

// acc += a b (as ArithDF::acc_fma in each half).
QL_DEV void df2_acc_fma(df2& acc, const df2n& a, const df2& b) {
  const f2 p = f2_mul(a.hi, b.hi);
  f2 ne = f2_fma(a.nhi, b.hi, p);  // -(a.hi b.hi - p)
  ne = f2_fma(a.nlo, b.lo, ne);
  ne = f2_fma(a.nhi, b.lo, ne);
  ne = f2_fma(a.nlo, b.hi, ne);
  const f2 s = f2_add(acc.hi, p);
  const f2 bb = f2_sub(s, acc.hi);
  const f2 t = f2_add(f2_sub(acc.hi, f2_sub(s, bb)), f2_sub(p, bb));
  acc.hi = s;
  acc.lo = f2_add(acc.lo, f2_sub(t, ne));
}
// The two halves of a finished accumulator.
QL_DEV void df2_rows(const df2& a, df& r0, df& r1) {
  float h0, h1, l0, l1;
  f2_split(a.hi, h0, h1);
  f2_split(a.lo, l0, l1);
  r0 = df_make(h0, l0);
  r1 = df_make(h1, l1);
}

}  // namespace ql
