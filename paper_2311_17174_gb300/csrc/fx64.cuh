// fx64.cuh -- 64-bit fixed-point arithmetic on the integer pipe, for the inner
// loops of the FP64 mode.
//
// An FP64 instruction of this GPU occupies an SM sub-partition for 76 cycles
// (measured, DFMA, one warp), a 32 x 32 + 64 -> 64 bit integer multiply-add
// for 4 and the two pipes run side by side.  A value in "Qk" is the signed
// 64-bit integer round(x 2^k).  A product of two 64-bit values keeps the terms
// high*high and high*low + low*high of the 32-bit halves (low*low is below
// the last kept bit): three multiply-adds, and one more to put them together.
// With 57 to 62 fraction bits each step rounds at least as finely as the
// double it replaces (2^-53 of a value near one).
#pragma once
#include <stdint.h>

namespace emri {
namespace fx {

typedef long long i64;
typedef unsigned long long u64;

#define FX_HD __host__ __device__ __forceinline__

// a b + c (32 x 32 + 64 -> 64 bits).  Waveform kernel, 128 walkers x 2^21, n_max
// 20: 50.0 ms with the C expression, 32.8 ms with mad.wide, 30.8 ms with
// mul.wide and a C sum.
FX_HD i64 wide(int a, int b, i64 c) {
#ifdef __CUDA_ARCH__
  i64 r;
  asm("mul.wide.s32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r + c;
#else
  return (i64)a * (i64)b + c;
#endif
}
FX_HD u64 wideu(uint32_t a, uint32_t b, u64 c) { return (u64)a * (u64)b + c; }
FX_HD int hi(i64 v) { return (int)(v >> 32); }
FX_HD uint32_t lo(i64 v) { return (uint32_t)v; }
// the low half's top 31 (27) bits, non-negative as a signed operand
FX_HD int lo31(i64 v) { return (int)((uint32_t)v >> 1); }
FX_HD int lo27(i64 v) { return (int)((uint32_t)v >> 5); }
FX_HD int mulhi(int a, int b) { return (int)(((i64)a * (i64)b) >> 32); }

// 64-bit operand in the two parts a product takes
struct Op {
  int h, l;
};
FX_HD Op op(i64 v) { return Op{hi(v), lo31(v)}; }

// Sum of products: acc.h gathers high*high, acc.c the cross terms (2^33 below
// it, rounded to nearest by the start value).  get() = sum a b 2^-64: operands in Qx and Qy give
// Q(x + y - 64).  |cross sum| < 2^63 holds for up to two products of
// operands below 2^62.
struct Sum {
  i64 h, c;
  FX_HD Sum() : h(0), c((i64)1 << 31) {}
  FX_HD explicit Sum(i64 h0) : h(h0), c((i64)1 << 31) {}
  FX_HD void add(Op a, Op b) {
    h = wide(a.h, b.h, h);
    c = wide(a.h, b.l, c);
    c = wide(a.l, b.h, c);
  }
  FX_HD i64 get() const { return wide(hi(c), 2, h); }
};

FX_HD i64 mul(Op a, Op b) {
  Sum s;
  s.add(a, b);
  return s.get();
}

// Operand with a signed low half: value = h 2^32 + l, |l| <= 2^31.  One
// instruction more than op(), but no bit is dropped and low*low averages to
// zero and stays below 2^62.
FX_HD Op bal(i64 v) { return Op{(int)((v + 0x80000000LL) >> 32), (int)(uint32_t)v}; }
FX_HD i64 value(Op a) { return ((i64)a.h << 32) + a.l; }

// a f 2^-32 for 0 <= f < 2^31
FX_HD i64 mul31(i64 a, int f) {
  const u64 l = wideu(lo(a), (uint32_t)f, 0);
  return wide(hi(a), f, (i64)(l >> 32));
}

// cos(2 pi p), sin(2 pi p) in Q62 of a phase p in cycles (Q64, mod 1): p =
// k/1024 + d with |d| <= 2^-11, exp(2 pi i k/1024) from the table (Q62), and
//   sin(2 pi d) = d (2 pi - d^2 ((2 pi)^3/3! - d^2 (2 pi)^5/5!)),
//   cos(2 pi d) - 1 = -d^2 ((2 pi)^2/2! - d^2 (2 pi)^4/4!)
// (first omitted terms (2 pi d)^7/7! < 6e-22, (2 pi d)^6/6! < 2e-18).  About
// 26 multiply-adds and 35 other integer instructions, ~180 cycles a warp, for
// the 13 FP64 instructions (990 cycles) of the same steps in double.
constexpr int kTrigLen = 1024;

struct Trig {
  i64 c, s;
};

FX_HD Trig sincos_cycles(u64 p, const Trig* __restrict__ tab) {
  const uint32_t ph = (uint32_t)(p >> 32);
  const uint32_t k = (ph + (1u << 21)) >> 22;
  const i64 D = (i64)((p - ((u64)k << 54)) << 9);        // d in Q73
  const Op d = op(D);
  const i64 E = wide(hi(wide(d.h, d.l, 0)), 4, wide(d.h, d.h, 0));   // d^2 in Q82
  const Op e = op(E);
  // 2 pi in Q60
  const i64 P0 = 0x6487ED5110B4611ALL;
  const int k3 = 693598668 - mulhi(e.h, 5223);           // (2 pi)^3/6 = 41.3417022404 in Q24
  const i64 P = P0 - (wide(e.h, k3, 0) >> 14);
  const Op sx = op(mul(d, op(P)));                       // sin(2 pi d) in Q69
  // (2 pi)^2/2 = 19.7392088021787172 in Q51, (2 pi)^4/24 = 64.9393940227 in Q21
  const i64 K = 44448746703040243LL - (wide(e.h, 136187780, 0) >> 20);
  const Op cx = op(-mul(e, op(K)));                      // cos(2 pi d) - 1 in Q69
  const Trig t = tab[k & (kTrigLen - 1)];
  const Op tc = op(t.c), ts = op(t.s);
  Sum c, s;                                              // Q67
  c.add(tc, cx);
  s.add(ts, cx);
  s.add(tc, sx);
  Sum c2;
  c2.add(ts, sx);
  return Trig{t.c + ((c.get() - c2.get()) >> 5), t.s + (s.get() >> 5)};
}

}  // namespace fx
}  // namespace emri
