// wave_fixed.cuh -- harmonic sums and response of one sample in 64-bit fixed
// point (fx64.cuh): the FP64 waveform kernel's inner loop (k_wave.cu), callable
// on the host as well.
#pragma once
#include <cuda_runtime.h>
#include <math.h>
#include <string.h>
#include "fx64.cuh"

namespace emri {

// Harmonic coefficients of a segment in fixed point: the quadratics
// q0 + rho (q1 + rho q2) of a_n, b_n, c_n in rho = r/1024 (r: sample offset),
// each times 2^k split as 2^27 h + l (0 <= l < 2^27), or q2 in h alone; signed
// for the recurrence of harmonics_fixed.
struct __align__(16) HarmX {
  int4 a, b, c;   // (h0, l0, h1, l1)
  int h2[4], l2[4];
};

// Block exponents of the coefficients and the shifts that align the sums.
// S0, S1, S2: sums over harmonics and quantities of |q0|, |q1|, |q2|.  Every
// accumulator of harmonics_fixed stays below 2^63: sum |q0| 2^k0 < 2^56,
// sum |q1| 2^k1 < 2^50, sum |q2| 2^k2 < 2^31 (one word, and products with the
// 30-bit cosines below 2^61) or 2^51.  One word rounds each coefficient by half
// a unit, a sum over 32 harmonics by 2^-30 S2 (rms): taken where S2 is below
// 2^-23 S0, as it is on all of an inspiral but its last hours.  With the rest the
// sums are then within 2.5e-16 of S0 (rms 0.5e-16; n <= 32, e <= 0.9), and in
// either form closer than the same sums in double.
struct HarmScale {
  int k0, k1, k2, sh1, sh2, two;
};
FX_HD HarmScale harm_scale(float S0, float S1, float S2) {
  S0 = fmaxf(S0, 1e-20f);
  S1 = fmaxf(fmaxf(S1, S2), S0 * 0x1p-24f);
  S2 = fmaxf(S2, S1 * 0x1p-24f);
  S0 = fmaxf(S0, 128.f * S1);
  HarmScale o;
  const int e0 = ilogbf(S0), e1 = ilogbf(S1), e2 = ilogbf(S2);
  o.k0 = 55 - e0;
  o.k1 = 49 - e1;
  o.two = S2 > S0 * 0x1p-23f;
  o.k2 = (o.two ? 50 : 30) - e2;
  o.sh1 = o.k1 - o.k0 - 1;                      // in [0, 18]
  o.sh2 = o.k2 - o.k1 + (o.two ? -1 : 23);      // in [0, 29]
  return o;
}

// exact 2^k as a double, |k| < 1000
FX_HD double pow2d(int k) {
  const fx::i64 b = (fx::i64)(k + 1023) << 52;
#ifdef __CUDA_ARCH__
  return __longlong_as_double(b);
#else
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}

// Coefficient p of quantity f (a, b, c) of harmonic index m: v, of (r/span)^p
FX_HD void harm_put(HarmX& o, int m, int f, int p, double v, const HarmScale& hs, int span) {
  if ((m + 1) & 2) v = -v;   // the signs of the recurrence
  v *= pow2d(p == 0 ? hs.k0 : p == 1 ? hs.k1 : hs.k2);
  if (span != 1024) {        // to rho = r / 1024
    const double rs = 1024.0 / (double)span;
    v *= p == 0 ? 1.0 : p == 1 ? rs : rs * rs;
  }
  const fx::i64 q = llrint(v);
  int* oh = p < 2 ? reinterpret_cast<int*>(&o) + 4 * f + 2 * p : o.h2 + f;
  int* ol = p < 2 ? oh + 1 : o.l2 + f;
  const bool one = p == 2 && !hs.two;
  *oh = (int)(one ? q : q >> 27);
  *ol = one ? 0 : (int)(q & ((1 << 27) - 1));
}

// C = sum_n a_n cos(n Phi), S = sum_n b_n sin(n Phi), R = sum_n c_n cos(n Phi)
// in units of 2^-(6 + k0) at sample offset r of the segment; cs: cos, sin of
// Phi in Q62.
//
// d_n = +-cos(n Phi) follows d_{n+1} = -+ T d_n + d_{n-1}, T = 2 cos Phi (the
// minus for odd n; signs + + - - over n mod 4, which the coefficients carry),
// in Q59 -- the previous value is then the addend of the first multiply-add
// and the product needs no shift.  Rounding per step ~2^-59, against ~2^-54 in
// double.  Per harmonic 8 multiply-adds advance cosine and sine, 9 add the
// constant, 9 the linear and 3 the quadratic coefficients (which are ~2^-9 and
// ~2^-20 of the constant ones, so q2 mostly keeps one word, else kTwo): 29
// multiply-adds and ~12 others, ~150 cycles a warp, for 11 FP64 instructions
// (836 cycles).
template <bool kTwo>
FX_HD void harmonics_fixed(fx::Trig cs, int r, const HarmX* __restrict__ hx, int n_max, int sh1,
                                                int sh2, fx::i64& C, fx::i64& S, fx::i64& R) {
  using namespace fx;
  const Op tp = op(cs.c), tm = op(-cs.c);   // 2 cos Phi and its negative, Q61
  i64 c0 = (i64)1 << 59, s0 = 0, c1 = cs.c >> 3, s1 = cs.s >> 3;
  i64 h0[3] = {0, 0, 0}, x0[3] = {0, 0, 0}, h1[3] = {0, 0, 0}, x1[3] = {0, 0, 0}, h2[3] = {0, 0, 0},
      x2[3] = {0, 0, 0};
  auto acc = [&](int q, int4 k, int kh, int kl, int vh, int vl) {
    h0[q] = wide(k.x, vh, h0[q]);
    x0[q] = wide(k.x, vl, x0[q]);
    x0[q] = wide(k.y, vh, x0[q]);
    h1[q] = wide(k.z, vh, h1[q]);
    x1[q] = wide(k.z, vl, x1[q]);
    x1[q] = wide(k.w, vh, x1[q]);
    h2[q] = wide(kh, vh, h2[q]);
    if (kTwo) {
      x2[q] = wide(kh, vl, x2[q]);
      x2[q] = wide(kl, vh, x2[q]);
    }
  };
  // one harmonic: adds it to the sums; (p0, p1) -> the next value in p0
  auto step = [&](const HarmX& k, Op T, i64& cp, i64 cn, i64& sp, i64 sn) {
    const i64 cv = cn << 3, sv = sn << 3;   // Q62
    const int ch = hi(cv), sh = hi(sv);
    acc(0, k.a, k.h2[0], k.l2[0], ch, lo27(cv));
    acc(1, k.b, k.h2[1], k.l2[1], sh, lo27(sv));
    acc(2, k.c, k.h2[2], k.l2[2], ch, lo27(cv));
    Sum nc(cp), ns(sp);
    nc.add(T, Op{ch, lo31(cv)});
    ns.add(T, Op{sh, lo31(sv)});
    cp = nc.get();
    sp = ns.get();
  };
  int n = 0;
#pragma unroll 1
  for (; n + 1 < n_max; n += 2) {
    step(hx[n], tm, c0, c1, s0, s1);
    step(hx[n + 1], tp, c1, c0, s1, s0);
  }
  if (n < n_max) step(hx[n], tm, c0, c1, s0, s1);
  const int rho = r << 21;   // 2^31 r / 1024
  i64 v[3];
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    const i64 w2 = kTwo ? (h2[q] << 3) + (x2[q] >> 24) : h2[q];
    const i64 w1 = (h1[q] << 3) + (x1[q] >> 24) + (mul31(w2, rho) >> sh2);
    v[q] = (h0[q] << 3) + (x0[q] >> 24) + (mul31(w1, rho) >> sh1);
  }
  C = v[0];
  S = v[1];
  R = v[2];
}

// Geometry constants of the response, Q62 (spS, sqS: Q60)
struct GeoX {
  fx::Op pe1, pe2n, qe1, qe2n, cpe1, cpe2, cqe1, cqe2;
  fx::i64 spSn, sqSn;
};

// response() in fixed point: H+ and Hx in units of 2^-(2 + k0) from the sums
// in units of 2^-(6 + k0).  |z_1|, |z_2| <= 1 (projections of unit vectors).
FX_HD void response_fixed(const GeoX& g, fx::Trig gm, fx::Trig al, fx::i64 Cs, fx::i64 Ss,
                                               fx::i64 Rs, fx::i64& Hp, fx::i64& Hx) {
  using namespace fx;
  const Op ca = op(al.c), sa = op(al.s);
  auto proj = [&](Op x, Op kx, Op y, Op ky, i64 add) {   // Q60 sums, returned in Q62
    Sum s(add);
    s.add(x, kx);
    s.add(y, ky);
    return s.get() << 2;
  };
  const i64 z1r = proj(sa, g.pe1, ca, g.pe2n, 0), z1i = proj(sa, g.qe1, ca, g.qe2n, 0);
  const i64 z2r = proj(ca, g.cpe1, sa, g.cpe2, g.spSn), z2i = proj(ca, g.cqe1, sa, g.cqe2, g.sqSn);
  i64 a, b, y;   // A = 1: (Rs + X)/4, (Rs - X)/4, 2 Y/4
  {
    const Op c = op(Cs), s = op(Ss), g2c = op(gm.c);
    Sum X, Y;
    X.add(c, g2c);
    X.add(s, op(-gm.s));
    Y.add(c, op(gm.s));
    Y.add(s, g2c);
    const i64 x = X.get();
    a = (Rs >> 2) + x;
    b = (Rs >> 2) - x;
    y = Y.get() << 1;
  }
  const Op z1ro = op(z1r), z1io = op(z1i), z2ro = op(z2r), z2io = op(z2i), ao = op(a), bo = op(b), yo = op(y);
  Sum p, q, c;
  p.add(ao, op(mul(op(z1r - z1i), op(z1r + z1i)) << 2));
  p.add(bo, op(mul(op(z2r - z2i), op(z2r + z2i)) << 2));
  q.add(yo, op((mul(z1ro, z2ro) - mul(z1io, z2io)) << 2));
  Hp = p.get() + q.get();
  c.add(z1ro, z2io);
  c.add(z1io, z2ro);
  Sum u, w;
  u.add(ao, op(mul(z1ro, z1io) << 3));
  u.add(bo, op(mul(z2ro, z2io) << 3));
  w.add(yo, op(c.get() << 2));
  Hx = u.get() + w.get();
}

}  // namespace emri
