// The FP64 waveform kernel's fixed-point sines, harmonic sums and response on
// the host, beside the same steps in double and in long double.
#include <vector>
#include "wave_fixed.cuh"

using namespace emri;
typedef long double LD;
static const LD kPi = 3.141592653589793238462643383279502884L;

static const fx::Trig* table() {
  static std::vector<fx::Trig> t = [] {
    std::vector<fx::Trig> v(fx::kTrigLen);
    for (int k = 0; k < fx::kTrigLen; ++k) {
      const LD a = 2.0L * kPi * k / fx::kTrigLen;
      v[k] = fx::Trig{llrintl(cosl(a) * 0x1p62L), llrintl(sinl(a) * 0x1p62L)};
    }
    return v;
  }();
  return t.data();
}

static LD turns(uint64_t p) { return 2.0L * kPi * ((LD)(int64_t)p * 0x1p-64L); }

// cos, sin of a phase as the kernel's double form takes them: a table of 512
// steps and Taylor polynomials to x^4 and x^5
static void sincos_double(uint64_t p, double& c, double& s) {
  const uint64_t k = (p + (1ull << 54)) >> 55;
  const double x = (double)(int64_t)(p - (k << 55)) * 0x1p-64 * 6.283185307179586, x2 = x * x;
  const LD a = 2.0L * kPi * (LD)(k & 511) / 512;
  const double tc = (double)cosl(a), ts = (double)sinl(a);
  const double sx = fma(x2 * x, fma(x2, 1.0 / 120.0, -1.0 / 6.0), x), cx = fma(x2, fma(x2, 1.0 / 24.0, -0.5), 1.0);
  s = fma(ts, cx, tc * sx);
  c = fma(tc, cx, -ts * sx);
}

// Errors of cos and sin of the phases p (cycles, Q64), [count][2], in fixed
// point and in double.
extern "C" void sincos_errors(const uint64_t* p, int count, double* fixed, double* dbl) {
  for (int i = 0; i < count; ++i) {
    const fx::Trig t = fx::sincos_cycles(p[i], table());
    const LD c = cosl(turns(p[i])), s = sinl(turns(p[i]));
    double dc, ds;
    sincos_double(p[i], dc, ds);
    fixed[2 * i] = (double)((LD)t.c * 0x1p-62L - c);
    fixed[2 * i + 1] = (double)((LD)t.s * 0x1p-62L - s);
    dbl[2 * i] = (double)(dc - c);
    dbl[2 * i + 1] = (double)(ds - s);
  }
}

// q[n_max][3][3]: quadratics (in rho = r / 1024) of a_n, b_n, c_n; p, r: phase
// (cycles, Q64) and sample offset of each sample.  Errors of the three sums,
// [count][3], in fixed point and in double (Chebyshev recurrence and quadratics
// in double, as the kernel's double form), relative to sum |q0|.  Returns 1
// when the quadratic coefficients take two words.
extern "C" int harmonic_errors(const double* q, int n_max, const uint64_t* p, const int* r, int count, double* fixed,
                               double* dbl) {
  float s0 = 0.f, s1 = 0.f, s2 = 0.f;
  LD norm = 0;
  for (int i = 0; i < 3 * n_max; ++i) {
    s0 += fabsf((float)q[3 * i]);
    s1 += fabsf((float)q[3 * i + 1]);
    s2 += fabsf((float)q[3 * i + 2]);
    norm += fabs(q[3 * i]);
  }
  const HarmScale hs = harm_scale(1.0001f * s0, 1.0001f * s1, 1.0001f * s2);
  std::vector<HarmX> hx(n_max);
  for (int m = 0; m < n_max; ++m)
    for (int f = 0; f < 3; ++f)
      for (int k = 0; k < 3; ++k) harm_put(hx[m], m, f, k, q[9 * m + 3 * f + k], hs, 1024);
  for (int i = 0; i < count; ++i) {
    const fx::Trig cs = fx::sincos_cycles(p[i], table());
    fx::i64 C, S, R;
    if (hs.two) harmonics_fixed<true>(cs, r[i], hx.data(), n_max, hs.sh1, hs.sh2, C, S, R);
    else harmonics_fixed<false>(cs, r[i], hx.data(), n_max, hs.sh1, hs.sh2, C, S, R);
    LD ref[3] = {0, 0, 0};
    const LD rho = (LD)r[i] / 1024;
    for (int m = 0; m < n_max; ++m) {
      const LD c = cosl((m + 1) * turns(p[i])), s = sinl((m + 1) * turns(p[i]));
      for (int f = 0; f < 3; ++f) {
        const double* k = q + 9 * m + 3 * f;
        ref[f] += (k[0] + rho * (k[1] + rho * (LD)k[2])) * (f == 1 ? s : c);
      }
    }
    double c1, sn1;
    sincos_double(p[i], c1, sn1);
    const double st = r[i] / 1024.0;
    double cn = c1, sn = sn1, cp = 1.0, sp = 0.0, d[3] = {0, 0, 0};
    for (int m = 0; m < n_max; ++m) {
      for (int f = 0; f < 3; ++f) {
        const double* k = q + 9 * m + 3 * f;
        d[f] = fma(fma(fma(k[2], st, k[1]), st, k[0]), f == 1 ? sn : cn, d[f]);
      }
      const double tc = fma(2.0 * c1, cn, -cp), ts = fma(2.0 * c1, sn, -sp);
      cp = cn; sp = sn; cn = tc; sn = ts;
    }
    const fx::i64 v[3] = {C, S, R};
    for (int f = 0; f < 3; ++f) {
      fixed[3 * i + f] = (double)((ldexpl((LD)v[f], -6 - hs.k0) - ref[f]) / norm);
      dbl[3 * i + f] = (double)((d[f] - ref[f]) / norm);
    }
  }
  return hs.two;
}

// g[10] = pe1, pe2, qe1, qe2, cpe1, cpe2, cqe1, cqe2, spS, sqS; per sample
// phases of 2 gamma~ and alpha (Q64) and the sums (Q60).  Errors of H+ and Hx,
// [count][2], in fixed point and in double.
extern "C" void response_errors(const double* g, const uint64_t* gm, const uint64_t* al, const int64_t* sums, int count,
                                double* fixed, double* dbl) {
  GeoX x;
  const double sg[10] = {1, -1, 1, -1, 1, 1, 1, 1, -1, -1};
  for (int i = 0; i < 8; ++i) (&x.pe1)[i] = fx::op(llrint(sg[i] * g[i] * 0x1p62));
  for (int i = 8; i < 10; ++i) (&x.spSn)[i - 8] = llrint(sg[i] * g[i] * 0x1p60);
  // the same steps in T (k_wave.cu's response() at A = 1)
  auto steps = [&](auto ca, auto sa, auto c2, auto s2, auto C, auto S, auto R, auto& hp, auto& hx) {
    typedef decltype(C) T;
    const T z1r = sa * g[0] - ca * g[1], z1i = sa * g[2] - ca * g[3];
    const T z2r = ca * g[4] + sa * g[5] - g[8], z2i = ca * g[6] + sa * g[7] - g[9];
    const T X = C * c2 - S * s2, Y = C * s2 + S * c2, a = R + X, b = R - X, y = 2 * Y;
    hp = a * (z1r * z1r - z1i * z1i) + b * (z2r * z2r - z2i * z2i) + y * (z1r * z2r - z1i * z2i);
    hx = 2 * (a * (z1r * z1i) + b * (z2r * z2i)) + y * (z1r * z2i + z1i * z2r);
  };
  for (int i = 0; i < count; ++i) {
    const int64_t* u = sums + 3 * i;
    fx::i64 Hp, Hx;
    response_fixed(x, fx::sincos_cycles(gm[i], table()), fx::sincos_cycles(al[i], table()), u[0], u[1], u[2], Hp, Hx);
    LD hp, hx;
    double dp, dx, ca, sa, c2, s2;
    steps(cosl(turns(al[i])), sinl(turns(al[i])), cosl(turns(gm[i])), sinl(turns(gm[i])), (LD)u[0] * 0x1p-60L,
          (LD)u[1] * 0x1p-60L, (LD)u[2] * 0x1p-60L, hp, hx);
    sincos_double(al[i], ca, sa);
    sincos_double(gm[i], c2, s2);
    steps(ca, sa, c2, s2, (double)u[0] * 0x1p-60, (double)u[1] * 0x1p-60, (double)u[2] * 0x1p-60, dp, dx);
    fixed[2 * i] = (double)((LD)Hp * 0x1p-56L - hp);   // the sums' unit is 2^-4 of H's
    fixed[2 * i + 1] = (double)((LD)Hx * 0x1p-56L - hx);
    dbl[2 * i] = (double)(dp - hp);
    dbl[2 * i + 1] = (double)(dx - hx);
  }
}
