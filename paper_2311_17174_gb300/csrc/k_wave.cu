// k_wave.cu -- steps S2-S4: dense orbit, LISA response and the
// Peters-Mathews harmonic sum of Eq. (2), one CTA per one or four 1024-sample
// segments (FP64) or per segment of up to 4096 samples (mixed).
//
// Per segment (set-up):
//  * the cubic Hermite interpolant of every orbit quantity over each knot
//    interval (values and rates at both knots);
//  * the Bessel amplitudes of every harmonic at the segment's start, middle
//    and end, fitted by a quadratic in time.  The amplitudes depend on time
//    only through e(t), which moves by ~1e-4 relative per 256 samples, so the
//    quadratic is exact to ~1e-14 over 1024 and the per-sample cost of a
//    harmonic drops from a Bessel evaluation to a few FMAs;
//  * the four antenna patterns in a fixed sky polarisation basis at four
//    nodes of each 256-sample tile, fitted by a cubic in time (they depend on
//    time only through the LISA orbital phase, a one-year period).
// Per sample:
//  * phases Phi_D (Doppler folded in), 2 gamma~ and alpha from the Hermite
//    polynomials, modulo one cycle, and their sin/cos;
//  * the harmonic sum written as three running sums
//      C = sum_n n pa_n cos(n Phi), S = sum_n n sqrt(1-e^2) pb_n sin(n Phi),
//      R = sum_n 2 pc_n cos(n Phi),
//    with cos(n Phi), sin(n Phi) by the Chebyshev recurrence (or complex
//    rotation), Eq. (2)'s sum of A+_n and Ax_n regrouped;
//  * the response as a contraction in the fixed basis: (C, S) rotated by
//    2 gamma~, a quadratic form in the orbital-plane projections (linear in
//    cos alpha, sin alpha), times the fitted patterns -- identical to the
//    psi / beta form of the Barack-Cutler response, without either angle;
//  * z = h_I + i h_II.
// FP64 variant: phases, sums and response in 64-bit fixed point, the slowly
// varying factors in double (all of it in double outside the fixed-point
// ranges).  Mixed variant: the phases in 64-bit fixed point (linear term) plus
// an FP32 correction, the rest in FP32; no FP64 instruction runs per sample.
#include <vector>
#include "emri_common.cuh"
#include "emri_internal.h"
#include "wave_fixed.cuh"

namespace emri {

constexpr int kTile = 256;

// --------------------------------------------------------------- Bessel
// J_m(x) by its power series (x/2)^m / m! * sum_k a_k y^k, y = x^2/4,
// a_k = (-1)^k m! / (k! (m+k)!), evaluated by Horner's rule (one FMA per
// term) over the first K = min(ceil(12 + 1.05 x), 48) terms.  Wherever the
// series is used (orders m >= n + 1 at x = n e, n <= 32, e < 0.999) the
// omitted tail is below 1e-16 of the sum.  bc[m * kBesselTerms + k] = a_k and
// ifact[m] = 1/m! are tables (host long double, rounded once).
template <typename T>
__device__ __forceinline__ T bessel_series(int m, T x, const T* __restrict__ bc, const T* __restrict__ ifact) {
  const T half = T(0.5) * x;
  T lead = T(1);
  T p = half;
  for (int k = m; k; k >>= 1) {     // (x/2)^m by squaring
    if (k & 1) lead *= p;
    p *= p;
  }
  lead *= ifact[m];
  const T y = half * half;
  int K = (int)(T(12) + T(1.05) * x) + 1;
  if ((unsigned)(K - 1) >= (unsigned)kBesselTerms) K = kBesselTerms;
  const T* a = bc + m * kBesselTerms;
  T sum = a[K - 1];
#pragma unroll 4
  for (int k = K - 2; k >= 0; --k) sum = fma(sum, y, a[k]);
  return lead * sum;
}

// Amplitudes of harmonic n at eccentricity e:
//   a = n pa, b = n sqrt(1-e^2) pb, c = 2 pc  with the Peters-Mathews brackets
//   pa = J_{n-2} - 2e J_{n-1} + (2/n) J_n + 2e J_{n+1} - J_{n+2},
//   pb = J_{n-2} - 2 J_n + J_{n+2},  pc = J_n   (argument x = n e).
// J_{n+2}, J_{n+1} by series, the lower orders by the (stable) downward
// recurrence J_{m-1} = (2m/x) J_m - J_{m+1}, which also gives J_{-1} = -J_1.
template <typename T>
__device__ __forceinline__ void harmonic_amps(int n, T e, T out[3], const T* __restrict__ bc,
                                              const T* __restrict__ ifact) {
  T jm2, jm1, j0, jp1, jp2;
  if (e < T(1e-12)) {               // J_m(0) = delta_m0
    jm2 = n == 2 ? T(1) : T(0);
    jm1 = n == 1 ? T(1) : T(0);
    j0 = jp1 = jp2 = T(0);
  } else {
    const T x = T(n) * e;
    const T ix = T(1) / x;
    jp2 = bessel_series<T>(n + 2, x, bc, ifact);
    jp1 = bessel_series<T>(n + 1, x, bc, ifact);
    j0 = T(2 * (n + 1)) * ix * jp1 - jp2;
    jm1 = T(2 * n) * ix * j0 - jp1;
    jm2 = T(2 * (n - 1)) * ix * jm1 - j0;
  }
  const T pa = jm2 - T(2) * e * jm1 + (T(2) / T(n)) * j0 + T(2) * e * jp1 - jp2;
  const T pb = jm2 - T(2) * j0 + jp2;
  out[0] = T(n) * pa;
  out[1] = T(n) * sqrt(T(1) - e * e) * pb;
  out[2] = T(2) * j0;
}

// Series tables (once per context): a_k(m) = a_{k-1}(m) * (-1) / (k (m+k))
// and 1/m! in long double, rounded once to double and to float.
int upload_bessel_tables(const BesselTab& t) {
  std::vector<double> c64((size_t)kBesselOrders * kBesselTerms), f64(kBesselOrders);
  std::vector<float> c32(c64.size()), f32(kBesselOrders);
  long double fact = 1.0L;
  for (int m = 0; m < kBesselOrders; ++m) {
    if (m > 0) fact *= (long double)m;
    f64[m] = (double)(1.0L / fact);
    f32[m] = (float)(1.0L / fact);
    long double a = 1.0L;
    for (int k = 0; k < kBesselTerms; ++k) {
      if (k > 0) a = -a / ((long double)k * (long double)(m + k));
      c64[(size_t)m * kBesselTerms + k] = (double)a;
      c32[(size_t)m * kBesselTerms + k] = (float)a;
    }
  }
  bool ok = cudaMemcpy(t.c64, c64.data(), c64.size() * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess;
  ok = ok && cudaMemcpy(t.c32, c32.data(), c32.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess;
  ok = ok && cudaMemcpy(t.f64, f64.data(), f64.size() * sizeof(double), cudaMemcpyHostToDevice) == cudaSuccess;
  ok = ok && cudaMemcpy(t.f32, f32.data(), f32.size() * sizeof(float), cudaMemcpyHostToDevice) == cudaSuccess;
  return ok ? 0 : -1;
}

// exp(2 pi i k / 512), k = 0..511, for the FP64 sin/cos of phases in
// cycles; filled from the host (long double) at context creation.
constexpr int kExpLen = 512;
__device__ double2 g_exp512[kExpLen];
// exp(2 pi i k / 1024) in Q62 for the fixed-point sin/cos
__device__ fx::Trig g_trig[fx::kTrigLen];

static bool wave_smem_limits();

int upload_exp512() {
  double2 h[kExpLen];
  const long double pi = 3.141592653589793238462643383279502884L;
  for (int k = 0; k < kExpLen; ++k) {
    const long double a = 2.0L * pi * (long double)k / (long double)kExpLen;
    h[k] = make_double2((double)cosl(a), (double)sinl(a));
  }
  std::vector<fx::Trig> q(fx::kTrigLen);
  for (int k = 0; k < fx::kTrigLen; ++k) {
    const long double a = 2.0L * pi * (long double)k / (long double)fx::kTrigLen;
    q[k].c = llrintl(cosl(a) * 0x1p62L);
    q[k].s = llrintl(sinl(a) * 0x1p62L);
  }
  const bool ok = wave_smem_limits() && cudaMemcpyToSymbol(g_exp512, h, sizeof(h)) == cudaSuccess &&
                  cudaMemcpyToSymbol(g_trig, q.data(), q.size() * sizeof(fx::Trig)) == cudaSuccess;
  return ok ? 0 : -1;
}

// cos(2 pi f), sin(2 pi f) for a phase f in cycles (|f| < 2^20; whole cycles
// need not be removed first): f = k/512 + d with |d| <= 1/1024,
// exp(2 pi i k/512) from the table at k mod 512 and the Taylor polynomials
// of sin to x^5 and cos to x^4 at x = 2 pi d (|x| <= 0.00614: the first
// omitted terms, x^7/7! and x^6/6!, are below 7e-20 and 8e-17).  The
// nearest integer k of 512 f comes from adding 1.5 * 2^52: the sum rounds to
// an integer, its low word is k (two's complement) and subtracting the
// constant back gives k exactly, so no separate rounding or conversion
// instruction runs; d = f - k/512 is exact.  About 13 FP64 operations.
__device__ __forceinline__ void sincos2pi_tab(double f, const double2* __restrict__ tab, double& s, double& c) {
  constexpr double kRound = 6755399441055744.0;   // 1.5 * 2^52
  const double kb = fma(f, 512.0, kRound);
  const double kd = kb - kRound;
  const int k = __double2loint(kb);
  const double d = fma(kd, -0.001953125, f);   // exact
  const double x = d * 6.283185307179586;
  const double x2 = x * x;
  const double sx = fma(x2 * x, fma(x2, 1.0 / 120.0, -1.0 / 6.0), x);
  const double cx = fma(x2, fma(x2, 1.0 / 24.0, -0.5), 1.0);
  const double2 t = tab[k & (kExpLen - 1)];
  s = fma(t.y, cx, t.x * sx);
  c = fma(t.x, cx, -t.y * sx);
}

// ----------------------------------------------------- interval polynomials
// Cubic Hermite p(s) = c0 + c1 s + c2 s^2 + c3 s^3 on s in [0,1] from values
// y0, y1 and rates r0, r1 over an interval of length h.
__device__ __forceinline__ void hermite(double y0, double d, double r0, double r1, double h, double c[4]) {
  c[0] = y0;
  c[1] = h * r0;
  c[2] = 3.0 * d - h * (2.0 * r0 + r1);
  c[3] = h * (r0 + r1) - 2.0 * d;
}

template <typename T>
__device__ __forceinline__ T poly3(const T c[4], T s) {
  return ((c[3] * s + c[2]) * s + c[1]) * s + c[0];
}

struct IvD {           // FP64 interval data (gm: of 2 gamma~)
  double ph[4], gm[4], al[4], am[4], ec[4];
};

__device__ __forceinline__ double frac0(double hi, double lo) {
  return (hi - floor(hi)) + lo;
}

__device__ __forceinline__ void interval_phase(double ahi, double alo, double ar, double bhi, double blo,
                                               double br, double h, double c[4]) {
  const double d = (bhi - ahi) + (blo - alo);
  hermite(frac0(ahi, alo), d, ar, br, h, c);
}

__device__ void build_iv(const Knot& a, const Knot& b, double h, IvD& o) {
  interval_phase(a.phd_hi, a.phd_lo, a.phd_rate, b.phd_hi, b.phd_lo, b.phd_rate, h, o.ph);
  interval_phase(a.gam_hi, a.gam_lo, a.gam_rate, b.gam_hi, b.gam_lo, b.gam_rate, h, o.gm);
  for (int q = 0; q < 4; ++q) o.gm[q] *= 2.0;   // the kernel uses 2 gamma~ (exact scaling)
  interval_phase(a.alp_hi, a.alp_lo, a.alp_rate, b.alp_hi, b.alp_lo, b.alp_rate, h, o.al);
  hermite(a.amp, b.amp - a.amp, a.amp_rate, b.amp_rate, h, o.am);
  hermite(a.e, b.e - a.e, a.e_rate, b.e_rate, h, o.ec);
}

__device__ __forceinline__ unsigned long long to_q64(double f) {
  f -= floor(f);                                   // [0, 1)
  return (unsigned long long)(f * 18446744073709551616.0);
}

// a per-sample phase increment [cycles] as a signed Q0.64 fraction: the
// phase is kept mod 1, so the increment is reduced to [-1/2, 1/2) first (at
// long sample intervals it exceeds half a cycle)
__device__ __forceinline__ long long to_q64s(double f) {
  f -= rint(f);
  if (f >= 0.5) f -= 1.0;
  return (long long)llrint(f * 18446744073709551616.0);
}

__device__ void build_iv_mixed(const Knot& a, const Knot& b, double h, int ks, IvM& o) {
  double c[4];
  interval_phase(a.phd_hi, a.phd_lo, a.phd_rate, b.phd_hi, b.phd_lo, b.phd_rate, h, c);
  o.ph_base = to_q64(c[0]);
  o.ph_inc = to_q64s(c[1] / ks);
  o.ph_c[0] = (float)c[2];
  o.ph_c[1] = (float)c[3];
  interval_phase(a.gam_hi, a.gam_lo, a.gam_rate, b.gam_hi, b.gam_lo, b.gam_rate, h, c);
  for (int q = 0; q < 4; ++q) c[q] *= 2.0;   // the kernel uses 2 gamma~ (exact scaling)
  o.gm_base = to_q64(c[0]);
  o.gm_inc = to_q64s(c[1] / ks);
  o.gm_c[0] = (float)c[2];
  o.gm_c[1] = (float)c[3];
  interval_phase(a.alp_hi, a.alp_lo, a.alp_rate, b.alp_hi, b.alp_lo, b.alp_rate, h, c);
  o.al_base = to_q64(c[0]);
  o.al_inc = to_q64s(c[1] / ks);
  o.al_c[0] = (float)c[2];
  o.al_c[1] = (float)c[3];
  hermite(a.amp, b.amp - a.amp, a.amp_rate, b.amp_rate, h, c);
  for (int q = 0; q < 4; ++q) o.am[q] = (float)c[q];
  hermite(a.e, b.e - a.e, a.e_rate, b.e_rate, h, c);
  for (int q = 0; q < 4; ++q) o.ec[q] = (float)c[q];
}

// eccentricity on an interval, in the record's precision
__device__ __forceinline__ double iv_e(const IvD& v, double s) { return poly3<double>(v.ec, s); }
__device__ __forceinline__ float iv_e(const IvM& v, float s) { return poly3<float>(v.ec, s); }

static_assert(sizeof(IvM) == kIvMBytes, "interval record size");

// Knots -> mixed interval records, one thread per (interval, walker).
__global__ void k1b_intervals(const Knot* __restrict__ knots, int64_t nk, int ks, double dt, IvM* __restrict__ out) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= nk) return;
  const int64_t wk = blockIdx.y;
  const Knot* kn = knots + wk * (nk + 1);
  build_iv_mixed(kn[k], kn[k + 1], (double)ks * dt, ks, out[wk * nk + k]);
}

// cos, sin of the LISA orbital phase phibar = 2 pi t / T: the four
// pattern-fit nodes of each 256-sample tile (offsets 0, 256/3, 512/3, 256;
// tiles[4 tile + q]) and the knots every ks samples.
// They are the same for every walker, and a sine and cosine cost ~50 FP64
// instructions.
__global__ void k_lisa(int64_t ntiles, int64_t nknots, int ks, double t0, double dt, double2* __restrict__ tiles,
                       double2* __restrict__ knots) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, k = i - 4 * ntiles;
  if (k >= nknots) return;
  const double at = k >= 0 ? (double)(k * ks) : (double)((i >> 2) * 256) + 256.0 * (double)(i & 3) / 3.0;
  double f = (t0 + at * dt) / kYear;
  f -= floor(f);
  double sn, cs;
  sincospi(2.0 * f, &sn, &cs);
  (k >= 0 ? knots[k] : tiles[i]) = make_double2(cs, sn);
}

void launch_intervals_mixed(const Knot* knots, int w, int64_t n, int ks, double dt, void* ivs, cudaStream_t s) {
  if (w <= 0) return;
  const int64_t nk = n / ks;
  // walkers on grid y, at most kMaxGridY per launch
  for (int w0 = 0; w0 < w; w0 += kMaxGridY) {
    const int ww = w - w0 < kMaxGridY ? w - w0 : kMaxGridY;
    dim3 g((unsigned)((nk + 127) / 128), (unsigned)ww);
    k1b_intervals<<<g, 128, 0, s>>>(knots + (int64_t)w0 * (nk + 1), nk, ks, dt, (IvM*)ivs + (int64_t)w0 * nk);
  }
}

void launch_lisa(int64_t n, int ks, double t0, double dt, double* tiles, double2* knots, cudaStream_t s) {
  const int64_t nt = n / 256, nkn = n / ks + 1;
  k_lisa<<<(unsigned)((4 * nt + nkn + 127) / 128), 128, 0, s>>>(nt, nkn, ks, t0, dt, (double2*)tiles, knots);
}

// --------------------------------------------------- response + harmonics
template <typename T>
__device__ __forceinline__ T rcp_fast(T x) { return T(1) / x; }
template <>
__device__ __forceinline__ float rcp_fast<float>(float x) { return __fdividef(1.f, x); }

// (x, y) -> (cos 2 atan2(y, x), sin 2 atan2(y, x)); (1, 0) when degenerate
template <typename T>
__device__ __forceinline__ void double_angle(T x, T y, T& c2, T& s2, bool degenerate) {
  const T r2 = x * x + y * y;
  if (degenerate || !(r2 > T(0))) {
    c2 = T(1);
    s2 = T(0);
  } else {
    const T inv = rcp_fast(r2);
    c2 = (x * x - y * y) * inv;
    s2 = T(2) * x * y * inv;
  }
}

// cos(n Phi), sin(n Phi) for n = 1, 2, ...: complex rotation (FP32) or the
// Chebyshev three-term recurrence c_{n+1} = 2 cos(Phi) c_n - c_{n-1} (FP64,
// whose error growth ~n^2 eps is harmless at n <= 32 in double).
template <typename T>
struct HarmStep {
  T cn, sn, cp, sp, c1, s1;
  __device__ __forceinline__ void init(T c, T s) {
    cn = c; sn = s; cp = T(1); sp = T(0); c1 = c; s1 = s;
  }
  __device__ __forceinline__ void next();
};
template <>
__device__ __forceinline__ void HarmStep<double>::next() {
  const double tc = 2.0 * c1 * cn - cp, ts = 2.0 * c1 * sn - sp;
  cp = cn; sp = sn; cn = tc; sn = ts;
}

// a_n, b_n, c_n of harmonic index n at fit time st (FP64 layout: 9 per harmonic)
__device__ __forceinline__ void amps_at(const double* __restrict__ bq, int n, double st, double& an, double& bn,
                                        double& rn) {
  const double* b = bq + 9 * n;
  an = (b[2] * st + b[1]) * st + b[0];
  bn = (b[5] * st + b[4]) * st + b[3];
  rn = (b[8] * st + b[7]) * st + b[6];
}

// Harmonic sums at one sample (FP64): Cs = sum_n a_n cos(n Phi), Ss =
// sum_n b_n sin(n Phi), Rs = sum_n c_n cos(n Phi), with the amplitudes from
// the tile's fit bq at time st in [0, 1]; cph/sph: cos/sin of the Doppler
// orbital phase; (cos, sin)(n Phi) by the Chebyshev recurrence.
__device__ __forceinline__ void harmonic_sums(double cph, double sph, double st, const double* __restrict__ bq,
                                              int n_max, double& Cs, double& Ss, double& Rs) {
  Cs = 0.0;
  Ss = 0.0;
  Rs = 0.0;
  HarmStep<double> hs;
  hs.init(cph, sph);
  for (int n = 0; n < n_max; ++n) {
    double an, bn, rn;
    amps_at(bq, n, st, an, bn, rn);
    Cs += an * hs.cn;
    Ss += bn * hs.sn;
    Rs += rn * hs.cn;
    hs.next();
  }
}

// ----------------------------------------------------------- response
// The LISA response of Sec. 2 (Eq. 2 with the Barack-Cutler antenna
// patterns) contracts the detector tensor with the polarisation tensors, and
// the AK polarisations are the transverse-traceless projection of the
// orbit's quadrupole tensor
//   M = X (u1 u1 - u2 u2) + Y (u1 u2 + u2 u1) + Rs (u1 u1 + u2 u2),
// u1, u2 the orbital-plane basis of Geo (pericentre at angle gamma~ from u1),
// (X, Y) the harmonic sums (Cs, Ss) rotated by 2 gamma~.  The contraction does
// not depend on the polarisation basis, so it is taken in the fixed sky basis
// (P, Q) of Geo: the angle beta and the L-dependent polarisation angle psi
// drop out, and
//   h_I = F+_I H+ + Fx_I Hx,  H+ + i Hx = (Rs + X) z1^2 + (Rs - X) z2^2 + 2 Y z1 z2,
// z_k = P.u_k + i Q.u_k, with F_I, F_II the antenna patterns at the
// polarisation angle psi_P of P (tan psi_P = (z_d.Q)/(z_d.P), z_d the
// detector normal).  The patterns depend on time only through the LISA
// orbital phase phibar, a one-year period, so each tile fits them by a cubic.

// The four patterns (sqrt3/2 F+_I, sqrt3/2 Fx_I, sqrt3/2 F+_II, sqrt3/2 Fx_II)
// times scale at phibar = atan2(sb, cb): detector-frame polar angle
// cos(theta_d) = z_d.N, azimuth phi_d = phibar + atan2(sqrt3 cos thS + sin thS
// cos(phibar - phS), 2 sin thS sin(phibar - phS)), channel II at phi_d - pi/4.
template <typename T>
__device__ __forceinline__ void antenna_fixed(const Geo<T>& g, T cb, T sb, T scale, T F[4]) {
  const T h3 = T(kSqrt3Half);
  const T cdp = cb * g.cos_phs + sb * g.sin_phs;
  const T sdp = sb * g.cos_phs - cb * g.sin_phs;
  const T ct = T(0.5) * g.cos_ths - h3 * g.sin_ths * cdp;
  T c2x, s2x, c2p, s2p;
  double_angle<T>(T(2) * g.sin_ths * sdp, T(1.7320508075688772) * g.cos_ths + g.sin_ths * cdp, c2x, s2x, false);
  double_angle<T>(h3 * sdp, h3 * g.cos_ths * cdp + T(0.5) * g.sin_ths, c2p, s2p, false);
  const T c2b = cb * cb - sb * sb, s2b = T(2) * sb * cb;
  const T c2f = c2b * c2x - s2b * s2x;   // cos, sin of 2 phi_d
  const T s2f = s2b * c2x + c2b * s2x;
  const T q = T(0.5) * (T(1) + ct * ct);
  const T k = h3 * scale;
  F[0] = k * (q * c2f * c2p - ct * s2f * s2p);
  F[1] = k * (q * c2f * s2p + ct * s2f * c2p);
  F[2] = k * (q * s2f * c2p + ct * c2f * s2p);
  F[3] = k * (q * s2f * s2p - ct * c2f * c2p);
}

// Cubic c0 + c1 s + c2 s^2 + c3 s^3 through y0..y3 at s = 0, 1/3, 2/3, 1
// (Newton forward differences in u = 3 s).
template <typename T>
__device__ __forceinline__ void fit_cubic4(T y0, T y1, T y2, T y3, T* c) {
  const T d1 = y1 - y0, d2 = (y2 - y1) - d1, d3 = ((y3 - y2) - (y2 - y1)) - d2;
  c[0] = y0;
  c[1] = T(3) * (d1 - T(0.5) * d2 + d3 * T(1.0 / 3.0));
  c[2] = T(4.5) * (d2 - d3);
  c[3] = T(4.5) * d3;
}

template <typename T>
__device__ __forceinline__ T cubic_at(const T* c, T s) {
  return ((c[3] * s + c[2]) * s + c[1]) * s + c[0];
}

// Channels from the harmonic sums at one sample.  c2gt/s2gt: cos/sin of
// 2 gamma~; ca/sa: of alpha; A = x^(2/3); F: the four patterns at the sample.
template <typename T>
__device__ __forceinline__ void response(const Geo<T>& g, T c2gt, T s2gt, T ca, T sa, T A, T Cs, T Ss, T Rs,
                                         const T F[4], T& hI, T& hII) {
  const T z1r = sa * g.pe1 - ca * g.pe2, z1i = sa * g.qe1 - ca * g.qe2;
  const T z2r = ca * g.cpe1 + sa * g.cpe2 - g.spS, z2i = ca * g.cqe1 + sa * g.cqe2 - g.sqS;
  const T X = Cs * c2gt - Ss * s2gt, Y = Cs * s2gt + Ss * c2gt;
  const T a = A * (Rs + X), b = A * (Rs - X), y = T(2) * A * Y;
  const T Hp = a * (z1r * z1r - z1i * z1i) + b * (z2r * z2r - z2i * z2i) + y * (z1r * z2r - z1i * z2i);
  const T Hx = T(2) * (a * (z1r * z1i) + b * (z2r * z2i)) + y * (z1r * z2i + z1i * z2r);
  hI = F[0] * Hp + F[1] * Hx;
  hII = F[2] * Hp + F[3] * Hx;
}

__device__ __forceinline__ float2 neg2(float2 v) { return make_float2(-v.x, -v.y); }
__device__ __forceinline__ float2 lo2(float4 v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(float4 v) { return make_float2(v.z, v.w); }

// response<float> for two samples at once, every quantity a (sample A,
// sample B) pair and every step one paired FP32 instruction.  gk: the
// walker's geometry constants as duplicated pairs,
//   gk[0] = (pe1 pe1 -pe2 -pe2), gk[1] = (qe1 qe1 -qe2 -qe2),
//   gk[2] = (cpe1 cpe1 cpe2 cpe2), gk[3] = (cqe1 cqe1 cqe2 cqe2),
//   gk[4] = (-spS -spS -sqS -sqS).
__device__ __forceinline__ void response_pair(const float4* gk, float2 c2gt, float2 s2gt, float2 ca, float2 sa,
                                              float2 A, float2 Cs, float2 Ss, float2 Rs, const float2 F[4],
                                              float2& hI, float2& hII) {
  const float4 k0 = gk[0], k1 = gk[1], k2 = gk[2], k3 = gk[3], k4 = gk[4];
  const float2 z1r = __ffma2_rn(sa, lo2(k0), __fmul2_rn(ca, hi2(k0)));
  const float2 z1i = __ffma2_rn(sa, lo2(k1), __fmul2_rn(ca, hi2(k1)));
  const float2 z2r = __ffma2_rn(ca, lo2(k2), __ffma2_rn(sa, hi2(k2), lo2(k4)));
  const float2 z2i = __ffma2_rn(ca, lo2(k3), __ffma2_rn(sa, hi2(k3), hi2(k4)));
  const float2 X = __ffma2_rn(Cs, c2gt, neg2(__fmul2_rn(Ss, s2gt)));
  const float2 Y = __ffma2_rn(Cs, s2gt, __fmul2_rn(Ss, c2gt));
  const float2 a = __fmul2_rn(A, __fadd2_rn(Rs, X));
  const float2 b = __fmul2_rn(A, __fadd2_rn(Rs, neg2(X)));
  const float2 y = __fmul2_rn(__fadd2_rn(A, A), Y);
  const float2 u1 = __ffma2_rn(z1r, z1r, neg2(__fmul2_rn(z1i, z1i)));
  const float2 u2 = __ffma2_rn(z2r, z2r, neg2(__fmul2_rn(z2i, z2i)));
  const float2 u3 = __ffma2_rn(z1r, z2r, neg2(__fmul2_rn(z1i, z2i)));
  const float2 Hp = __ffma2_rn(a, u1, __ffma2_rn(b, u2, __fmul2_rn(y, u3)));
  const float2 v3 = __ffma2_rn(z1r, z2i, __fmul2_rn(z1i, z2r));
  const float2 w = __ffma2_rn(a, __fmul2_rn(z1r, z1i), __fmul2_rn(b, __fmul2_rn(z2r, z2i)));
  const float2 Hx = __ffma2_rn(y, v3, __fadd2_rn(w, w));
  hI = __ffma2_rn(F[0], Hp, __fmul2_rn(F[1], Hx));
  hII = __ffma2_rn(F[2], Hp, __fmul2_rn(F[3], Hx));
}

// Channels at one sample (harmonic sums, then the response).
__device__ __forceinline__ void channels(const Geo<double>& g, double cph, double sph, double c2gt, double s2gt,
                                         double ca, double sa, double A, double st, const double* __restrict__ bq,
                                         int n_max, const double F[4], double& hI, double& hII) {
  double Cs, Ss, Rs;
  harmonic_sums(cph, sph, st, bq, n_max, Cs, Ss, Rs);
  response<double>(g, c2gt, s2gt, ca, sa, A, Cs, Ss, Rs, F, hI, hII);
}


// quadratic in [0, 1] through f0, fh, f1 at 0, 1/2, 1
template <typename T>
__device__ __forceinline__ void fit3(T f0, T fh, T f1, T* q) {
  q[0] = f0;
  q[1] = T(-3) * f0 + T(4) * fh - f1;
  q[2] = T(2) * f0 - T(4) * fh + T(2) * f1;
}

// Amplitudes of one harmonic over a block of kBlk samples: a, b, c as
// A0 + A1 u + A2 u^2 in the sample offset u from the block's centre, each
// coefficient twice, so that the paired (f32x2) instructions of harmonic_sums4
// take natural register pairs.
struct __align__(16) BlkAmp {
  float4 a, b, c;   // (A0, A0, A1, A1)
  float4 ab2, c2;   // (A2 of a, twice, A2 of b, twice), (A2 of c, twice, -, -)
};
constexpr int kBlk = 128;

// FP32, four samples at once, as two (A, B) pairs of every quantity --
// cos(n Phi), sin(n Phi), the three amplitudes and the three sums -- so each
// step is one paired (f32x2) instruction on operands that are natural
// register pairs, and the coefficients of a harmonic (three 16-byte loads, five
// with kCurved) are loaded once for all four samples.  c1, s1: cos, sin of the
// Doppler orbital phase; u: offsets from the block's centre; C, S, R: sum_n a_n
// cos(n Phi), sum_n b_n sin(n Phi), sum_n c_n cos(n Phi).
template <bool kCurved>
__device__ __forceinline__ void harmonic_sums4(const float2 (&c1)[2], const float2 (&s1)[2], const float2 (&u)[2],
                                               const BlkAmp* __restrict__ amp, int n_max, bool cheb, float2 (&C)[2],
                                               float2 (&S)[2], float2 (&R)[2]) {
  for (int p = 0; p < 2; ++p) C[p] = S[p] = R[p] = make_float2(0.f, 0.f);
  auto harm = [&](int n, const float2 (&c)[2], const float2 (&sn)[2]) {
    const float4 xa = amp[n].a, xb = amp[n].b, xc = amp[n].c;
    float2 a1[2] = {hi2(xa), hi2(xa)}, b1[2] = {hi2(xb), hi2(xb)}, r1[2] = {hi2(xc), hi2(xc)};
    if (kCurved) {
      const float4 y = amp[n].ab2, w = amp[n].c2;
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        a1[p] = __ffma2_rn(lo2(y), u[p], a1[p]);
        b1[p] = __ffma2_rn(hi2(y), u[p], b1[p]);
        r1[p] = __ffma2_rn(lo2(w), u[p], r1[p]);
      }
    }
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      C[p] = __ffma2_rn(__ffma2_rn(a1[p], u[p], lo2(xa)), c[p], C[p]);
      S[p] = __ffma2_rn(__ffma2_rn(b1[p], u[p], lo2(xb)), sn[p], S[p]);
      R[p] = __ffma2_rn(__ffma2_rn(r1[p], u[p], lo2(xc)), c[p], R[p]);
    }
  };
  float2 cu[2] = {c1[0], c1[1]}, su[2] = {s1[0], s1[1]};
  int n = 0;
  if (cheb) {
    const float2 tc[2] = {make_float2(2.f * c1[0].x, 2.f * c1[0].y), make_float2(2.f * c1[1].x, 2.f * c1[1].y)};
    float2 cv[2] = {make_float2(1.f, 1.f), make_float2(1.f, 1.f)}, sv[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
    for (; n + 1 < n_max; n += 2) {
      harm(n, cu, su);
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        cv[p] = __ffma2_rn(tc[p], cu[p], neg2(cv[p]));
        sv[p] = __ffma2_rn(tc[p], su[p], neg2(sv[p]));
      }
      harm(n + 1, cv, sv);
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        cu[p] = __ffma2_rn(tc[p], cv[p], neg2(cu[p]));
        su[p] = __ffma2_rn(tc[p], sv[p], neg2(su[p]));
      }
    }
  } else {
    const float2 ns[2] = {neg2(s1[0]), neg2(s1[1])};
    for (; n + 1 < n_max; n += 2) {
      harm(n, cu, su);
      float2 cv[2], sv[2];
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        cv[p] = __ffma2_rn(cu[p], c1[p], __fmul2_rn(su[p], ns[p]));
        sv[p] = __ffma2_rn(su[p], c1[p], __fmul2_rn(cu[p], s1[p]));
      }
      harm(n + 1, cv, sv);
#pragma unroll
      for (int p = 0; p < 2; ++p) {
        cu[p] = __ffma2_rn(cv[p], c1[p], __fmul2_rn(sv[p], ns[p]));
        su[p] = __ffma2_rn(sv[p], c1[p], __fmul2_rn(cv[p], s1[p]));
      }
    }
  }
  if (n < n_max) harm(n, cu, su);
}

// Bessel amplitudes of a segment (FP32): nodes at sample offsets 0, L/2, L
// (L = span: the segment's length, or the last valid offset when the orbit
// plunges inside it), fitted by quadratics in t / L: bq[n][3 f + p] =
// coefficient p of quantity f.
constexpr int kQuadStride = 12;

__device__ __forceinline__ void tile_harmonics(const IvM* iv, int ni, int64_t j0, int64_t kfirst, int ks, int n_max,
                                               int span, float* bnode, float* bq, const float* __restrict__ bc,
                                               const float* __restrict__ ifact) {
  const int t = threadIdx.x;
  if (t < 3 * n_max) {
    // harmonic-major: a warp holds neighbouring n, whose series lengths
    // (growing with x = n e) are alike
    const int node = t % 3, n = t / 3 + 1;
    // node at offset span*node/2: integer arithmetic in half samples, so no
    // FP64 instruction runs here
    const int64_t pos2 = 2 * j0 + (int64_t)span * node;
    int64_t ki = pos2 / (2 * ks) - kfirst;
    if (ki > ni - 1) ki = ni - 1;
    if (ki < 0) ki = 0;
    const int64_t rem2 = pos2 - 2 * (kfirst + ki) * ks;
    float out[3];
    harmonic_amps<float>(n, iv_e(iv[ki], (float)rem2 / (float)(2 * ks)), out, bc, ifact);
    for (int f = 0; f < 3; ++f) bnode[(node * 32 + (n - 1)) * 3 + f] = out[f];
  }
  __syncthreads();
  if (t < 3 * n_max) {
    const int n = t / 3, f = t % 3;
    fit3(bnode[(0 * 32 + n) * 3 + f], bnode[(1 * 32 + n) * 3 + f], bnode[(2 * 32 + n) * 3 + f],
         bq + kQuadStride * n + 3 * f);
  }
}

// span of the Bessel fit: the L samples from j0, or up to the last sample
// before a plunge
__device__ __forceinline__ int tile_span(int64_t j0, int64_t jp, int L = kTile) {
  if (jp >= j0 + L) return L;
  const int64_t l = jp - 1 - j0;
  return l < 1 ? 1 : (int)l;
}

// ------------------------------------------------------------- kernels
// Above these sample intervals the per-tile cubic of the antenna patterns
// (error ~ (256 dt / T)^4) is replaced by their exact value per sample.
constexpr double kPatternFitDtMax64 = 64.0;     // [s]; fit error < 2e-12 below
constexpr double kPatternFitDtMaxM = 1024.0;    // [s]; fit error < 1e-7 below

// FP64 kernel: one CTA per segment of kSegF = 1024 samples (four tiles of
// 256; each thread evaluates its offset in the four tiles in turn), so the
// Bessel amplitude fit is made once per 1024 samples (its error over that
// span is ~1e-14 of the amplitudes) and the set-up's FP64 work, ~6 % of the
// kernel's at one fit per tile, drops four-fold.
constexpr int kSegF = 1024;

// The samples of a segment in double, for the segments the fixed-point form
// does not take: long sample intervals, whose antenna patterns
// are exact per sample, and orbits or geometries outside its ranges.
__device__ __noinline__ void wave_samples_f64(const IvD* iv, const double* bq, const double (*fq)[4][4],
                                              const Geo<double>& g, int64_t j0, int64_t kfirst, int64_t jplunge,
                                              int span, double dt, double t0, int ks, int n_max, double scale,
                                              int exact_f, double2* __restrict__ z) {
  constexpr int kTiles = kSegF / kTile;
  const int t = threadIdx.x;
  const double inv_span = 1.0 / (double)span;
  const int lks = __ffs(ks) - 1;   // ks: a power of two
  const double so = (double)t * (1.0 / kTile);
#pragma unroll 1
  for (int tt = 0; tt < kTiles; ++tt) {
    const int r = tt * kTile + t;   // offset in the segment
    const int64_t j = j0 + r;
    double2 out = make_double2(0.0, 0.0);
    if (j < jplunge) {
      const int ki = (int)((j >> lks) - kfirst);
      const double s = (double)(j - (kfirst + ki) * ks) * (1.0 / (double)ks);
      const IvD& v = iv[ki];
      // phases in cycles over the knot interval (|f| < 2^20: the table index
      // wraps them, no reduction to one cycle is needed)
      const double fph = poly3<double>(v.ph, s);
      const double fgm = poly3<double>(v.gm, s);
      const double fal = poly3<double>(v.al, s);
      const double A = poly3<double>(v.am, s);
      double F[4];
      if (!exact_f) {
#pragma unroll
        for (int q = 0; q < 4; ++q) F[q] = cubic_at<double>(fq[tt][q], so);
      } else {
        double f = (t0 + (double)j * dt) / kYear;
        f -= floor(f);
        double sb, cb;
        sincospi(2.0 * f, &sb, &cb);
        antenna_fixed<double>(g, cb, sb, scale, F);
      }
      double sph, cph, s2g, c2g, sa, ca;
      sincos2pi_tab(fph, g_exp512, sph, cph);
      sincos2pi_tab(fgm, g_exp512, s2g, c2g);
      sincos2pi_tab(fal, g_exp512, sa, ca);
      double hI, hII;
      channels(g, cph, sph, c2g, s2g, ca, sa, A, (double)r * inv_span, bq, n_max, F, hI, hII);
      out = make_double2(hI, hII);
    }
    z[j] = out;
  }
}

// ------------------------------------------- the same in fixed point (FP64)
// Phase of one knot interval in fixed point: base + inc tau (Q64, mod 1) plus
// s^2 (c2 + c3 s), s = tau / K_s, c2 in Q61 and c3 in Q62.
struct PhX {
  fx::u64 base;
  fx::i64 inc, c2, c3;
};
struct IvX {
  PhX ph, gm, al;
};

// false when the correction polynomial is outside its fixed-point range
__device__ __forceinline__ bool phase_fixed(const double c[4], int ks, PhX& o) {
  o.base = to_q64(c[0]);
  o.inc = to_q64s(c[1] / ks);
  o.c2 = llrint(c[2] * 0x1p61);
  o.c3 = llrint(c[3] * 0x1p62);
  return fabs(c[0]) < 1e9 && fabs(c[1]) < 1e9 && fabs(c[2]) < 1.0 && fabs(c[3]) < 1.0;   // (false for NaN)
}

// tau in [0, K_s), s31 = 2^31 tau / K_s
__device__ __forceinline__ fx::u64 phase_at(const PhX& v, int tau, int s31) {
  fx::i64 c = v.c2 + fx::mul31(v.c3, s31);      // Q61
  c = fx::mul31(fx::mul31(c, s31), s31);        // Q59
  return v.base + (fx::u64)tau * (fx::u64)v.inc + ((fx::u64)c << 5);
}

// Shared memory of one FP64 waveform CTA (kSub segments of kSegF samples).
template <int kSub>
struct WaveSmem {
  IvD iv[kSub * kSegF / 64];
  IvX ivx[kSub * kSegF / 64];
  fx::Trig ex[fx::kTrigLen];
  HarmX hx[kSub][32];
  double bnode[kSub][32][3][3];                // amplitudes [harmonic][a, b, c][node]
  double bq[kSub][32 * 9];
  double fn[kSub * kSegF / kTile][4][4];       // the four patterns at the four fit nodes of each tile
  double fq[kSub * kSegF / kTile][4][4];       // their cubics in (t mod 256) / 256
  Geo<double> g;
  GeoX gx;
  HarmScale hsc[kSub];
  int fixed_bad[kSub];
};

// In double a sample takes 333 FP64 instructions at n_max = 20, 76 cycles each:
// 156.3 ms for 128 walkers x 2^21 samples, 6.73 ms for 8 walkers x 2^21 at
// n_max = 10.  Here the phases, their sines and cosines, the harmonic sums and
// the response run in 64-bit fixed point on the integer pipe, ~800
// multiply-adds of 4 cycles and ~900 other instructions a sample at n_max = 20,
// and only the slowly varying factors (x^(2/3), the patterns) stay in double,
// beside them: 24 FP64 instructions.  30.1 and 1.35 ms, bound by the
// multiply-adds (~4500 cycles a warp in all).
//
// One CTA takes kSub segments: the set-up (Bessel amplitudes at three nodes a
// segment, antenna patterns, interval records) is a serial chain of ~200 FP64
// instructions, 20000 cycles, that few threads have work for in a single
// segment; four segments fill the CTA's warps with it and pay its latency once
// (56.7 -> 49.2 ms when the sums were slower).  A segment's result does not
// depend on kSub.  Three CTAs per SM at 80 registers, with spills of 64 (kSub =
// 1) and 52 bytes, against two at 126: 30.8 -> 30.1 ms, 16 sources x 2^16 0.141
// -> 0.128 ms.
template <int kSub>
__global__ void __launch_bounds__(kTile, 3) k2_wave_f64(const Knot* __restrict__ knots, const WalkerC* __restrict__ wcs,
                                                        int64_t n, double dt, double t0, int ks, int n_max,
                                                        double2* __restrict__ z, int unit_scale, int exact_f,
                                                        const double* __restrict__ bc, const double* __restrict__ ifact,
                                                        const double* __restrict__ lisa) {
  constexpr int kSub4 = kSegF / kTile, kTiles = kSub * kSub4;
  extern __shared__ __align__(16) unsigned char smraw[];
  WaveSmem<kSub>& S = *reinterpret_cast<WaveSmem<kSub>*>(smraw);
  const int wk = blockIdx.y;
  const WalkerC& C = wcs[wk];
  const int64_t nk = n / ks;
  const Knot* kn = knots + (int64_t)wk * (nk + 1);
  const int64_t j0 = (int64_t)blockIdx.x * (kSub * kSegF);
  const int lks = __ffs(ks) - 1;   // ks: a power of two, at most kSegF
  const int64_t kfirst = j0 >> lks;
  const int nis = kSegF >> lks;    // knot intervals per segment
  const int t = threadIdx.x;
  const double h = (double)ks * dt;
  const double scale = unit_scale ? C.gd.amp_scale : 1.0;
  z += (int64_t)wk * n;
  const int64_t jplunge = C.j_plunge;
  if (jplunge <= j0) {   // nothing left of the inspiral
    for (int r = t; r < kSub * kSegF; r += kTile) z[j0 + r] = make_double2(0.0, 0.0);
    return;
  }
  if (t < kSub) S.fixed_bad[t] = exact_f;
  __syncthreads();
  if (t < kSub * nis) {
    build_iv(kn[kfirst + t], kn[kfirst + t + 1], h, S.iv[t]);
    const bool ok0 = phase_fixed(S.iv[t].ph, ks, S.ivx[t].ph), ok1 = phase_fixed(S.iv[t].gm, ks, S.ivx[t].gm),
               ok2 = phase_fixed(S.iv[t].al, ks, S.ivx[t].al);
    if (!(ok0 && ok1 && ok2)) S.fixed_bad[t / nis] = 1;
  }
  if (t >= 256 - 4 * kTiles && !exact_f) {   // node q of tile tt
    const int i = t - (256 - 4 * kTiles), tt = i / 4, q = i % 4;
    const double* L = lisa + ((int64_t)blockIdx.x * kTiles + tt) * 8 + 2 * q;
    antenna_fixed<double>(C.gd, L[0], L[1], scale, S.fn[tt][q]);
  }
  if (t >= 160 && t < 170) {   // geometry constants, one per thread
    const Geo<double>& G = C.gd;
    const int i = t - 160;
    const double v = i == 0 ? G.pe1 : i == 1 ? -G.pe2 : i == 2 ? G.qe1 : i == 3 ? -G.qe2 : i == 4 ? G.cpe1
                   : i == 5 ? G.cpe2 : i == 6 ? G.cqe1 : i == 7 ? G.cqe2 : i == 8 ? -G.spS : -G.sqS;
    if (!(fabs(v) < 1.0000001))
      for (int q = 0; q < kSub; ++q) S.fixed_bad[q] = 1;
    if (i < 8) (&S.gx.pe1)[i] = fx::op(llrint(v * 0x1p62));
    else (&S.gx.spSn)[i - 8] = llrint(v * 0x1p60);
    if (i == 0) S.g = G;
  }
  for (int i = t; i < fx::kTrigLen; i += kTile) S.ex[i] = g_trig[i];
  __syncthreads();
  // Bessel amplitudes at a segment's start, middle and end (or last sample
  // before a plunge); neighbouring threads hold the same harmonic, whose
  // series lengths are alike
  for (int i = t; i < 3 * kSub * n_max; i += kTile) {
    const int m = i / (3 * kSub), sub = i % (3 * kSub) / 3, node = i % 3;
    const int64_t js = j0 + sub * kSegF;
    const int span = tile_span(js, jplunge, kSegF);
    const int64_t pos2 = 2 * js + (int64_t)span * node;   // in half samples
    int ki = (int)((pos2 >> (lks + 1)) - kfirst);
    if (ki > (sub + 1) * nis - 1) ki = (sub + 1) * nis - 1;
    const double s = (double)(pos2 - 2 * (kfirst + ki) * ks) / (double)(2 * ks);
    double out[3];
    harmonic_amps<double>(m + 1, iv_e(S.iv[ki], s), out, bc, ifact);
    for (int f = 0; f < 3; ++f) S.bnode[sub][m][f][node] = out[f];
  }
  __syncthreads();
  if (t < 32 * kSub) {   // quadratics and block exponents, a warp per segment and a lane per harmonic
    const int sub = t >> 5, m = t & 31;
    const float rs = (float)kSegF / (float)tile_span(j0 + sub * kSegF, jplunge, kSegF);
    float s0 = 0.f, s1 = 0.f, s2 = 0.f;
    if (m < n_max)
      for (int f = 0; f < 3; ++f) {
        const double* b = S.bnode[sub][m][f];
        double* o = S.bq[sub] + 9 * m + 3 * f;
        fit3(b[0], b[1], b[2], o);
        s0 += fabsf((float)o[0]);
        s1 += fabsf((float)o[1]) * rs;
        s2 += fabsf((float)o[2]) * (rs * rs);
      }
    for (int off = 16; off > 0; off >>= 1) {
      s0 += __shfl_xor_sync(0xffffffffu, s0, off);
      s1 += __shfl_xor_sync(0xffffffffu, s1, off);
      s2 += __shfl_xor_sync(0xffffffffu, s2, off);
    }
    if (m == 0) {
      S.hsc[sub] = harm_scale(1.0001f * s0, 1.0001f * s1, 1.0001f * s2);
      // amplitudes that move by more than 1/32 of their sum over the segment
      // (the unit of q0 follows 128 S1) or are not finite: in double
      if (!(s0 < 1e12f && 32.f * s1 < s0 && s2 < s0)) S.fixed_bad[sub] = 1;
    }
  }
  __syncthreads();
  for (int i = t; i < 9 * kSub * n_max; i += kTile) {
    const int sub = i / (9 * n_max), r = i % (9 * n_max), m = r / 9, f = (r % 9) / 3, p = r % 3;
    const HarmScale hs = S.hsc[sub];
    harm_put(S.hx[sub][m], m, f, p, S.bq[sub][r], hs, tile_span(j0 + sub * kSegF, jplunge, kSegF));
  }
  if (t >= 256 - 4 * kTiles && !exact_f) {   // pattern q of tile tt, in the sums' unit
    const int i = t - (256 - 4 * kTiles), tt = i / 4, q = i % 4;
    const double u = S.fixed_bad[tt / kSub4] ? 1.0 : pow2d(-2 - S.hsc[tt / kSub4].k0);
    fit_cubic4<double>(u * S.fn[tt][0][q], u * S.fn[tt][1][q], u * S.fn[tt][2][q], u * S.fn[tt][3][q], S.fq[tt][q]);
  }
  __syncthreads();
  const double so = (double)t * (1.0 / kTile);
  const double inv_ks = 1.0 / (double)ks;
#pragma unroll 1
  for (int tt = 0; tt < kTiles; ++tt) {
    const int sub = tt / kSub4;
    if (S.fixed_bad[sub]) {
      const int64_t js = j0 + sub * kSegF;
      wave_samples_f64(S.iv, S.bq[sub], S.fq + sub * kSub4, S.g, js, kfirst, jplunge, tile_span(js, jplunge, kSegF), dt,
                       t0, ks, n_max, scale, exact_f, z);
      tt += kSub4 - 1;
      continue;
    }
    const int rc = tt * kTile + t;     // offset in the CTA's samples
    const int64_t j = j0 + rc;
    double2 out = make_double2(0.0, 0.0);
    if (j < jplunge) {
      const int ki = rc >> lks, tau = rc & (ks - 1), s31 = tau << (31 - lks);
      const IvX& v = S.ivx[ki];
      const HarmX* hx = S.hx[sub];
      const int sh1 = S.hsc[sub].sh1, sh2 = S.hsc[sub].sh2, r = rc & (kSegF - 1);
      fx::i64 Cs, Ss, Rs, Hp, Hx;
      const fx::Trig ph = fx::sincos_cycles(phase_at(v.ph, tau, s31), S.ex);
      if (S.hsc[sub].two) harmonics_fixed<true>(ph, r, hx, n_max, sh1, sh2, Cs, Ss, Rs);
      else harmonics_fixed<false>(ph, r, hx, n_max, sh1, sh2, Cs, Ss, Rs);
      response_fixed(S.gx, fx::sincos_cycles(phase_at(v.gm, tau, s31), S.ex),
                     fx::sincos_cycles(phase_at(v.al, tau, s31), S.ex), Cs, Ss, Rs, Hp, Hx);
      const double A = poly3<double>(S.iv[ki].am, (double)tau * inv_ks);
      double F[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) F[q] = cubic_at<double>(S.fq[tt][q], so);
      const double hp = (double)Hp, hc = (double)Hx;
      out = make_double2(A * (F[0] * hp + F[1] * hc), A * (F[2] * hp + F[3] * hc));
    }
    z[j] = out;
  }
}

// Mixed kernel: one CTA per segment of kSegM = 1024, 2048 or 4096 samples, with
// the Bessel amplitude fit -- a quadratic in time per harmonic, from three
// nodes -- made once per segment.  The eccentricity moves by ~1e-4 relative per
// 256 samples, and the fit's error grows as the cube of the segment: ~5e-14 of
// the amplitudes over 2048 samples, far below FP32 resolution.  Longer
// segments spend less of the kernel in that set-up (its barrier waits); the
// launch takes the length from the series length alone (at least 16 segments
// per walker).
//
// A warp takes blocks of 128 samples, four per lane: the lanes first reduce the
// quadratics to the block (a lane per harmonic), where their curvature, ~2^-12
// of the segment's, is below FP32 resolution except close to a plunge
// (`curved`), so a harmonic takes 8 paired FMAs per pair of samples instead
// of 11 and three 16-byte loads instead of five; the samples of a pair lie 32
// apart in one knot interval, and share its record, the pattern cubics and the
// phase's 64-bit product.  Bound by instruction issue: 99 paired instructions, two slots each, and ~170 others
// a sample at n_max = 20 (114 paired with the quadratics evaluated per sample,
// 35.0 -> 33.8 ms for 1024 walkers x 2^21).  kOneIv (K_s >= 128): the block's
// four samples share one interval record; with it and 24 warps per SM at 80
// registers 33.2 -> 32.8 ms, although it then spills 72 bytes (stores; 92 of
// loads) that two records do not; at 64 registers it spills more: 34.1 ms.
// The set-up's barriers leave the other warps of a CTA idle: with four warps a
// CTA instead of eight 33.8 -> 33.3 ms (333 walkers x 2^18: 0.894 -> 0.869 ms);
// a call that does not fill the GPU keeps eight (8 walkers x 2^16: 16 against
// 22 us).
//
// exact_f: exact patterns per sample (long sample intervals), dphib: the
// LISA orbital phase step per sample [cycles] for them.  No FP64 instruction
// runs per thread: e0 is tested once per CTA.
template <int kSegM, int kMixThreads, bool kOneIv>
__global__ void __launch_bounds__(kMixThreads, 768 / kMixThreads) k2_wave_mixed(const WalkerC* __restrict__ wcs,
                                                          int64_t n, int exact_f, float dphib, int ks, int n_max,
                                                          float2* __restrict__ z, int unit_scale,
                                                          const float* __restrict__ bc, const float* __restrict__ ifact,
                                                          const double* __restrict__ lisa, const IvM* __restrict__ ivs) {
  constexpr int kTiles = kSegM / kTile;
  __shared__ IvM iv[kSegM / 64];
  __shared__ float bnode[3 * 32 * 3];
  __shared__ __align__(16) float bq[32 * kQuadStride];
  __shared__ BlkAmp amps[kMixThreads / 32][32];
  __shared__ float fn[kTiles][4][4];   // the four patterns at the fit nodes of each tile
  __shared__ __align__(16) float2 fq[kTiles][4][4];   // their cubics in (t mod 256) / 256, each coefficient twice
  __shared__ float cs0[kTiles][2];     // cos, sin phibar at each tile's start
  __shared__ Geo<float> g;
  __shared__ float4 gk[5];             // response_pair's duplicated geometry constants
  __shared__ int cheb_s;
  const int wk = blockIdx.y;
  const WalkerC& C = wcs[wk];
  const int64_t nk = n / ks;
  const int64_t j0 = (int64_t)blockIdx.x * kSegM;
  const int64_t kfirst = j0 / ks;
  const int ni = ks >= kSegM ? 1 : kSegM / ks;
  const int t = threadIdx.x, lane = t & 31, wq = t >> 5;
  const float scale = unit_scale ? C.gf.amp_scale : 1.f;
  const int64_t jplunge = C.j_plunge;
  z += (int64_t)wk * n + j0;
  if (jplunge <= j0) {   // nothing left of the inspiral
    for (int r = t; r < kSegM; r += kMixThreads) z[r] = make_float2(0.f, 0.f);
    return;
  }
  if (t < ni) iv[t] = ivs[(int64_t)wk * nk + kfirst + t];
  if (t >= kMixThreads - 4 * kTiles) {   // node q of tile tt
    const int i = t - (kMixThreads - 4 * kTiles), tt = i / 4, q = i % 4;
    const double* L = lisa + (blockIdx.x * kTiles + tt) * 8 + 2 * q;
    const float cb = (float)L[0], sb = (float)L[1];
    antenna_fixed<float>(C.gf, cb, sb, scale, fn[tt][q]);
    if (q == 0) {
      cs0[tt][0] = cb;
      cs0[tt][1] = sb;
    }
  }
  if (t == 0) {
    const Geo<float>& G = C.gf;
    g = G;
    gk[0] = make_float4(G.pe1, G.pe1, -G.pe2, -G.pe2);
    gk[1] = make_float4(G.qe1, G.qe1, -G.qe2, -G.qe2);
    gk[2] = make_float4(G.cpe1, G.cpe1, G.cpe2, G.cpe2);
    gk[3] = make_float4(G.cqe1, G.cqe1, G.cqe2, G.cqe2);
    gk[4] = make_float4(-G.spS, -G.spS, -G.sqS, -G.sqS);
    cheb_s = C.e0 < 0.5;
  }
  __syncthreads();
  if (t >= kMixThreads - 4 * kTiles) {   // pattern q of tile tt
    const int i = t - (kMixThreads - 4 * kTiles), tt = i / 4, q = i % 4;
    float cf[4];
    fit_cubic4<float>(fn[tt][0][q], fn[tt][1][q], fn[tt][2][q], fn[tt][3][q], cf);
#pragma unroll
    for (int k = 0; k < 4; ++k) fq[tt][q][k] = make_float2(cf[k], cf[k]);
  }
  const int span = tile_span(j0, jplunge, kSegM);
  const bool cheb = cheb_s != 0;   // per walker (uniform in the CTA)
  tile_harmonics(iv, ni, j0, kfirst, ks, n_max, span, bnode, bq, bc, ifact);
  __syncthreads();
  const float inv_span = 1.f / (float)span;
  const float inv_ks = 1.f / (float)ks;
  const int lks = __ffs(ks) - 1;   // ks is a power of two
  const int jv = (int)(jplunge - j0 < kSegM ? jplunge - j0 : kSegM);   // valid samples of the segment
  constexpr float kTwoPiF = 6.283185307179586f;
  // curvature over half a block against the amplitudes
  const float* q9 = bq + kQuadStride * lane;   // the lane's harmonic
  const float half = 0.5f * kBlk * inv_span;
  float m0 = 0.f, m2 = 0.f;
  if (lane < n_max) {
    m0 = fabsf(q9[0]) + fabsf(q9[3]) + fabsf(q9[6]);
    m2 = fabsf(q9[2]) + fabsf(q9[5]) + fabsf(q9[8]);
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    m0 += __shfl_xor_sync(0xffffffffu, m0, off);
    m2 += __shfl_xor_sync(0xffffffffu, m2, off);
  }
  const bool curved = !(m2 * (half * half) < 0x1p-26f * m0);
  BlkAmp* const amp = amps[wq];
  const float2 u[2] = {make_float2((float)(lane - 64), (float)(lane - 32)), make_float2((float)lane, (float)(lane + 32))};
  auto dup = [](float x) { return make_float2(x, x); };
  // cos, sin of a fixed-point phase (base + inc tau mod 1, plus s^2 (c0 + c1 s))
  // at tau and tau + 32 [the second 64-bit product is a sum], reduced to half a
  // cycle by adding and subtracting 1.5 * 2^23
  auto sincos2 = [&](unsigned long long base, long long inc, const float* c, int tau, float2 s, float2& cs, float2& sn) {
    const unsigned long long pa = base + (unsigned long long)tau * (unsigned long long)inc;
    const unsigned long long pb = pa + ((unsigned long long)inc << 5);
    float2 f = __fmul2_rn(__ffma2_rn(dup(c[1]), s, dup(c[0])), __fmul2_rn(s, s));
    f = __ffma2_rn(make_float2((float)(int)(unsigned)(pa >> 32), (float)(int)(unsigned)(pb >> 32)),
                   dup(2.3283064365386963e-10f), f);
    const float2 r = __fadd2_rn(__fadd2_rn(f, dup(12582912.f)), dup(-12582912.f));
    f = __fmul2_rn(__fadd2_rn(f, neg2(r)), dup(kTwoPiF));
    __sincosf(f.x, &sn.x, &cs.x);
    __sincosf(f.y, &sn.y, &cs.y);
  };
#pragma unroll 1
  for (int rb = wq * kBlk; rb < kSegM; rb += kMixThreads / 32 * kBlk) {
    if (rb >= jv) {
#pragma unroll
      for (int i = 0; i < 4; ++i) z[rb + 32 * i + lane] = make_float2(0.f, 0.f);
      continue;
    }
    __syncwarp();
    if (lane < n_max) {
      const float tc = (float)(rb + kBlk / 2) * inv_span;
      float A0[3], A1[3], A2[3];
#pragma unroll
      for (int f = 0; f < 3; ++f) {
        const float a = fmaf(q9[3 * f + 2], tc, q9[3 * f + 1]);
        A0[f] = fmaf(a, tc, q9[3 * f]);
        A1[f] = fmaf(q9[3 * f + 2], tc, a) * inv_span;
        A2[f] = q9[3 * f + 2] * (inv_span * inv_span);
      }
      BlkAmp& o = amp[lane];
      o.a = make_float4(A0[0], A0[0], A1[0], A1[0]);
      o.b = make_float4(A0[1], A0[1], A1[1], A1[1]);
      o.c = make_float4(A0[2], A0[2], A1[2], A1[2]);
      if (curved) {
        o.ab2 = make_float4(A2[0], A2[0], A2[1], A2[1]);
        o.c2 = make_float4(A2[2], A2[2], 0.f, 0.f);
      }
    }
    __syncwarp();
    // pair p: samples 64 p + lane (x) and 64 p + 32 + lane (y) of the block, in
    // one knot interval (K_s >= 64)
    float2 c1[2], s1[2], Cs[2], Ss[2], Rs[2];
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int ki = (kOneIv ? rb : rb + 64 * p) >> lks, tau = rb + 64 * p + lane - (ki << lks);
      const float2 s = make_float2((float)tau * inv_ks, (float)(tau + 32) * inv_ks);
      const IvM& v = iv[ki];
      sincos2(v.ph_base, v.ph_inc, v.ph_c, tau, s, c1[p], s1[p]);
    }
    if (curved) harmonic_sums4<true>(c1, s1, u, amp, n_max, cheb, Cs, Ss, Rs);
    else harmonic_sums4<false>(c1, s1, u, amp, n_max, cheb, Cs, Ss, Rs);
    const int tt = rb / kTile;
#pragma unroll
    for (int p = 0; p < 2; ++p) {
      const int ki = (kOneIv ? rb : rb + 64 * p) >> lks, tau = rb + 64 * p + lane - (ki << lks);
      const float2 s = make_float2((float)tau * inv_ks, (float)(tau + 32) * inv_ks);
      const IvM& v = iv[ki];
      float2 c2g, s2g, ca, sa, F[4], hI, hII;
      sincos2(v.gm_base, v.gm_inc, v.gm_c, tau, s, c2g, s2g);   // 2 gamma~
      sincos2(v.al_base, v.al_inc, v.al_c, tau, s, ca, sa);
      const float2 A = __ffma2_rn(__ffma2_rn(__ffma2_rn(dup(v.am[3]), s, dup(v.am[2])), s, dup(v.am[1])), s, dup(v.am[0]));
      const int ra = (rb & (kTile - 1)) + 64 * p + lane;      // offsets in the tile: ra, ra + 32
      if (!exact_f) {
        const float2 so = make_float2((float)ra * (1.f / kTile), (float)(ra + 32) * (1.f / kTile));
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float2* c = fq[tt][q];
          F[q] = __ffma2_rn(__ffma2_rn(__ffma2_rn(c[3], so, c[2]), so, c[1]), so, c[0]);
        }
      } else {
        float sd, cd, FA[4], FB[4];
        const float cb = cs0[tt][0], sb = cs0[tt][1];
        __sincosf(kTwoPiF * dphib * (float)ra, &sd, &cd);
        antenna_fixed<float>(g, cb * cd - sb * sd, sb * cd + cb * sd, scale, FA);
        __sincosf(kTwoPiF * dphib * (float)(ra + 32), &sd, &cd);
        antenna_fixed<float>(g, cb * cd - sb * sd, sb * cd + cb * sd, scale, FB);
#pragma unroll
        for (int q = 0; q < 4; ++q) F[q] = make_float2(FA[q], FB[q]);
      }
      response_pair(gk, c2g, s2g, ca, sa, A, Cs[p], Ss[p], Rs[p], F, hI, hII);
      const int r = rb + 64 * p + lane;
      z[r] = r < jv ? make_float2(hI.x, hII.x) : make_float2(0.f, 0.f);
      z[r + 32] = r + 32 < jv ? make_float2(hI.y, hII.y) : make_float2(0.f, 0.f);
    }
  }
}

static bool wave_smem_limits() {
  return cudaFuncSetAttribute(k2_wave_f64<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(WaveSmem<4>)) ==
             cudaSuccess &&
         cudaFuncSetAttribute(k2_wave_f64<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, sizeof(WaveSmem<1>)) ==
             cudaSuccess;
}

void launch_wave(const Knot* knots, const WalkerC* wc, int w, int64_t n, double dt, double t0,
                 const OptsN& o, void* z, bool unit_scale, const BesselTab& bt, const double* lisa, const void* ivs,
                 cudaStream_t s) {
  if (w <= 0) return;
  const int64_t nk = n / o.ks;
  // walkers on grid y, at most kMaxGridY per launch
  for (int w0 = 0; w0 < w; w0 += kMaxGridY) {
    const int ww = w - w0 < kMaxGridY ? w - w0 : kMaxGridY;
    const Knot* kn = knots + (int64_t)w0 * (nk + 1);
    if (o.precision == 0) {
      // four segments a CTA where that still gives every SM four CTAs
      const int sub = n >= 4 * kSegF && (n / (4 * kSegF)) * ww >= 4 * 152 ? 4 : 1;
      auto* kern = sub == 4 ? k2_wave_f64<4> : k2_wave_f64<1>;
      const size_t sm = sub == 4 ? sizeof(WaveSmem<4>) : sizeof(WaveSmem<1>);
      kern<<<dim3((unsigned)(n / (sub * kSegF)), (unsigned)ww), kTile, sm, s>>>(
          kn, wc + w0, n, dt, t0, o.ks, o.n_max, (double2*)z + (int64_t)w0 * n, unit_scale ? 1 : 0,
          dt > kPatternFitDtMax64 ? 1 : 0, bt.c64, bt.f64, lisa);
    } else {
      // segment length from the series length alone (so a walker's result
      // does not depend on the batch it is in): at least 16 segments per
      // walker, 1024 to 4096 samples
      const int seg = n >= (1 << 16) ? 4096 : n >= (1 << 15) ? 2048 : 1024;
      dim3 grid((unsigned)(n / seg), (unsigned)ww);
      const int ef = dt > kPatternFitDtMaxM ? 1 : 0;
      const float dpb = (float)(dt / kYear);
      float2* zz = (float2*)z + (int64_t)w0 * n;
      const IvM* iv = (const IvM*)ivs + (int64_t)w0 * nk;
      const int us = unit_scale ? 1 : 0;
#define EMRI_WAVE_MIXED(SEG, TH)                                                                                       \
  (o.ks >= kBlk ? k2_wave_mixed<SEG, TH, true> : k2_wave_mixed<SEG, TH, false>)<<<grid, TH, 0, s>>>(                   \
      wc + w0, n, ef, dpb, o.ks, o.n_max, zz, us, bt.c32, bt.f32, lisa, iv)
      // four warps a CTA where all CTA slots (six an SM) are taken, eight
      // where they are not; a sample's result is the same.  The shorter the
      // segment, the more its set-up waits for: 1024 walkers x 2^15 (2048
      // samples) 0.358 -> 0.301 ms, 2048 x 2^14 (1024) 0.452 -> 0.346 ms.
      const bool full = n / seg * ww >= 6 * 152;
      if (seg == 4096 && full) EMRI_WAVE_MIXED(4096, 128);
      else if (seg == 4096) EMRI_WAVE_MIXED(4096, 256);
      else if (seg == 2048 && full) EMRI_WAVE_MIXED(2048, 128);
      else if (seg == 2048) EMRI_WAVE_MIXED(2048, 256);
      else if (full) EMRI_WAVE_MIXED(1024, 128);
      else EMRI_WAVE_MIXED(1024, 256);
#undef EMRI_WAVE_MIXED
    }
  }
}

}  // namespace emri
