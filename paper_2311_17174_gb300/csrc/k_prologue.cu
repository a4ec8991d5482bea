// k_prologue.cu -- step S0: per-walker constants.
//
// From the structure-of-arrays parameters, per walker:
//  * the orbit constants G M/c^3, G mu/c^3 and the right-hand-side
//    prefactors, all formed in double-double and rounded once;
//  * the starting PN velocity v0 = (2 pi G M nu0 / c^3)^(1/3) to dd accuracy
//    (one Newton step on the cube), because a rounding of v0 is a systematic
//    frequency offset that the phase integrates over ~1e4-1e5 cycles;
//  * the LISA geometry vectors of the source and spin directions;
//  * the propagation factors of the paper's Sec. 2: d_L(z) (32-point
//    Gauss-Legendre quadrature of the flat Lambda-CDM comoving integral),
//    Xi(z) of Eq. (6), d_GW = Xi d_L, and the GW-speed delay of Eqs. (4)-(5)
//    for constant alpha_T, dt_GW = -(alpha_T/2) t_lookback(z), with the
//    lookback time in closed form evaluated in double-double.  The delay is
//    ~1e15 s; the per-bin phase needs frac(dt_GW / T) to ~1e-16 absolute, so
//    it is formed and reduced in dd.
// The kernel is a chain of dependent FP64 instructions (64 cycles of an SM
// sub-partition each, whatever the active lanes), so a CTA splits one group
// of walkers' four independent chains over its four warps, one per
// sub-partition; the dd constants of the cosmology come from the host, and a
// dd exponential takes ~400 instructions.  One thread per walker running all
// of it in turn took 0.22..0.27 ms for any number of walkers up to 1024; this
// takes 0.04 ms for 8 and 0.05 ms for 1024.
#include "emri_common.cuh"
#include "emri_internal.h"
#include "fx64.cuh"

namespace emri {

__device__ __forceinline__ bool finite_all(const double* th, int64_t ld, int i) {
  for (int p = 0; p < kNParam; ++p)
    if (!isfinite(th[p * ld + i])) return false;
  return true;
}

// Constants of the cosmology and units, in dd, from the host.
struct ProConst {
  dd tsun;      // G M_sun / c^3
  dd k_lb;      // (1/H0) 2 / (3 sqrt(OL))
  dd s, ash_s;  // sqrt(OL/Om) and its asinh
};

static ProConst pro_const(double omega_m, double h0) {
  ProConst k;
  const dd c3 = dd_mul_d(two_prod(kC, kC), kC);
  k.tsun = dd_div(dd_make(kGMsun), c3);
  const dd om = dd_make(omega_m);
  const dd ol = dd_add_d(dd_neg(om), 1.0);
  k.s = dd_sqrt(dd_div(ol, om));
  k.ash_s = dd_asinh(k.s);
  const dd hinv = dd_div(dd_make(kMpc), two_prod(h0, 1e5));
  k.k_lb = dd_div(dd_mul_d(hinv, 2.0), dd_mul_d(dd_sqrt(ol), 3.0));
  return k;
}

// lookback time (flat Lambda-CDM, closed form) in dd:
//   t_LB = (1/H0) (2/(3 sqrt(OL))) [asinh(s) - asinh(s (1+z)^(-3/2))], s = sqrt(OL/Om)
__host__ __device__ inline dd lookback_dd(double zz, const ProConst& k) {
  const dd zp = two_sum(1.0, zz);
  const dd u = dd_div(k.s, dd_mul(zp, dd_sqrt(zp)));
  return dd_mul(k.k_lb, dd_sub(k.ash_s, dd_asinh(u)));
}

constexpr int kProWalkers = 8;   // walkers per CTA (four lanes each in the quadrature)

__global__ void __launch_bounds__(128) k0_prologue(const double* __restrict__ theta, int64_t ld, int w, int64_t n,
                                                   double dt, int mode, double n_xi, double omega_m, double h0,
                                                   ProConst K, const double* __restrict__ gl,
                                                   WalkerC* __restrict__ out, int role0) {
  __shared__ int bad_dgw[kProWalkers];
  const int role = role0 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  const int slot = role == 2 ? lane >> 2 : lane;        // the quadrature takes four lanes per walker
  const int i = blockIdx.x * kProWalkers + slot;
  const bool mine = slot < kProWalkers && i < w;
  uint32_t st = 0;
  double M = 0, mu = 0, spin = 0, e0 = 0, nu0 = 0, z = 0;
  if (mine) {
    M = theta[P_M * ld + i];
    mu = theta[P_MU * ld + i];
    spin = theta[P_SPIN * ld + i];
    e0 = theta[P_E0 * ld + i];
    nu0 = theta[P_NU0 * ld + i];
    z = theta[P_Z * ld + i];
    if (!finite_all(theta, ld, i) || !(M > 0) || !(mu > 0) || !(spin >= 0 && spin <= 1) || !(e0 >= 0 && e0 < 1) ||
        !(z >= 0) || (mode == 0 && !(nu0 > 0)))
      st |= ST_BADPARAM;
  }
  const double zz = st ? 0.0 : z;
  if (role == 0 && mine) {
    // orbit constants
    WalkerC& c = out[i];
    dd ms = dd_mul_d(K.tsun, st ? 1.0 : M);
    dd mus = dd_mul_d(K.tsun, st ? 1.0 : mu);
    dd ms2 = dd_mul(ms, ms);
    c.m_s = ms.hi;
    c.mu_s = mus.hi;
    c.spin = st ? 0.0 : spin;
    c.kv = dd_div(dd_mul_d(mus, 32.0), dd_mul_d(ms2, 5.0)).hi;   // (32/5) mu/M^2
    c.ke = dd_div(mus, ms2).hi;                                  // mu/M^2
    dd twopi{kTwoPiHi, kTwoPiLo};
    dd twopim = dd_mul(twopi, ms);
    c.inv2pim = dd_div(dd_make(1.0), twopim).hi;
    // starting velocity v0 = x0^(1/3), x0 = 2 pi M nu0 (forward) or the LSO value
    dd x0;
    if (mode == 0) {
      x0 = dd_mul_d(twopim, st ? 1e-3 : nu0);
    } else {
      // nu_LSO: x_LSO = ((1 - e^2)/(6 + 2 e))^(3/2)
      dd p = dd_div(dd_add_d(dd_neg(two_prod(e0, e0)), 1.0), dd_add_d(dd_make(2.0 * e0), 6.0));
      x0 = dd_mul(p, dd_sqrt(p));
    }
    double v = cbrt(x0.hi);
    dd v3 = dd_mul_d(two_prod(v, v), v);
    dd resid = dd_sub(v3, x0);
    dd vd = dd_add_d(dd_make(v), -resid.hi / (3.0 * v * v));
    c.v0_hi = vd.hi;
    c.v0_lo = vd.lo;
    c.e0 = st ? 0.0 : e0;
    c.phi0c = theta[P_PHI0 * ld + i] / kTwoPiHi;
    c.gam0c = theta[P_GAM0 * ld + i] / kTwoPiHi;
    c.alp0c = theta[P_ALP0 * ld + i] / kTwoPiHi;
    c.amp_scale = mus.hi * kC;
  } else if (role == 1 && mine) {
    // geometry
    WalkerC& c = out[i];
    const double amp_scale = dd_mul_d(K.tsun, st ? 1.0 : mu).hi * kC;
    double sinlam, coslam, sts, cts, sps, cps, stk, ctk, spk, cpk;
    sincos(theta[P_LAM * ld + i], &sinlam, &coslam);
    sincos(theta[P_THS * ld + i], &sts, &cts);
    sincos(theta[P_PHS * ld + i], &sps, &cps);
    sincos(theta[P_THK * ld + i], &stk, &ctk);
    sincos(theta[P_PHK * ld + i], &spk, &cpk);
    c.sinlam = sinlam; c.coslam = coslam;
    c.nx = sts * cps; c.ny = sts * sps; c.nz = cts;
    const double S[3] = {stk * cpk, stk * spk, ctk};
    double e1[3] = {1.0, 0.0, 0.0};
    if (fabs(stk) > 1e-12) {
      // e1 = (z - S cos thK)/sin thK, written out
      e1[0] = (0.0 - S[0] * ctk) / stk; e1[1] = (0.0 - S[1] * ctk) / stk; e1[2] = (1.0 - S[2] * ctk) / stk;
    }
    const double e2[3] = {S[1] * e1[2] - S[2] * e1[1], S[2] * e1[0] - S[0] * e1[2], S[0] * e1[1] - S[1] * e1[0]};
    c.sx = S[0]; c.sy = S[1]; c.sz = S[2];
    c.e1x = e1[0]; c.e1y = e1[1]; c.e1z = e1[2];
    c.e2x = e2[0]; c.e2y = e2[1]; c.e2z = e2[2];
    c.sin_ths = sts; c.cos_ths = cts; c.sin_phs = sps; c.cos_phs = cps;
    c.dop = kAUc * sts;
    // projections on the fixed sky basis P = (-sin phS, cos phS, 0),
    // Q = P x N = (cos phS cos thS, sin phS cos thS, -sin thS)
    const double P[3] = {-sps, cps, 0.0}, Q[3] = {cps * cts, sps * cts, -sts};
    auto dot = [](const double* a, const double* b) { return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]; };
    Geo<double> g;
    g.pe1 = dot(P, e1); g.pe2 = dot(P, e2); g.qe1 = dot(Q, e1); g.qe2 = dot(Q, e2);
    g.cpe1 = coslam * g.pe1; g.cpe2 = coslam * g.pe2;
    g.cqe1 = coslam * g.qe1; g.cqe2 = coslam * g.qe2;
    g.spS = sinlam * dot(P, S); g.sqS = sinlam * dot(Q, S);
    g.sin_ths = sts; g.cos_ths = cts; g.sin_phs = sps; g.cos_phs = cps;
    g.amp_scale = amp_scale;
    c.gd = g;
    Geo<float>& f = c.gf;
    f.pe1 = (float)g.pe1; f.pe2 = (float)g.pe2; f.qe1 = (float)g.qe1; f.qe2 = (float)g.qe2;
    f.cpe1 = (float)g.cpe1; f.cpe2 = (float)g.cpe2; f.cqe1 = (float)g.cqe1; f.cqe2 = (float)g.cqe2;
    f.spS = (float)g.spS; f.sqS = (float)g.sqS;
    f.sin_ths = (float)sts; f.cos_ths = (float)cts; f.sin_phs = (float)sps; f.cos_phs = (float)cps;
    f.amp_scale = (float)g.amp_scale;
    c.pad[0] = c.pad[1] = c.pad[2] = 0.0;
    c.j_plunge = n;
    c.pad_u = 0;
  } else if (role == 2) {
    // d_L(z) = (1+z)(c/H0) int_0^z dz'/E(z'), E = sqrt(Om (1+z)^3 + 1 - Om);
    // lane sub of a walker's four takes the nodes q = sub mod 4
    const int sub = lane & 3;
    double acc = 0.0;
    for (int q = sub; q < 32; q += 4) {
      const double a = 1.0 + 0.5 * zz * (gl[q] + 1.0);
      acc += gl[32 + q] * rsqrt(omega_m * a * a * a + (1.0 - omega_m));
    }
    acc += __shfl_xor_sync(0xffffffffu, acc, 1);
    acc += __shfl_xor_sync(0xffffffffu, acc, 2);
    if (mine && sub == 0) {
      WalkerC& c = out[i];
      const double hinv = kMpc / (h0 * 1e5);   // 1/H0 [s]
      const double d_l = (1.0 + zz) * kC * hinv * 0.5 * zz * acc;
      const double xi0 = theta[P_XI0 * ld + i];
      const double xi = xi0 + (1.0 - xi0) / pow(1.0 + zz, n_xi);
      const double d_gw = xi * d_l;
      c.d_l = d_l;
      c.xi = xi;
      c.d_gw = d_gw;
      bad_dgw[slot] = !(d_gw > 0);
    }
  } else if (role == 3 && mine) {
    // GW-speed delay from the lookback time in dd
    WalkerC& c = out[i];
    const double alpt = st ? 0.0 : theta[P_ALPT * ld + i];
    double dt_gw = 0.0, r_hi = 0.0, r_lo = 0.0, cn = 1.0, sn = 0.0;
    if (alpt != 0.0 && zz > 0.0) {
      dd dtgw = dd_mul_d(lookback_dd(zz, K), -0.5 * alpt);
      dd tobs = two_prod((double)n, dt);
      dd r = dd_frac(dd_div(dtgw, tobs));
      dt_gw = dtgw.hi;
      r_hi = r.hi;
      r_lo = r.lo;
      // exp(+2 pi i frac(N r))
      dd nr = dd_add_d(two_prod((double)n, r.hi), (double)n * r.lo);
      sincospi(2.0 * dd_frac(nr).hi, &sn, &cn);
    }
    c.dt_gw = dt_gw;
    c.r_hi = r_hi;
    c.r_lo = r_lo;
    c.cn_re = cn;
    c.cn_im = sn;
    c.cnf[0] = (float)cn;
    c.cnf[1] = (float)sn;
  }
  __syncthreads();
  if (role == 0 && mine) out[i].status = st | (bad_dgw[slot] ? (uint32_t)ST_BADPARAM : 0u);
  // a walker whose d_GW is not positive has no delay either.  (The delay's own
  // launch does not know d_GW; nothing reads that walker's delay there, its
  // waveform is zero.)
  if (role == 3 && role0 == 0 && mine && bad_dgw[slot]) {
    WalkerC& c = out[i];
    c.dt_gw = c.r_hi = c.r_lo = c.cn_im = 0.0;
    c.cn_re = 1.0;
    c.cnf[0] = 1.f;
    c.cnf[1] = 0.f;
  }
}

// Per-walker delay tables for the factorisation
// exp(-2 pi i k r) = exp(-2 pi i k2 r) exp(-2 pi i n2 k1 r) of bin k = k2 + n2 k1:
// tab[k] = exp(-2 pi i frac(mult k r)), k < count (mult = n2 over k1 < n1, and
// mult = 1 over k2 < n2).  fold_neg: the entries with 2 k > count also carry
// exp(+2 pi i frac(N r)), the factor of the signed index k - N (negative
// frequencies).
// The FP32 tables take the fraction in fixed point: r as a 128-bit fraction,
// m r mod 1 from two 64-bit integer products (exact), its top 32 bits as the
// phase in [-1/2, 1/2) cycles, then the FP32 sincospif; no FP64 operation
// per entry.  The FP64 tables take it in double-double and FP64 sincospi.
template <typename C2>
__global__ void k0_delay_table(const WalkerC* __restrict__ wc, int n1, int n2, C2* __restrict__ tab,
                               C2* __restrict__ rtab) {
  // grid x: the n1 column entries, then the n2 row entries (one launch)
  const int x = blockIdx.x * blockDim.x + threadIdx.x;
  const int wk = blockIdx.y;
  if (x >= n1 + n2) return;
  const bool row = x >= n1;
  const int k1 = row ? x - n1 : x, mult = row ? 1 : n2;
  const bool fold = !row && 2 * k1 > n1;
  C2* dst = row ? rtab + (int64_t)wk * n2 + k1 : tab + (int64_t)wk * n1 + k1;
  const double rh = wc[wk].r_hi, rl = wc[wk].r_lo;
  if constexpr (sizeof(C2) == 8) {
    unsigned long long Rh, Rl;
    dd_to_fx128(dd{rh, rl}, Rh, Rl);
    const unsigned long long m = (unsigned long long)mult * (unsigned long long)k1;   // < 2^22
    const unsigned long long ph = m * Rh + __umul64hi(m, Rl);                          // m r mod 1, Q0.64
    const float f = (float)(int)(unsigned)(ph >> 32) * 2.3283064365386963e-10f;        // [-1/2, 1/2)
    float sf, cf;
    sincospif(2.f * f, &sf, &cf);
    float vx = cf, vy = -sf;
    if (fold) {
      const float cr = wc[wk].cnf[0], ci = wc[wk].cnf[1];
      const float t = vx * cr - vy * ci;
      vy = vx * ci + vy * cr;
      vx = t;
    }
    *dst = make_float2(vx, vy);
  } else {
    double m = (double)mult * (double)k1;
    dd p = dd_add_d(two_prod(m, rh), m * rl);
    dd f = dd_frac(p);
    double s, c;
    sincospi(2.0 * f.hi, &s, &c);
    double vx = c, vy = -s;
    if (fold) {
      const double cr = wc[wk].cn_re, ci = wc[wk].cn_im;
      const double t = vx * cr - vy * ci;
      vy = vx * ci + vy * cr;
      vx = t;
    }
    // columns of 256 rows or more: the fixed-point pass 2 takes the factors as
    // (cos.h, cos.l, sin.h, sin.l), Q62 in balanced halves
    if (!row && n1 >= 256) {
      const fx::Op a = fx::bal(llrint(vx * 0x1p62)), b = fx::bal(llrint(vy * 0x1p62));
      *reinterpret_cast<int4*>(dst) = make_int4(a.h, a.l, b.h, b.l);
    } else {
      *dst = make_double2(vx, vy);
    }
  }
}

__global__ void k0_export(const WalkerC* __restrict__ wc, int w, double* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= w) return;
  const WalkerC& c = wc[i];
  out[0 * (int64_t)w + i] = c.d_l;
  out[1 * (int64_t)w + i] = c.xi;
  out[2 * (int64_t)w + i] = c.d_gw;
  out[3 * (int64_t)w + i] = c.dt_gw;
  out[4 * (int64_t)w + i] = c.r_hi;
  out[5 * (int64_t)w + i] = c.r_lo;
}

void launch_prologue(const double* theta, int64_t ld, int w, int64_t n, double dt, const OptsN& o,
                     const double* gl, WalkerC* out, cudaStream_t s, ProPart part) {
  if (w <= 0) return;
  const int role0 = part == ProPart::kDelay ? 3 : 0, roles = part == ProPart::kAll ? 4 : part == ProPart::kDelay ? 1 : 3;
  k0_prologue<<<(w + kProWalkers - 1) / kProWalkers, 32 * roles, 0, s>>>(
      theta, ld, w, n, dt, o.mode, o.n_xi, o.omega_m, o.h0, pro_const(o.omega_m, o.h0), gl, out, role0);
}

void launch_delay_table(const WalkerC* wc, int w, int n1, int n2, bool fp32, void* tab, void* rtab, cudaStream_t s) {
  // walkers on grid y, at most kMaxGridY per launch
  for (int w0 = 0; w0 < w; w0 += kMaxGridY) {
    const int ww = w - w0 < kMaxGridY ? w - w0 : kMaxGridY;
    const dim3 g((n1 + n2 + 255) / 256, ww);
    if (fp32)
      k0_delay_table<float2><<<g, 256, 0, s>>>(wc + w0, n1, n2, (float2*)tab + (int64_t)w0 * n1,
                                               (float2*)rtab + (int64_t)w0 * n2);
    else
      k0_delay_table<double2><<<g, 256, 0, s>>>(wc + w0, n1, n2, (double2*)tab + (int64_t)w0 * n1,
                                                (double2*)rtab + (int64_t)w0 * n2);
  }
}

void launch_prologue_export(const WalkerC* wc, int w, double* out, cudaStream_t s) {
  if (w <= 0) return;
  k0_export<<<(w + 127) / 128, 128, 0, s>>>(wc, w, out);
}

// ----------------------------------------- frequency-dependent propagation
// beta_m = -(t_LB/2) b_m df^(m+1) / f_*^m (cycles per |k|^(m+1)), reduced mod 1
// in dd before the conversion to fixed point.
__global__ void k0_fdprop(const double* __restrict__ theta, int64_t ld, int w, int64_t n, double dt, ProConst K, int qm, int qt, double fstar, const double* __restrict__ coef, int64_t ldc,
                          FdW* __restrict__ out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= w) return;
  FdW f{};
  f.qm = qm;
  f.qt = qt;
  double z = theta[P_Z * ld + i];
  if (!(z >= 0.0) || !isfinite(z)) z = 0.0;   // such a walker is flagged by the prologue
  f.nlz_half = -0.5 * log1p(z);
  const dd tobs = two_prod((double)n, dt);
  const dd df = dd_div(dd_make(1.0), tobs);
  f.xs = dd_div(df, dd_make(fstar)).hi;
  for (int m = 0; m < qm; ++m) f.a[m] = coef[(int64_t)m * ldc + i];
  if (qt > 0) {
    const dd tlb = z > 0.0 ? lookback_dd(z, K) : dd_make(0.0);
    const dd q = dd_div(df, dd_make(fstar));
    dd base = dd_mul(dd_mul_d(tlb, -0.5), df);   // -(t_LB/2) df
    for (int m = 0; m < qt; ++m) {
      base = dd_mul(base, q);                     // -(t_LB/2) df (df/f_*)^(m+1)
      const dd beta = dd_frac(dd_mul_d(base, coef[(int64_t)(qm + m) * ldc + i]));
      dd_to_fx128(beta, f.bhi[m], f.blo[m]);
    }
  }
  out[i] = f;
}

void launch_fdprop(const double* theta, int64_t ld, int w, int64_t n, double dt, const OptsN& o, int qm, int qt,
                   double fstar, const double* coef, int64_t ldc, FdW* fd, cudaStream_t s) {
  if (w <= 0) return;
  k0_fdprop<<<(w + 127) / 128, 128, 0, s>>>(theta, ld, w, n, dt, pro_const(o.omega_m, o.h0), qm, qt, fstar, coef,
                                               ldc, fd);
}

}  // namespace emri
