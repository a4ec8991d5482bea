// k_orbit.cu -- step S1: the AK orbit of Eq. (1), FP64.
//
// The paper integrates Y = {Phi, nu, e, gamma~, alpha} with a standard
// solver on the time grid (Sec. 3, "Waveform computation"; the right-hand
// side is the AK system of Barack & Cutler 2004 that the paper cites).
// A step-by-step integrator is a serial FP64 dependency chain per walker, and
// on this GPU one FP64 warp instruction occupies its SM sub-partition for ~64
// cycles; so the orbit is integrated in parallel in time.  The series is cut
// into segments (mcpi_segment), the solution on each represented by its
// values at the 32 Chebyshev-Gauss-Lobatto nodes (one per lane), and the
// collocation system y(t) = y(t_a) + int f(y) of all segments is solved at
// once by Newton's method (Chebyshev-Picard collocation, multiple shooting):
//   k1a_coarse   FP32 Picard sweeps over the segments in sequence: a starting
//                guess (~1e-6), one warp per walker;
//   k1b_eval     one warp per segment, three (rarely four) times: the FP64
//                rates at the nodes and the FP64 residual of the collocation
//                equations; the linearised correction is solved in FP32 (its
//                relative error, ~1e-4 to 1e-3, is the contraction per
//                evaluation: 1e-6 -> 1e-10 -> 1e-14 -> below rounding;
//                orbit_rule.cuh measures it and decides), with the
//                corrections of the segments' start values carried across
//                segments by the product of their 2x2 propagators;
//   k1c_final    the last correction, then all five rates at the nodes and
//                their integral over the segment;
//   k1d_starts   the segments' start states, compensated (hi + lo) sums in
//                time order, one warp per walker;
//   k1e_knots    the knots every K_s samples, read off the segment's
//                polynomial (integral weights at the knot positions), one
//                knot per lane over the whole GPU;
//   k1f_tail     walkers whose orbit reaches the LSO: the plunge sample, from
//                the knots around it; walkers whose orbit turns non-finite
//                or does not settle: the rest of the orbit from the first such
//                segment, in sequence (Picard sweeps, then knot-step RK4).
// The bound is the FP64 pipe when many walkers fill the GPU and the latency
// of the launch chain when few do.  One warp per walker doing all of it in
// sequence took 9.97 ms for 8 walkers x 2^21 samples at K_s = 128 (2.06 ms at
// K_s = 1024), 9.3 ms for 128 walkers at K_s = 128 and 3.6 ms for 1024 walkers
// at K_s = 1024; this takes 0.24 (0.14), 1.9 and 3.0 ms.  A single segment
// (8 walkers x 2^16) takes the same 0.10 ms either way.
// The same system is written in the variable
// v = x^(1/3) = (2 pi G M nu / c^3)^(1/3) instead of nu: then x^(2/3) = v^2,
// x^(11/3) = v^11 and (1-e^2)^(-k/2) = s^k with one s = 1/sqrt(1-e^2), so the
// right-hand side is polynomial apart from one reciprocal square root.
// With v = x^(1/3):
//   dv/dt      = (32/5)(mu/M^2) v^9 s^9 B_nu(v, e)
//   de/dt      = -(e/15)(mu/M^2) s^7 v^8 B_e(v, e) + e (mu/M^2) a cos(lam) v^11 s^8 C_e(e)
//   dPhi/dt/2pi = nu = v^3 / (2 pi M)
//   dgamma~/dt/2pi = 3 nu v^2 s^2 [1 + v^2 s^2 (26 - 15 e^2)/4] - 6 nu cos(lam) a v^3 s^3
//   dalpha/dt/2pi  = 2 nu a v^3 s^3
// which is dnu/dt = 3 nu v^-1 dv/dt applied to the paper's equations.
// All five states are compensated (hi + lo) sums over the segments, so the
// phase has no rounding drift.  Each knot stores the state and its rates;
// the Doppler delay nu (R/c) sin(theta_S) cos(phibar - phi_S) is folded into
// the stored phase, and the sample at which nu reaches nu_LSO(e) (paper
// Sec. 3) is located inside the crossing knot interval.
#include "emri_common.cuh"
#include "emri_internal.h"
#include "orbit_rule.cuh"

namespace emri {

template <typename T>
struct OrbSrcT {
  T kv, ke, inv2pim, spin, cl;
  int pn;
};
using OrbSrc = OrbSrcT<double>;

__device__ __forceinline__ OrbSrc orb_src(const WalkerC& c, int pn) {
  return OrbSrc{c.kv, c.ke, c.inv2pim, c.spin, c.coslam, pn};
}

__device__ __forceinline__ double rsqrt_t(double x) { return rsqrt(x); }
__device__ __forceinline__ float rsqrt_t(float x) { return rsqrtf(x); }

template <typename T>
__device__ __forceinline__ void ak_rhs_v(const OrbSrcT<T>& s, T v, T e, T& dv, T& de, T& dph, T& dg, T& da) {
  const T e2 = e * e, e4 = e2 * e2, e6 = e4 * e2;
  const T om = T(1.0) - e2;
  const T sq = rsqrt_t(om);
  const T s2 = sq * sq, s3 = s2 * sq, s4 = s2 * s2, s7 = s4 * s3, s8 = s4 * s4, s9 = s8 * sq;
  const T v2 = v * v, v3 = v2 * v, v4 = v2 * v2, v8 = v4 * v4, v9 = v8 * v, v11 = v9 * v2;
  const T a = s.spin, cl = s.cl;
  T br = (T(1.0) + T(73.0 / 24.0) * e2 + T(37.0 / 96.0) * e4) * om;
  T eb = (T(304.0) + T(121.0) * e2) * om;
  if (s.pn) {
    br += v2 * (T(1273.0 / 336.0) - T(2561.0 / 224.0) * e2 - T(3885.0 / 128.0) * e4 - T(13147.0 / 5376.0) * e6);
    br -= v3 * a * cl * sq *
          (T(73.0 / 12.0) + T(1211.0 / 24.0) * e2 + T(3143.0 / 96.0) * e4 + T(65.0 / 64.0) * e6);
    eb = eb * (T(1.0) + T(12.0) * v2) -
         T(1.0 / 56.0) * v2 * (T(8.0 * 16705.0) + T(12.0 * 9082.0) * e2 - T(25211.0) * e4);
  }
  dv = s.kv * v9 * s9 * br;
  de = -(e * T(1.0 / 15.0)) * s.ke * s7 * v8 * eb;
  if (s.pn)
    de += e * s.ke * a * cl * v11 * s8 * (T(1364.0 / 5.0) + T(5032.0 / 15.0) * e2 + T(263.0 / 10.0) * e4);
  const T nu = v3 * s.inv2pim;
  dph = nu;
  T g1 = T(3.0) * nu * v2 * s2;
  if (s.pn) g1 *= T(1.0) + T(0.25) * v2 * s2 * (T(26.0) - T(15.0) * e2);
  dg = g1 - T(6.0) * nu * cl * a * v3 * s3;
  da = T(2.0) * nu * a * v3 * s3;
}

template <typename T>
__device__ __forceinline__ void ak_rate_ve(const OrbSrcT<T>& s, T v, T e, T& dv, T& de) {
  T d0, d1, d2;
  ak_rhs_v(s, v, e, dv, de, d0, d1, d2);
}

struct OrbState {
  double v_hi, v_lo, e_hi, e_lo, p_hi, p_lo, g_hi, g_lo, a_hi, a_lo;
};

__device__ __forceinline__ bool plunged(double v, double e) {
  // nu >= nu_LSO(e)  <=>  x^(2/3) = v^2 >= (1 - e^2)/(6 + 2 e)
  return v * v >= (1.0 - e * e) / (6.0 + 2.0 * e);
}

__device__ __forceinline__ bool state_finite(const OrbState& y) {
  return isfinite(y.v_hi) && isfinite(y.e_hi) && isfinite(y.p_hi) && isfinite(y.g_hi) && isfinite(y.a_hi);
}

// One RK4 step of size h; k1 holds the rates at the current state.
__device__ __forceinline__ void rk4_step(const OrbSrc& s, OrbState& y, double h, const double k1[5]) {
  double k2[5], k3[5], k4[5];
  const double hh = 0.5 * h;
  ak_rhs_v(s, y.v_hi + hh * k1[0], y.e_hi + hh * k1[1], k2[0], k2[1], k2[2], k2[3], k2[4]);
  ak_rhs_v(s, y.v_hi + hh * k2[0], y.e_hi + hh * k2[1], k3[0], k3[1], k3[2], k3[3], k3[4]);
  ak_rhs_v(s, y.v_hi + h * k3[0], y.e_hi + h * k3[1], k4[0], k4[1], k4[2], k4[3], k4[4]);
  const double h6 = h / 6.0;
  double d[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) d[q] = h6 * (k1[q] + 2.0 * k2[q] + 2.0 * k3[q] + k4[q]);
  comp_add_small(y.v_hi, y.v_lo, d[0]);
  comp_add(y.e_hi, y.e_lo, d[1]);
  comp_add(y.p_hi, y.p_lo, d[2]);
  comp_add(y.g_hi, y.g_lo, d[3]);
  comp_add(y.a_hi, y.a_lo, d[4]);
}

// knot k of a walker; cs: cos, sin of the LISA orbital phase at the knots
__device__ __forceinline__ void write_knot(Knot* kn, int64_t kidx, const OrbState& y, const double r[5],
                                           const WalkerC& c, const double2* __restrict__ cs, int doppler) {
  Knot k;
  const double v = y.v_hi, nu = v * v * v * c.inv2pim;
  const double nudot = 3.0 * v * v * r[0] * c.inv2pim;
  double dsh = 0.0, dshdot = 0.0;
  if (doppler) {
    const double2 b = cs[kidx];
    const double cdp = b.x * c.cos_phs + b.y * c.sin_phs;
    const double sdp = b.y * c.cos_phs - b.x * c.sin_phs;
    dsh = c.dop * cdp;                                 // (R/c) sin thS cos(phibar - phiS) [s]
    dshdot = -c.dop * sdp * (kTwoPiHi / kYear);
  }
  dd ph = two_sum(y.p_hi, nu * dsh);
  ph = quick_two_sum(ph.hi, ph.lo + y.p_lo);
  k.phd_hi = ph.hi;
  k.phd_lo = ph.lo;
  k.phd_rate = r[2] + nudot * dsh + nu * dshdot;
  k.gam_hi = y.g_hi; k.gam_lo = y.g_lo; k.gam_rate = r[3];
  k.alp_hi = y.a_hi; k.alp_lo = y.a_lo; k.alp_rate = r[4];
  k.amp = v * v;
  k.amp_rate = 2.0 * v * r[0];
  k.e = y.e_hi;
  k.e_rate = r[1];
  k.pad0 = k.pad1 = k.pad2 = 0.0;
  kn[kidx] = k;
}

// Serial compensated RK4 at the knot step from knot k0 (state y, already
// written) over knots k0+1..k1.  Returns true if the orbit stayed inside the
// LSO; otherwise locates the plunge sample jp by re-integrating the crossing
// interval at the sampling step, writes the first knot past the crossing
// (the right end of the interval holding the last valid samples) and sets
// last to it.
__device__ bool rk4_span(const OrbSrc& s, const WalkerC& c, OrbState& y, int64_t k0, int64_t k1, int ks, double dt,
                         const double2* cs, int doppler, int64_t n, Knot* kn, int64_t& jp, uint32_t& st, int64_t& last) {
  const double h = (double)ks * dt;
  double r[5];
  ak_rhs_v(s, y.v_hi, y.e_hi, r[0], r[1], r[2], r[3], r[4]);
  for (int64_t k = k0; k < k1; ++k) {
    OrbState y0 = y;
    rk4_step(s, y, h, r);
    if (!state_finite(y) || plunged(y.v_hi, y.e_hi)) {
      OrbState f = y0;
      int64_t j = (k + 1) * ks;
      bool found = false;
      for (int q = 1; q <= ks; ++q) {
        double rr[5];
        ak_rhs_v(s, f.v_hi, f.e_hi, rr[0], rr[1], rr[2], rr[3], rr[4]);
        rk4_step(s, f, dt, rr);
        if (!state_finite(f) || plunged(f.v_hi, f.e_hi)) {
          j = k * ks + q;
          found = true;
          st |= state_finite(f) ? ST_PLUNGE : ST_NONFINITE;
          break;
        }
      }
      if (!found) st |= state_finite(y) ? ST_PLUNGE : ST_NONFINITE;
      jp = j < n ? j : n;
      if (jp == n) st &= ~(uint32_t)ST_PLUNGE;
      if (state_finite(y)) {
        ak_rhs_v(s, y.v_hi, y.e_hi, r[0], r[1], r[2], r[3], r[4]);
        write_knot(kn, k + 1, y, r, c, cs, doppler);
      } else {
        kn[k + 1] = kn[k];
      }
      last = k + 1;
      return false;
    }
    ak_rhs_v(s, y.v_hi, y.e_hi, r[0], r[1], r[2], r[3], r[4]);
    write_knot(kn, k + 1, y, r, c, cs, doppler);
    last = k + 1;
  }
  return true;
}

// ------------------------------------------- Chebyshev-Picard collocation
// Tables: qn[j*32 + i] = int_0^{tau_i} l_j(tau) dtau (transposed, nodes
// tau_i = (1 - cos(pi i/31))/2 on the unit segment); qk[q*32 + j] =
// int_0^{q/128} l_j, q = 0..128 (knot positions of the finest knot grid).
// Built on the host.
constexpr int kSeg = 65536;        // most samples per segment
// for parallelism alone, segments are not cut below so many samples and knots
constexpr int kSegLeast = 4096, kSegKnots = 32;

// Samples per segment (a power of two): at most 65536 and 128 knot intervals
// (the knot-weight table has 129 rows), and short enough for eight segments
// per walker as long as they keep 4096 samples and 32 knots, so that a small
// call's segments spread over the GPU.  A segment costs the same work whatever
// its length (32 nodes), which counts once walkers fill the GPU: at K_s = 1024,
// 1024 walkers x 2^15 take 0.20 ms in one segment each and 0.51 in eight, 8
// walkers x 2^16 0.099 in two and 0.107 in eight.
__host__ __device__ __forceinline__ int64_t mcpi_segment(int64_t n, int ks) {
  int64_t seg = kSeg;
  if (seg > 128 * (int64_t)ks) seg = 128 * (int64_t)ks;
  const int64_t least = kSegLeast > (int64_t)kSegKnots * ks ? kSegLeast : (int64_t)kSegKnots * ks;
  while (seg > least && 8 * seg > n) seg >>= 1;
  if (seg > n) seg = n;
  return seg;
}

// One coarse segment of the starting guess covers this many segments: a
// quarter of the sequential sweeps where there are many segments.
__host__ __device__ __forceinline__ int coarse_ratio(int64_t nseg) { return nseg >= 64 ? 4 : 1; }

// Solver state of one walker (segments in integration order i = 0..ns-1;
// backward mode integrates from the window's end).
struct OrbWork {
  double* nodes;   // [ns][2][32]   v, e at the nodes less the segment's start values
  char* work;      // [ns][1280 B]  J[4][32], Psi[4][32], dp[2][32] (float), then the final rates f5[5][32] (double)
  double* sums;    // [2][ns][6]    by evaluation parity: start v and e (hi, lo each), increments of v, e
  float* lin;      // [ns][8]       propagator P (4), then the end correction by parity (2 x 2)
  double* inc;     // [ns][5]       final increments of the five states
  double* start;   // [ns + 1][10]  compensated start states
  float* coarse;   // [ns / ratio][2][32] starting guess at the coarse nodes
  int* flag;       // [0] segments solved, [1] first segment with a bad knot, [2..4] sizes of the updates applied by
                   // evaluations 1..3 (float bits), [5] segments the starting guess covers, [6] first bad knot
};
constexpr int kOrbFlags = 8;

__host__ __device__ __forceinline__ size_t orb_walker_bytes(int64_t ns) {
  const int64_t nc = ns / coarse_ratio(ns);
  size_t b = (size_t)ns * (512 + 1280 + 96 + 32 + 40) + (size_t)(ns + 1) * 80 + (size_t)nc * 256 + kOrbFlags * 4;
  return (b + 255) & ~(size_t)255;
}

__device__ __forceinline__ OrbWork orb_work(char* base, int64_t wk, int64_t ns) {
  char* p = base + (size_t)wk * orb_walker_bytes(ns);
  OrbWork o;
  o.nodes = (double*)p;            p += ns * 512;
  o.work = p;                      p += ns * 1280;
  o.sums = (double*)p;             p += ns * 96;
  o.lin = (float*)p;               p += ns * 32;
  o.inc = (double*)p;              p += ns * 40;
  o.start = (double*)p;            p += (ns + 1) * 80;
  o.coarse = (float*)p;            p += (ns / coarse_ratio(ns)) * 256;
  o.flag = (int*)p;
  return o;
}

// Walker's start state in integration order: the prologue's values, and in
// backward mode (paper Sec. 3: initial conditions at the LSO, integrated back
// in time; the LSO state sits at the last sample t0 + (n-1) dt) one RK4 step
// of +dt to the last knot (sample n); the AK system is regular at the LSO.
__device__ __forceinline__ OrbState start_state(const OrbSrc& s, const WalkerC& c, int back, double dt) {
  OrbState y{c.v0_hi, c.v0_lo, c.e0, 0.0, c.phi0c, 0.0, c.gam0c, 0.0, c.alp0c, 0.0};
  if (back) {
    double r[5];
    ak_rhs_v(s, y.v_hi, y.e_hi, r[0], r[1], r[2], r[3], r[4]);
    rk4_step(s, y, dt, r);
  }
  return y;
}

// Starting guess: FP32 Picard sweeps over the coarse segments in sequence,
// one warp per walker, lane = node.  Each segment starts from the previous
// one's node increments scaled by the ratio of the start rates.  Bound by the
// latency of the FP32 chain, ~0.5 us per sweep.
__global__ void __launch_bounds__(32) k1a_coarse(const WalkerC* __restrict__ wcs, int64_t n, double dt, int ks, int pn,
                                                 int back, const double* __restrict__ qn_g, char* __restrict__ orb) {
  __shared__ float4 fx[16];      // (fv, fe) of the 32 nodes
  const int lane = threadIdx.x;
  const int64_t wk = blockIdx.x;
  const int64_t ns = n / mcpi_segment(n, ks);
  const int ratio = coarse_ratio(ns);
  const int nc = (int)(ns / ratio);
  const OrbWork o = orb_work(orb, wk, ns);
  const WalkerC& c = wcs[wk];
  float q[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) q[j] = (float)qn_g[j * 32 + lane];
  const OrbSrc s = orb_src(c, pn);
  const OrbState y = start_state(s, c, back, dt);
  if (lane == 0) {
    double* st = o.start;
    st[0] = y.v_hi; st[1] = y.v_lo; st[2] = y.e_hi; st[3] = y.e_lo; st[4] = y.p_hi; st[5] = y.p_lo;
    st[6] = y.g_hi; st[7] = y.g_lo; st[8] = y.a_hi; st[9] = y.a_lo;
  }
  const OrbSrcT<float> sf{(float)s.kv, (float)s.ke, (float)s.inv2pim, (float)s.spin, (float)s.cl, pn};
  const float H = (float)((double)(n / nc) * dt) * (back ? -1.f : 1.f);
  const float taui = 0.5f * (1.f - cospif((float)lane / 31.f));
  float va = (float)y.v_hi, ea = (float)y.e_hi;
  int good = (c.status & ST_BADPARAM) || !state_finite(y) || (!back && plunged(y.v_hi, y.e_hi)) ? 0 : nc;
  bool warm = false;
  float dvp = 0.f, dep = 0.f, fvp = 0.f, fep = 0.f;
  float2* fw = reinterpret_cast<float2*>(fx);
  for (int g = 0; g < nc && good == nc; ++g) {
    float f0v, f0e;
    ak_rate_ve(sf, va, ea, f0v, f0e);
    float v = va + (warm && fvp != 0.f ? dvp * (f0v / fvp) : H * taui * f0v);
    float e = ea + (warm && fep != 0.f ? dep * (f0e / fep) : H * taui * f0e);
    bool conv = false;
    for (int it = 0; it < 24; ++it) {
      float fv, fe;
      ak_rate_ve(sf, v, e, fv, fe);
      __syncwarp();
      fw[lane] = make_float2(fv, fe);
      __syncwarp();
      float sv0 = 0.f, se0 = 0.f, sv1 = 0.f, se1 = 0.f;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float4 a = fx[j];
        sv0 = fmaf(q[2 * j], a.x, sv0);
        se0 = fmaf(q[2 * j], a.y, se0);
        sv1 = fmaf(q[2 * j + 1], a.z, sv1);
        se1 = fmaf(q[2 * j + 1], a.w, se1);
      }
      const float vn = fmaf(H, sv0 + sv1, va), en = fmaf(H, se0 + se1, ea);
      const bool near = fabsf(vn - v) <= 4e-7f * fabsf(va) && fabsf(en - e) <= 4e-7f;
      v = vn;
      e = en;
      const bool ok = isfinite(v) && isfinite(e) && e * e < 1.f;
      if (__any_sync(0xffffffffu, !ok)) break;
      if (__all_sync(0xffffffffu, near)) {
        conv = true;
        break;
      }
    }
    if (!conv) {   // from here on in sequence
      good = g;
      break;
    }
    o.coarse[g * 64 + lane] = v;
    o.coarse[g * 64 + 32 + lane] = e;
    warm = true;
    dvp = v - va;
    dep = e - ea;
    fvp = f0v;
    fep = f0e;
    va = __shfl_sync(0xffffffffu, v, 31);
    ea = __shfl_sync(0xffffffffu, e, 31);
    // past the LSO at some node: the last segment needed (the system is
    // regular at the LSO)
    if (__any_sync(0xffffffffu, !back && v * v >= (1.f - e * e) / (6.f + 2.f * e))) {
      good = g + 1;
      break;
    }
  }
  if (lane < kOrbFlags)
    o.flag[lane] = lane == 0 || lane == 5 ? good * ratio : lane == 1 ? (int)ns : lane == 6 ? (int)(n / ks) + 1 : 0;
}

// Correction (v, e) of segment i's start value, from the previous
// evaluation's sums (parity p): d_{j+1} = m_j + P_j d_j over the segments
// j < i, m_j the mismatch between segment j's end and segment j+1's start
// plus the end value of j's own correction.  Lanes take 32 segments at a time
// and compose their affine maps in a tree.
__device__ __forceinline__ float2 start_correction(const OrbWork& o, int64_t ns, int i, int p, int lane) {
  float dv = 0.f, de = 0.f;
  const double* sm = o.sums + (int64_t)p * ns * 6;
  for (int j0 = 0; j0 < i; j0 += 32) {
    const int j = j0 + lane;
    float a = 1.f, b = 0.f, c = 0.f, d = 1.f, mv = 0.f, me = 0.f;
    if (j < i) {
      const double* u = sm + 6 * (int64_t)j;
      const float4 P = reinterpret_cast<const float4*>(o.lin + 8 * (int64_t)j)[0];
      const float2 ed = reinterpret_cast<const float2*>(o.lin + 8 * (int64_t)j + 4)[p];
      a = P.x; b = P.y; c = P.z; d = P.w;
      mv = (float)(((u[0] - u[6]) + u[4]) + (u[1] - u[7])) + ed.x;
      me = (float)(((u[2] - u[8]) + u[5]) + (u[3] - u[9])) + ed.y;
    }
#pragma unroll
    for (int off = 1; off < 32; off <<= 1) {   // own map first, the later lanes' after it
      const float a2 = __shfl_down_sync(0xffffffffu, a, off), b2 = __shfl_down_sync(0xffffffffu, b, off);
      const float c2 = __shfl_down_sync(0xffffffffu, c, off), d2 = __shfl_down_sync(0xffffffffu, d, off);
      const float mv2 = __shfl_down_sync(0xffffffffu, mv, off), me2 = __shfl_down_sync(0xffffffffu, me, off);
      const float na = a2 * a + b2 * c, nb = a2 * b + b2 * d, nc = c2 * a + d2 * c, nd = c2 * b + d2 * d;
      const float nv = a2 * mv + b2 * me + mv2, ne = c2 * mv + d2 * me + me2;
      a = na; b = nb; c = nc; d = nd; mv = nv; me = ne;
    }
    a = __shfl_sync(0xffffffffu, a, 0); b = __shfl_sync(0xffffffffu, b, 0);
    c = __shfl_sync(0xffffffffu, c, 0); d = __shfl_sync(0xffffffffu, d, 0);
    mv = __shfl_sync(0xffffffffu, mv, 0); me = __shfl_sync(0xffffffffu, me, 0);
    const float tv = a * dv + b * de + mv, te = c * dv + d * de + me;
    dv = tv;
    de = te;
  }
  return make_float2(dv, de);
}

// (v, e) at this lane's node: the segment's start values as (hi, lo) pairs --
// a rounding of the start would be a frequency offset over the whole segment
// -- and the node's increments from them.
struct NodeState {
  double vh, vl, eh, el, uv, ue;
  __device__ __forceinline__ double v() const { return vh + (vl + uv); }
  __device__ __forceinline__ double e() const { return eh + (el + ue); }
};

// The stored values plus the segment's own correction dp and the propagated
// start correction.  m: the size of the update over the segment (relative
// for v).
__device__ __forceinline__ NodeState apply_update(const OrbWork& o, int64_t ns, int i, int p, int lane, float& m) {
  const float2 d = start_correction(o, ns, i, p, lane);
  const float* wk = reinterpret_cast<const float*>(o.work + (int64_t)i * 1280);
  const float uv = wk[256 + lane] + (wk[128 + lane] - 1.f) * d.x + wk[160 + lane] * d.y;
  const float ue = wk[288 + lane] + wk[192 + lane] * d.x + (wk[224 + lane] - 1.f) * d.y;
  const double* u = o.sums + ((int64_t)p * ns + i) * 6;
  NodeState s;
  const dd v = two_sum(u[0], u[1] + (double)d.x), e = two_sum(u[2], u[3] + (double)d.y);
  s.vh = v.hi;
  s.vl = v.lo;
  s.eh = e.hi;
  s.el = e.lo;
  s.uv = o.nodes[(int64_t)i * 64 + lane] + (double)uv;
  s.ue = o.nodes[(int64_t)i * 64 + 32 + lane] + (double)ue;
  const float t = fmaxf(fabsf(uv + d.x) / (float)s.vh, fabsf(ue + d.y));
  // NaN compares above every limit: its bits as an integer are larger
  m = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(t == t ? t : __uint_as_float(0x7fc00000u))));
  return s;
}

constexpr int kEvalWarps = 4;   // segments per CTA (they share the integration matrix)

// x = r + H Q (J x) at the nodes, by FP32 iteration (contraction ~ H |J|,
// 0.03..0.3); lane = node, qf the FP32 integration matrix [j][node].
__device__ __forceinline__ float2 solve_linear(float2 r, const float4& J, float H, const float* qf, float2* xw,
                                               int lane) {
  float2 x = r;
  const float sv = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(r.x))));
  const float se = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(r.y))));
  const float tol = 1e-5f * fmaxf(sv, se);
  const float4* x4 = reinterpret_cast<const float4*>(xw);
  for (int it = 0; it < 30; ++it) {
    __syncwarp();
    xw[lane] = make_float2(J.x * x.x + J.y * x.y, J.z * x.x + J.w * x.y);
    __syncwarp();
    float a0 = 0.f, b0 = 0.f, a1 = 0.f, b1 = 0.f;
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const float4 t = x4[j];
      const float q0 = qf[2 * j * 32 + lane], q1 = qf[(2 * j + 1) * 32 + lane];
      a0 = fmaf(q0, t.x, a0);
      b0 = fmaf(q0, t.y, b0);
      a1 = fmaf(q1, t.z, a1);
      b1 = fmaf(q1, t.w, b1);
    }
    const float2 xn = make_float2(fmaf(H, a0 + a1, r.x), fmaf(H, b0 + b1, r.y));
    const bool near = fabsf(xn.x - x.x) <= tol && fabsf(xn.y - x.y) <= tol;
    x = xn;
    if (__all_sync(0xffffffffu, near)) break;
  }
  return x;
}

// One evaluation: the node values of this evaluation (the starting guess or
// the previous values plus their correction), the FP64 rates, the residual of
// the collocation equations and the segment's own FP32 correction.  kIt = 0
// also builds the node Jacobians and the propagators; kIt = 3 runs only for
// walkers that need it (orbit_again).  About 145 FP64
// instructions per lane and evaluation (70 for the rates, 64 for the node
// sums), which bound it.
template <int kIt>
__global__ void __launch_bounds__(32 * kEvalWarps) k1b_eval(const WalkerC* __restrict__ wcs, int64_t n, double dt,
                                                            int ks, int pn, int back,
                                                            const double* __restrict__ qn_g, char* __restrict__ orb) {
  __shared__ double qn[32 * 32];
  __shared__ float qf[32 * 32];
  __shared__ double2 fx[kEvalWarps][32];
  __shared__ __align__(16) float2 xw[kEvalWarps][32];
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  const int64_t wk = blockIdx.y;
  const int64_t seg = mcpi_segment(n, ks), ns = n / seg;
  const OrbWork o = orb_work(orb, wk, ns);
  const int good = o.flag[0];
  if ((int)(blockIdx.x * kEvalWarps) >= good) return;
  if (kIt == 3 && !orbit_again(__int_as_float(o.flag[2]), __int_as_float(o.flag[3]))) return;
  for (int t = threadIdx.x; t < 32 * 32; t += blockDim.x) {
    const double q = qn_g[t];
    qn[t] = q;
    qf[t] = (float)q;
  }
  __syncthreads();
  const int i = blockIdx.x * kEvalWarps + wq;
  if (i >= good) return;
  const WalkerC& c = wcs[wk];
  const OrbSrc s = orb_src(c, pn);
  const double H = (double)seg * dt * (back ? -1.0 : 1.0);
  constexpr int p = kIt & 1;
  float* wf = reinterpret_cast<float*>(o.work + (int64_t)i * 1280);
  NodeState y;
  if constexpr (kIt == 0) {
    // the coarse segment's Lagrange polynomial at this segment's nodes (the
    // node itself when the segments coincide), barycentric form
    const int ratio = coarse_ratio(ns);
    const float* cs = o.coarse + (int64_t)(i / ratio) * 64;
    float v, e;
    if (ratio == 1) {
      v = cs[lane];
      e = cs[32 + lane];
    } else {
      const float tau = ((float)(i % ratio) + 0.5f * (1.f - cospif((float)lane / 31.f))) / (float)ratio;
      const float x = 1.f - 2.f * tau;   // cos(theta), nodes at cos(pi j / 31)
      float num_v = 0.f, num_e = 0.f, den = 0.f, hit_v = 0.f, hit_e = 0.f;
      bool hit = false;
      for (int j = 0; j < 32; ++j) {
        const float cv = cs[j], ce = cs[32 + j];
        const float dx = x - cospif((float)j / 31.f);
        if (fabsf(dx) < 1e-6f) {
          hit = true;
          hit_v = cv;
          hit_e = ce;
        }
        const float wj = ((j & 1) ? -1.f : 1.f) * (j == 0 || j == 31 ? 0.5f : 1.f) / dx;
        num_v += wj * cv;
        num_e += wj * ce;
        den += wj;
      }
      v = hit ? hit_v : num_v / den;
      e = hit ? hit_e : num_e / den;
    }
    const float va = __shfl_sync(0xffffffffu, v, 0), ea = __shfl_sync(0xffffffffu, e, 0);
    y.uv = (double)(v - va);
    y.ue = (double)(e - ea);
    // the first segment starts from the walker's start value exactly
    y.vh = i == 0 ? o.start[0] : (double)va;
    y.vl = i == 0 ? o.start[1] : 0.0;
    y.eh = i == 0 ? o.start[2] : (double)ea;
    y.el = i == 0 ? o.start[3] : 0.0;
  } else {
    float m;
    y = apply_update(o, ns, i, p ^ 1, lane, m);
    if (lane == 0) atomicMax(&o.flag[1 + kIt], __float_as_int(m));
  }
  o.nodes[(int64_t)i * 64 + lane] = y.uv;
  o.nodes[(int64_t)i * 64 + 32 + lane] = y.ue;
  const double v = y.v(), e = y.e();
  double fv, fe;
  ak_rate_ve(s, v, e, fv, fe);
  fx[wq][lane] = make_double2(fv, fe);
  __syncwarp();
  double sv0 = 0.0, se0 = 0.0, sv1 = 0.0, se1 = 0.0;
#pragma unroll 8
  for (int j = 0; j < 32; j += 2) {
    const double q0 = qn[j * 32 + lane], q1 = qn[(j + 1) * 32 + lane];
    const double2 f0 = fx[wq][j], f1 = fx[wq][j + 1];
    sv0 = fma(q0, f0.x, sv0);
    se0 = fma(q0, f0.y, se0);
    sv1 = fma(q1, f1.x, sv1);
    se1 = fma(q1, f1.y, se1);
  }
  const double iv = H * (sv0 + sv1), ie = H * (se0 + se1);
  const float2 r = make_float2((float)(iv - y.uv), (float)(ie - y.ue));
  if (lane == 31) {
    double* u = o.sums + ((int64_t)p * ns + i) * 6;
    u[0] = y.vh;
    u[1] = y.vl;
    u[2] = y.eh;
    u[3] = y.el;
    u[4] = iv;
    u[5] = ie;
  }
  float4 J;
  const float Hf = (float)H;
  if constexpr (kIt == 0) {
    // central differences of the FP32 rates, steps of v/128 and (1 - e^2)/128
    // (relative error up to 9e-4: v^11)
    const OrbSrcT<float> sf{(float)s.kv, (float)s.ke, (float)s.inv2pim, (float)s.spin, (float)s.cl, pn};
    const float vf = (float)v, ef = (float)e;
    const float hv = vf * 0.0078125f, he = 0.0078125f * (1.f - ef * ef);
    float a0, b0, a1, b1;
    ak_rate_ve(sf, vf + hv, ef, a1, b1);
    ak_rate_ve(sf, vf - hv, ef, a0, b0);
    J.x = (a1 - a0) / (2.f * hv);
    J.z = (b1 - b0) / (2.f * hv);
    ak_rate_ve(sf, vf, ef + he, a1, b1);
    ak_rate_ve(sf, vf, ef - he, a0, b0);
    J.y = (a1 - a0) / (2.f * he);
    J.w = (b1 - b0) / (2.f * he);
    wf[lane] = J.x;
    wf[32 + lane] = J.y;
    wf[64 + lane] = J.z;
    wf[96 + lane] = J.w;
    const float2 c0 = solve_linear(make_float2(1.f, 0.f), J, Hf, qf, xw[wq], lane);
    const float2 c1 = solve_linear(make_float2(0.f, 1.f), J, Hf, qf, xw[wq], lane);
    wf[128 + lane] = c0.x;
    wf[160 + lane] = c1.x;
    wf[192 + lane] = c0.y;
    wf[224 + lane] = c1.y;
    if (lane == 31) reinterpret_cast<float4*>(o.lin + 8 * (int64_t)i)[0] = make_float4(c0.x, c1.x, c0.y, c1.y);
  } else {
    J = make_float4(wf[lane], wf[32 + lane], wf[64 + lane], wf[96 + lane]);
  }
  const float2 d = solve_linear(r, J, Hf, qf, xw[wq], lane);
  wf[256 + lane] = d.x;
  wf[288 + lane] = d.y;
  // the mismatch of start_correction compares the integrated end with the
  // next start; this is the part the own correction adds to the end: the
  // node-31 correction less the residual it already includes
  if (lane == 31) reinterpret_cast<float2*>(o.lin + 8 * (int64_t)i + 4)[p] = make_float2(d.x - r.x, d.y - r.y);
}

// The last correction, the five rates at the corrected nodes and their
// integrals over the segment.  A segment that has not settled leaves the
// walker's segments from it on to k1f_tail (those before it do not depend on
// it).
__global__ void __launch_bounds__(32 * kEvalWarps) k1c_final(const WalkerC* __restrict__ wcs, int64_t n, double dt,
                                                             int ks, int pn, int back,
                                                             const double* __restrict__ qn_g, char* __restrict__ orb) {
  const int lane = threadIdx.x & 31, wq = threadIdx.x >> 5;
  const int64_t wk = blockIdx.y;
  const int64_t seg = mcpi_segment(n, ks), ns = n / seg;
  const OrbWork o = orb_work(orb, wk, ns);
  const int i = blockIdx.x * kEvalWarps + wq;
  // [5]: segments the coarse pass reached; [0] is lowered here
  if (i >= o.flag[5]) return;
  const float u1 = __int_as_float(o.flag[2]), u2 = __int_as_float(o.flag[3]);
  const int p = orbit_again(u1, u2) ? 1 : 0;
  float m;
  const NodeState y = apply_update(o, ns, i, p, lane, m);
  if (!(p ? orbit_settled(u2, __int_as_float(o.flag[4]), m) : orbit_settled(u1, u2, m))) {
    if (lane == 0) atomicMin(&o.flag[0], i);
    return;
  }
  const OrbSrc s = orb_src(wcs[wk], pn);
  double f[5];
  ak_rhs_v(s, y.v(), y.e(), f[0], f[1], f[2], f[3], f[4]);
  const double H = (double)seg * dt * (back ? -1.0 : 1.0);
  const double wend = qn_g[lane * 32 + 31];   // node 31 is the segment's end
  double* f5 = reinterpret_cast<double*>(o.work + (int64_t)i * 1280);
  __syncwarp();   // every lane has read the segment's corrections
#pragma unroll
  for (int q = 0; q < 5; ++q) f5[q * 32 + lane] = f[q];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    double t = wend * f[q];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) t += __shfl_xor_sync(0xffffffffu, t, off);
    if (lane == 0) o.inc[(int64_t)i * 5 + q] = H * t;
  }
}

// The segments' start states as compensated sums in integration order: lanes
// 0..4 take one state each.
__global__ void __launch_bounds__(32) k1d_starts(int64_t n, int ks, char* __restrict__ orb) {
  extern __shared__ double inc[];
  const int lane = threadIdx.x;
  const int64_t ns = n / mcpi_segment(n, ks);
  const OrbWork o = orb_work(orb, blockIdx.x, ns);
  const int good = o.flag[0];
  for (int t = lane; t < 5 * good; t += 32) inc[t] = o.inc[t];
  __syncwarp();
  if (lane >= 5) return;
  double hi = o.start[2 * lane], lo = o.start[2 * lane + 1];
  for (int i = 0; i < good; ++i) {
    comp_add(hi, lo, inc[5 * i + lane]);
    o.start[(int64_t)(i + 1) * 10 + 2 * lane] = hi;
    o.start[(int64_t)(i + 1) * 10 + 2 * lane + 1] = lo;
  }
}

__device__ __forceinline__ OrbState load_start(const OrbWork& o, int64_t i) {
  const double* a = o.start + i * 10;
  return OrbState{a[0], a[1], a[2], a[3], a[4], a[5], a[6], a[7], a[8], a[9]};
}

// State at knot q (1..K) of a segment from its start state y and node rates
// f5 (weights row w): y + H sum_j w_j f_j, compensated.
__device__ __forceinline__ void knot_state(OrbState& y, const double* f5, const double* w, double H) {
  double sm[5] = {0, 0, 0, 0, 0};
#pragma unroll 4
  for (int j = 0; j < 32; ++j) {
    const double wj = w[j];
#pragma unroll
    for (int cc = 0; cc < 5; ++cc) sm[cc] = fma(wj, f5[cc * 32 + j], sm[cc]);
  }
  comp_add_small(y.v_hi, y.v_lo, H * sm[0]);
  comp_add(y.e_hi, y.e_lo, H * sm[1]);
  comp_add(y.p_hi, y.p_lo, H * sm[2]);
  comp_add(y.g_hi, y.g_lo, H * sm[3]);
  comp_add(y.a_hi, y.a_lo, H * sm[4]);
}

// Knots 1..n/K_s in integration order, one per lane (a warp's 32 knots lie in
// one segment, or in 32/K of them when a segment has K < 32 knots), and the
// start knot.  ~400 FP64 instructions per knot, 160 of them the node sums:
// bound by the FP64 pipe.  A knot past the LSO (forward) or not finite lowers
// flag[1] to its segment and flag[6] to itself.
constexpr int kRateStride = 161;   // doubles per segment in shared memory (odd: no bank conflicts between segments)
__global__ void __launch_bounds__(32) k1e_knots(const WalkerC* __restrict__ wcs, int64_t n, double dt,
                                                const double2* __restrict__ cs, int ks, int pn, int back, int doppler,
                                                const double* __restrict__ qk_g, char* __restrict__ orb,
                                                Knot* __restrict__ knots) {
  extern __shared__ double f5s[];
  const int lane = threadIdx.x;
  const int64_t wk = blockIdx.y;
  const int64_t seg = mcpi_segment(n, ks), ns = n / seg, nk = n / ks;
  const int K = (int)(seg / ks);
  const OrbWork o = orb_work(orb, wk, ns);
  const int good = o.flag[0];
  const int64_t q0 = (int64_t)blockIdx.x * 32;       // knots q0 + 1 .. q0 + 32
  const int s0 = (int)(q0 / K);
  if (s0 >= good) return;
  const int nsg = K >= 32 ? 1 : (int)((nk - q0 < 32 ? nk - q0 : 32) / K);
  for (int g = 0; g < nsg && s0 + g < good; ++g) {
    const double* src = reinterpret_cast<const double*>(o.work + (int64_t)(s0 + g) * 1280);
    for (int t = lane; t < 160; t += 32) f5s[g * kRateStride + t] = src[t];
  }
  __syncwarp();
  const int64_t kq = q0 + lane;                      // knot kq + 1
  const int i = (int)(kq / K), q = (int)(kq - (int64_t)i * K) + 1;
  const WalkerC& c = wcs[wk];
  const OrbSrc s = orb_src(c, pn);
  Knot* kn = knots + wk * (nk + 1);
  double r[5];
  if (kq < nk && i < good) {
    OrbState y = load_start(o, i);
    knot_state(y, f5s + (i - s0) * kRateStride, qk_g + (size_t)q * (128 / K) * 32,
               (double)seg * dt * (back ? -1.0 : 1.0));
    if (!state_finite(y) || (!back && plunged(y.v_hi, y.e_hi))) {
      atomicMin(&o.flag[1], i);
      atomicMin(&o.flag[6], (int)kq + 1);
    } else {
      const int64_t k = back ? nk - 1 - kq : kq + 1;
      ak_rhs_v(s, y.v_hi, y.e_hi, r[0], r[1], r[2], r[3], r[4]);
      write_knot(kn, k, y, r, c, cs, doppler);
    }
  }
  if (blockIdx.x == 0 && lane == 0) {
    const OrbState y = load_start(o, 0);
    const int64_t k = back ? nk : 0;
    ak_rhs_v(s, y.v_hi, y.e_hi, r[0], r[1], r[2], r[3], r[4]);
    write_knot(kn, k, y, r, c, cs, doppler);
  }
}

// Serial knot-step RK4 backwards over knots k0-1..k1 (state y at knot k0).
__device__ bool rk4_span_back(const OrbSrc& s, const WalkerC& c, OrbState& y, int64_t k0, int64_t k1, int ks,
                              double dt, const double2* cs, int doppler, Knot* kn) {
  const double h = -(double)ks * dt;
  double r[5];
  ak_rhs_v(s, y.v_hi, y.e_hi, r[0], r[1], r[2], r[3], r[4]);
  for (int64_t k = k0; k > k1; --k) {
    rk4_step(s, y, h, r);
    if (!state_finite(y)) return false;
    ak_rhs_v(s, y.v_hi, y.e_hi, r[0], r[1], r[2], r[3], r[4]);
    write_knot(kn, k - 1, y, r, c, cs, doppler);
  }
  return true;
}

__device__ __forceinline__ double bcast(double x, int src) { return __shfl_sync(0xffffffffu, x, src); }

__device__ __forceinline__ OrbState bcast_state(const OrbState& a, int src) {
  return OrbState{bcast(a.v_hi, src), bcast(a.v_lo, src), bcast(a.e_hi, src), bcast(a.e_lo, src),
                  bcast(a.p_hi, src), bcast(a.p_lo, src), bcast(a.g_hi, src), bcast(a.g_lo, src),
                  bcast(a.a_hi, src), bcast(a.a_lo, src)};
}

// One RK4 step of (v, e), rates (k1v, k1e) at the start.
__device__ __forceinline__ void rk4_ve(const OrbSrc& s, double& v, double& e, double h, double k1v, double k1e) {
  double k2v, k2e, k3v, k3e, k4v, k4e;
  ak_rate_ve(s, v + 0.5 * h * k1v, e + 0.5 * h * k1e, k2v, k2e);
  ak_rate_ve(s, v + 0.5 * h * k2v, e + 0.5 * h * k2e, k3v, k3e);
  ak_rate_ve(s, v + h * k3v, e + h * k3e, k4v, k4e);
  v += h / 6.0 * (k1v + 2.0 * (k2v + k3v) + k4v);
  e += h / 6.0 * (k1e + 2.0 * (k2e + k3e) + k4e);
}

// Samples from a knot inside the LSO (state y0) to the first sample past it
// (1..ks; the next knot is past it), by the whole warp: one RK4 step from the
// knot to each 32nd of the interval, then one from the last of these inside
// the LSO to each sample after it.  The steps are accurate where the state
// moves slowly, which is checked: two half steps have to give the same
// distance from the LSO to 1e-4 of what it changes by in one sample, else -1
// (the caller steps through the samples).  ~1000 FP64 instructions in
// sequence, 45 us; stepping sample by sample took ks times 12 us.
__device__ int plunge_sample(const OrbSrc& s, const OrbState& y0, int ks, double dt, int lane) {
  auto past = [](double v, double e) { return !(isfinite(v) && isfinite(e)) || plunged(v, e); };
  auto margin = [](double v, double e) { return v * v * (6.0 + 2.0 * e) - (1.0 - e * e); };
  const int sub = ks / 32;   // ks >= 64, a power of two
  const double v0 = y0.v_hi + y0.v_lo, e0 = y0.e_hi + y0.e_lo, h = (double)((lane + 1) * sub) * dt;
  double fv, fe;
  ak_rate_ve(s, v0, e0, fv, fe);
  double v = v0, e = e0, v2 = v0, e2 = e0, gv, ge;
  rk4_ve(s, v, e, h, fv, fe);
  rk4_ve(s, v2, e2, 0.5 * h, fv, fe);
  ak_rate_ve(s, v2, e2, gv, ge);
  rk4_ve(s, v2, e2, 0.5 * h, gv, ge);
  const double rate = fabs(2.0 * v0 * (6.0 + 2.0 * e0) * fv + 2.0 * (v0 * v0 + e0) * fe) * dt;
  if (!__all_sync(0xffffffffu, fabs(margin(v, e) - margin(v2, e2)) <= 1e-4 * rate)) return -1;
  const unsigned b = __ballot_sync(0xffffffffu, past(v, e));
  if (!b) return ks;
  const int m = __ffs(b) - 1;                       // the crossing lies in (m sub, (m + 1) sub]
  v = m ? bcast(v, m - 1) : v0;
  e = m ? bcast(e, m - 1) : e0;
  ak_rate_ve(s, v, e, fv, fe);
  rk4_ve(s, v, e, (double)(lane + 1) * dt, fv, fe);
  const unsigned c = __ballot_sync(0xffffffffu, lane < sub && past(v, e));
  return m * sub + (c ? __ffs(c) : sub);
}

// The rest of a walker's orbit from its first segment that the parallel
// solution does not cover (none for most walkers: then this only writes the
// status), one warp per walker.  A solved segment that passes the LSO at a
// knot: the plunge sample (plunge_sample), the knots being there already.
// Otherwise in sequence: per segment FP64 Picard sweeps, the knots from the
// segment polynomial and the plunge sample as in a solved segment; where the
// sweeps do not settle, or the plunge moves too fast for that, knot-step RK4
// by lane 0, which also locates the plunge sample.  In backward mode no plunge check applies; an orbit that
// turns non-finite gives a zero waveform and ST_NONFINITE.
__global__ void __launch_bounds__(32) k1f_tail(WalkerC* __restrict__ wcs, int64_t n, double dt,
                                               const double2* __restrict__ cs, int ks,
                                               int pn, int back, int doppler, const double* __restrict__ qn_g,
                                               const double* __restrict__ qk_g, char* __restrict__ orb,
                                               Knot* __restrict__ knots) {
  __shared__ double f[5 * 32];
  const int lane = threadIdx.x;
  const int64_t wk = blockIdx.x;
  const int64_t seg = mcpi_segment(n, ks), ns = n / seg, nk = n / ks;
  const int K = (int)(seg / ks);
  const OrbWork o = orb_work(orb, wk, ns);
  const int g0 = min(o.flag[0], o.flag[1]);
  if (g0 >= ns) {
    if (lane == 0) wcs[wk].j_plunge = n;
    return;
  }
  const WalkerC& c = wcs[wk];
  const uint32_t st0 = c.status;
  Knot* kn = knots + wk * (nk + 1);
  if (st0 & ST_BADPARAM) {
    if (lane == 0) wcs[wk].j_plunge = 0;   // no sample and no knot is looked at
    return;
  }
  const OrbSrc s = orb_src(c, pn);
  const double H = (double)seg * dt * (back ? -1.0 : 1.0);
  const double taui = 0.5 * (1.0 - cospi((double)lane / 31.0));
  OrbState y = load_start(o, g0);   // identical in every lane
  int64_t jp = n;
  uint32_t st = 0;
  bool fail = false;                // backward: the orbit turned non-finite
  const int64_t kstart = back ? nk - (int64_t)g0 * K : (int64_t)g0 * K;
  int64_t last = kstart;            // forward: last knot written
  bool done = false;
  // The plunge sample where knot q of the segment that starts at knot kb (state
  // ys, node rates f5) is its first past the LSO; the knots before it are there
  // already.  false: not found this way.
  auto plunge_in = [&](const OrbState& ys, const double* f5, int64_t kb, int q) {
    OrbState ym = ys, yq = ys;      // knots q - 1 and q
    if (q > 1) knot_state(ym, f5, qk_g + (size_t)(q - 1) * (128 / K) * 32, H);
    knot_state(yq, f5, qk_g + (size_t)q * (128 / K) * 32, H);
    const int d = state_finite(yq) ? plunge_sample(s, ym, ks, dt, lane) : -1;
    if (d <= 0) return false;
    last = kb + q;
    jp = (last - 1) * ks + d;
    if (jp < n) st |= ST_PLUNGE;
    else jp = n;
    double r[5];
    ak_rhs_v(s, yq.v_hi, yq.e_hi, r[0], r[1], r[2], r[3], r[4]);
    if (lane == 0) write_knot(kn, last, yq, r, c, cs, doppler);
    return true;
  };
  if (!back && g0 < o.flag[0])      // solved: the first knot past the LSO, counted from the segment's start
    done = plunge_in(y, reinterpret_cast<const double*>(o.work + (int64_t)g0 * 1280), kstart, o.flag[6] - g0 * K);
  if (done) {
  } else if (back && !state_finite(y)) {
    fail = true;
  } else {
    double r[5];
    ak_rhs_v(s, y.v_hi, y.e_hi, r[0], r[1], r[2], r[3], r[4]);
    if (lane == 0) write_knot(kn, kstart, y, r, c, cs, doppler);
    if (!back && plunged(y.v_hi, y.e_hi)) {
      jp = kstart * ks;
      st |= ST_PLUNGE;
    }
  }
  for (int64_t g = g0; g < ns && jp == n && !fail && !done; ++g) {
    const OrbState ys = y;          // segment start
    const int64_t kb = back ? nk - g * (int64_t)K : g * (int64_t)K;   // its knot
    double fv, fe;
    ak_rate_ve(s, y.v_hi, y.e_hi, fv, fe);
    double v = y.v_hi + (y.v_lo + H * taui * fv), e = y.e_hi + (y.e_lo + H * taui * fe);
    bool serial = true;
    for (int it = 0; it < 30; ++it) {
      ak_rate_ve(s, v, e, fv, fe);
      __syncwarp();
      f[lane] = fv;
      f[32 + lane] = fe;
      __syncwarp();
      double sv = 0.0, se = 0.0;
#pragma unroll 8
      for (int j = 0; j < 32; ++j) {
        const double q = qn_g[j * 32 + lane];
        sv = fma(q, f[j], sv);
        se = fma(q, f[32 + j], se);
      }
      const double vn = y.v_hi + (y.v_lo + H * sv);
      const double en = y.e_hi + (y.e_lo + H * se);
      // settled to within about two ulps (iterates can cycle at rounding level)
      const bool conv = fabs(vn - v) <= 4e-16 * fabs(y.v_hi) && fabs(en - e) <= 2e-16;
      v = vn;
      e = en;
      const bool ok = isfinite(v) && isfinite(e);
      if (__all_sync(0xffffffffu, conv || !ok)) {
        serial = !__all_sync(0xffffffffu, conv && ok);
        break;
      }
    }
    if (!serial) {
      double r[5];
      ak_rhs_v(s, v, e, r[0], r[1], r[2], r[3], r[4]);
      __syncwarp();
#pragma unroll
      for (int q = 0; q < 5; ++q) f[q * 32 + lane] = r[q];
      __syncwarp();
      int qbad = 0;                  // first knot past the LSO or not finite
      for (int q0 = 1; q0 <= K; q0 += 32) {
        const int q = q0 + lane;
        bool bad = false;
        OrbState yk = ys;
        if (q <= K) {
          knot_state(yk, f, qk_g + (size_t)q * (128 / K) * 32, H);
          bad = !state_finite(yk) || (!back && plunged(yk.v_hi, yk.e_hi));
          if (!bad) {
            const int64_t k = back ? kb - q : kb + q;
            double rk[5];
            ak_rhs_v(s, yk.v_hi, yk.e_hi, rk[0], rk[1], rk[2], rk[3], rk[4]);
            write_knot(kn, k, yk, rk, c, cs, doppler);
          }
        }
        const unsigned b = __ballot_sync(0xffffffffu, bad);
        if (b && !qbad) qbad = q0 + __ffs(b) - 1;
        if (K - q0 < 32) y = bcast_state(yk, K - q0);   // the end state, every lane's next start
      }
      if (qbad) {
        if (!back && plunge_in(ys, f, kb, qbad)) {
          done = true;
          break;
        }
        serial = true;
      }
    }
    if (serial) {
      // lane 0 redoes the segment with knot-step RK4 from the segment start;
      // its knots replace any written above
      __syncwarp();
      int valid = 1;
      y = ys;
      if (lane == 0) {
        double r[5];
        ak_rhs_v(s, y.v_hi, y.e_hi, r[0], r[1], r[2], r[3], r[4]);
        write_knot(kn, kb, y, r, c, cs, doppler);
        valid = back ? rk4_span_back(s, c, y, kb, kb - K, ks, dt, cs, doppler, kn)
                     : rk4_span(s, c, y, kb, kb + K, ks, dt, cs, doppler, n, kn, jp, st, last);
      }
      valid = __shfl_sync(0xffffffffu, valid, 0);
      jp = __shfl_sync(0xffffffffu, jp, 0);
      st = __shfl_sync(0xffffffffu, st, 0);
      last = __shfl_sync(0xffffffffu, last, 0);
      y = bcast_state(y, 0);
      if (back) fail = !valid;
      if (!valid) break;
    }
    last = kb + K;
  }
  __syncwarp();
  // forward: knots past a plunge repeat the last one written, up to the end of
  // the 4096 samples that the waveform kernels treat together (the samples
  // after the plunge are zeroed, whole segments of them without the knots)
  const int64_t kend = min(nk, last + 4096 / ks);
  if (!back)
    for (int64_t q = last + 1 + lane; q <= kend; q += 32) kn[q] = kn[last];
  if (lane == 0) {
    wcs[wk].j_plunge = back ? (fail ? 0 : n) : jp;
    wcs[wk].status = st0 | st | (fail ? (uint32_t)ST_NONFINITE : 0u);
  }
}

size_t orbit_bytes(int64_t n, int ks) { return orb_walker_bytes(n / mcpi_segment(n, ks)); }

int launch_orbit(WalkerC* wc, int w, int64_t n, double dt, const double2* cs, const OptsN& o, Knot* knots,
                 const double* mcpi_tab, char* orb, int64_t fit, cudaStream_t s) {
  if (w <= 0) return 0;
  const int64_t seg = mcpi_segment(n, o.ks), ns = n / seg, nk = n / o.ks;
  const int K = (int)(seg / o.ks), back = o.mode == 1, pn = o.pn_terms;
  const double* qn = mcpi_tab;
  const double* qk = mcpi_tab + 32 * 32;
  const int nsg = K >= 32 ? 1 : (int)((nk < 32 ? nk : 32) / K);
  int launches = 0;
  // walkers on grid y of the segment kernels: at most kMaxGridY per launch, and
  // no more than the solver state holds
  const int step = (int)(fit < 1 ? 1 : fit < kMaxGridY ? fit : kMaxGridY);
  for (int w0 = 0; w0 < w; w0 += step) {
    const int ww = w - w0 < step ? w - w0 : step;
    WalkerC* c = wc + w0;
    Knot* kn = knots + (int64_t)w0 * (nk + 1);
    const dim3 ge((unsigned)((ns + kEvalWarps - 1) / kEvalWarps), (unsigned)ww);
    const dim3 gk((unsigned)((nk + 31) / 32), (unsigned)ww);
    k1a_coarse<<<ww, 32, 0, s>>>(c, n, dt, o.ks, pn, back, qn, orb);
    k1b_eval<0><<<ge, 32 * kEvalWarps, 0, s>>>(c, n, dt, o.ks, pn, back, qn, orb);
    k1b_eval<1><<<ge, 32 * kEvalWarps, 0, s>>>(c, n, dt, o.ks, pn, back, qn, orb);
    k1b_eval<2><<<ge, 32 * kEvalWarps, 0, s>>>(c, n, dt, o.ks, pn, back, qn, orb);
    k1b_eval<3><<<ge, 32 * kEvalWarps, 0, s>>>(c, n, dt, o.ks, pn, back, qn, orb);
    k1c_final<<<ge, 32 * kEvalWarps, 0, s>>>(c, n, dt, o.ks, pn, back, qn, orb);
    k1d_starts<<<ww, 32, (size_t)ns * 40, s>>>(n, o.ks, orb);
    k1e_knots<<<gk, 32, (size_t)nsg * kRateStride * 8, s>>>(c, n, dt, cs, o.ks, pn, back, o.doppler, qk, orb, kn);
    k1f_tail<<<ww, 32, 0, s>>>(c, n, dt, cs, o.ks, pn, back, o.doppler, qn, qk, orb, kn);
    launches += 9;
  }
  return launches;
}

}  // namespace emri
