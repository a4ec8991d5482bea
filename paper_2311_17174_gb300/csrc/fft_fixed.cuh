// fft_fixed.cuh -- the FP64 transforms of 256 to 4096 points in 64-bit fixed
// point (fx64.cuh says why: an FP64 instruction costs ~17 integer multiply-
// adds of 32 bits here).  Included by k_fft.cu.
//
// N = 2^LG points of NB adjacent transforms by NB T threads, T = N/8, eight
// points each in registers: radix-8 Stockham stages, the last one radix 4 or
// 2, exchanged through shared memory.  The points come and go in double.
//
// Scaling: L = sum |x_j| (from above) bounds every intermediate value and
// output of the transform (each is a sum of inputs times unit phases), so with
// L 2^k < 2^62 nothing overflows.  For 1024 points and more that leaves too few
// bits to the inputs (L ~ N |x|): the first two radix-8 stages, whose values are
// at most 64 max |x_j|, then run at a finer scale of their own, and the second
// one rounds to the scale of L.  RMS error, 2^16 to 2^22 points of noise or
// signal: 0.7e-16 to 1.8e-16 relative, against 2.8e-16 to 3.4e-16 in double.
// 128 walkers x 2^21 (passes of 1024 and 2048 points): pass 1 17.6 -> 3.9 ms,
// pass 2 with the inner products 23.2 -> 4.3 ms; 23 transforms of 2^19 points
// 1.49 -> 0.39 ms.
// Transforms that hold NaN, infinities, or numbers outside [1e-30, 1e30] in
// sum take the FP64 Stockham form (their CTA does).
#pragma once

namespace fxfft {

using fx::i64;
using fx::Op;
using fx::Sum;
using fx::wide;

// exp(-2 pi i r k / (8 NS)), r = 1..7, k < NS at kBase(NS) + (r - 1) NS + k for
// NS = 8, 64, 512 (radix-8 stages; radix 4 reads r = 2, 4, 6 and radix 2 r = 4
// of the same NS), then exp(-2 pi i m / 4096) and exp(-2 pi i m / 2^22); each
// (cos.h, cos.l, sin.h, sin.l), Q62 in balanced halves.
constexpr int kStageLen = 7 * (8 + 64 + 512);
__host__ __device__ constexpr int kBase(int ns) { return ns - 8; }   // 7 (8 + ... + NS/8)
__device__ int4 g_stage[kStageLen];
__device__ int4 g_ta[4096];
__device__ int4 g_tb[1024];
__device__ fx::Trig g_trig[fx::kTrigLen];   // exp(2 pi i k / 1024), Q62

FX_HD int4 pack(i64 c, i64 s) {
  const Op a = fx::bal(c), b = fx::bal(s);
  return make_int4(a.h, a.l, b.h, b.l);
}

// Fills the tables of the current device on stream s, which nothing else waits
// for, from long double values kept by the process (a second context's upload
// rewrites them unchanged).
static bool upload_tables(cudaStream_t s) {
  static const std::vector<int4> host = [] {
    std::vector<int4> t;
    auto put = [&](long double turns) {
      const long double x = -2.0L * 3.141592653589793238462643383279502884L * turns;
      t.push_back(pack(llrintl(cosl(x) * 0x1p62L), llrintl(sinl(x) * 0x1p62L)));
    };
    for (int ns = 8; ns <= 512; ns *= 8)
      for (int r = 1; r < 8; ++r)
        for (int k = 0; k < ns; ++k) put((long double)(r * k) / (8 * ns));
    for (int i = 0; i < 4096; ++i) put((long double)i / 4096);
    for (int i = 0; i < 1024; ++i) put((long double)i / 4194304);
    return t;
  }();
  static const std::vector<fx::Trig> trig = [] {
    std::vector<fx::Trig> t(fx::kTrigLen);
    for (int k = 0; k < fx::kTrigLen; ++k) {
      const long double x = 2.0L * 3.141592653589793238462643383279502884L * k / fx::kTrigLen;
      t[k] = fx::Trig{llrintl(cosl(x) * 0x1p62L), llrintl(sinl(x) * 0x1p62L)};
    }
    return t;
  }();
  const auto put = [s](const auto& symbol, const void* src) {
    return cudaMemcpyToSymbolAsync(symbol, src, sizeof(symbol), 0, cudaMemcpyHostToDevice, s) == cudaSuccess;
  };
  return put(g_trig, trig.data()) && put(g_stage, host.data()) && put(g_ta, host.data() + kStageLen) &&
         put(g_tb, host.data() + kStageLen + 4096);
}

struct Z {
  i64 x, y;
};

FX_HD Z add(Z a, Z b) { return Z{a.x + b.x, a.y + b.y}; }
FX_HD Z sub(Z a, Z b) { return Z{a.x - b.x, a.y - b.y}; }

// A sum of products in two accumulators, high*high and cross terms (2^32 below
// it).
struct Acc {
  i64 h, c;
  FX_HD void add(Op a, Op b) {
    h = wide(a.h, b.h, h);
    c = wide(a.h, b.l, c);
    c = wide(a.l, b.h, c);
  }
};
constexpr i64 kHalf4 = (i64)1 << 29;   // half of the last bit of get4
// x 2^-62 (Q62 factor: the unit stays), rounded to the last bit
FX_HD i64 get4(const Acc& s) { return (s.h << 2) + (s.c >> 30); }

// a w, w = (cos.h, cos.l, sin.h, sin.l) in Q62, |a| < 2^62: error ~0.55 of the
// last bit (rms; low*low 0.47, the rounding 0.29).  With op()'s halves it was
// ~1.7, the larger part of a transform's error.
FX_HD Z cmul(Z a, int4 w) {
  const Op ax = fx::bal(a.x), ay = fx::bal(a.y), c{w.x, w.y}, s{w.z, w.w};
  Acc re{0, kHalf4}, im{0, kHalf4}, t{0, 0};
  re.add(ax, c);
  t.add(ay, s);
  re.h -= t.h;
  re.c -= t.c;
  im.add(ax, s);
  im.add(ay, c);
  return Z{get4(re), get4(im)};
}

// x sqrt(1/2) = x - x (1 - sqrt(1/2)), the factor 0.29289... in Q64
FX_HD i64 mul_h(i64 x) {
  Acc s{0, (i64)1 << 31};
  s.add(fx::bal(x), Op{0x4AFB0CCC, 0x06219B7C});
  return x - (s.h + (s.c >> 32));
}

FX_HD void dft4(Z& a0, Z& a1, Z& a2, Z& a3) {
  const Z s0 = add(a0, a2), s1 = sub(a0, a2), s2 = add(a1, a3), d = sub(a1, a3);
  a0 = add(s0, s2);
  a2 = sub(s0, s2);
  a1 = Z{s1.x + d.y, s1.y - d.x};   // s1 - i d
  a3 = Z{s1.x - d.y, s1.y + d.x};
}

// X_q = sum_r a_r exp(-2 pi i q r / 8), in place
FX_HD void dft8(Z (&a)[8]) {
  Z b0 = add(a[0], a[4]), b1 = add(a[1], a[5]), b2 = add(a[2], a[6]), b3 = add(a[3], a[7]);
  const Z d0 = sub(a[0], a[4]), d1 = sub(a[1], a[5]), d2 = sub(a[2], a[6]), d3 = sub(a[3], a[7]);
  const Z c1{mul_h(d1.x + d1.y), mul_h(d1.y - d1.x)};
  const Z c3{mul_h(d3.y - d3.x), mul_h(-(d3.x + d3.y))};
  dft4(b0, b1, b2, b3);
  const Z s0{d0.x + d2.y, d0.y - d2.x}, s1{d0.x - d2.y, d0.y + d2.x};   // d0 -+ i d2
  const Z s2 = add(c1, c3), dd = sub(c1, c3);
  a[0] = b0; a[2] = b1; a[4] = b2; a[6] = b3;
  a[1] = add(s0, s2);
  a[5] = sub(s0, s2);
  a[3] = Z{s1.x + dd.y, s1.y - dd.x};
  a[7] = Z{s1.x - dd.y, s1.y + dd.x};
}

// |v| as a float (truncated; 0 below 2^-126, infinity above 2^128 and for NaN)
FX_HD float abs_float(double v) {
#ifdef __CUDA_ARCH__
  const int h = __double2hiint(v) & 0x7fffffff, l = __double2loint(v);
  const int e = min(max(h - (896 << 20), 0), 0x0ff00000);
  return __int_as_float((int)(((unsigned)e << 3) | ((unsigned)l >> 29)) & (e == 0x0ff00000 ? 0x7f800000 : -1));
#else
  return (float)fabs(v);
#endif
}

// round(v 2^k), |v| 2^k < 2^62
FX_HD i64 to_fixed(double v, int k) {
#ifdef __CUDA_ARCH__
  const int h = __double2hiint(v);
  const fx::u64 b = (fx::u64)__double_as_longlong(v);
#else
  fx::u64 b;
  memcpy(&b, &v, 8);
  const int h = (int)(b >> 32);
#endif
  const int ex = (h >> 20) & 0x7ff;
  const fx::u64 m = ((b & 0xfffffffffffffULL) | 0x10000000000000ULL) << 10;   // 63 bits
  int sh = 1084 - k - ex;   // one bit kept for the rounding; >= 0
  if (sh > 63) sh = 63;
  const i64 r = (i64)(((m >> sh) + 1) >> 1);
  const i64 sg = (i64)(h >> 31);
  return (r ^ sg) - sg;
}

// v 2^-k (v = 0 stays 0; the result is a normal number)
__device__ __forceinline__ double from_fixed(i64 v, int k) {
  const double d = (double)v;
  return v == 0 ? 0.0 : __hiloint2double(__double2hiint(d) - (k << 20), __double2loint(d));
}

// v 2^-k for v = 0 or 2^32 <= v < 2^63, on the integer pipe (a conversion
// takes the FP64 pipe for 64 cycles): round to 53 bits, the leading bit carries
// into the exponent
__device__ __forceinline__ double from_fixed_pos(i64 v, int k) {
  const int lz = __clz(fx::hi(v));
  const fx::u64 m = (((fx::u64)v << (lz - 1)) + 0x200) >> 10;
  const double d = __longlong_as_double((long long)(m + ((fx::u64)(1085 - lz - k) << 52)));
  return v == 0 ? 0.0 : d;
}

template <int LG, int NB>
struct Cfg {
  static constexpr int N = 1 << LG, T = N / 8, kThreads = NB * T;
  static constexpr size_t kSmem = (size_t)NB * (N + N / 8) * 16;
  static_assert(LG >= 8 && LG <= 12, "256 to 4096 points");
};

// element i of transform c: one 16-byte column in eight is skipped, so that
// eight threads' accesses fall into different banks at every stage
template <int NB>
__device__ __forceinline__ int at(int i, int c) { return (i + (i >> 3)) * NB + c; }

// Exponent of a transform's values: 2^k from the inputs to the second stage,
// 2^(k - down) after it.
struct Scale {
  int k, down;
  __device__ __forceinline__ int out() const { return k - down; }
};
// From this length on the second stage changes the scale.
constexpr int kTwoScales = 10;

// v (point t + q T in slot q) -> bin t + q T in slot q.  xb: Cfg::kSmem bytes.
template <int LG, int NB, int NS>
__device__ __forceinline__ void stages(Z (&v)[8], longlong2* xb, int t, int c, int down) {
  constexpr int N = 1 << LG, T = N / 8;
  if constexpr (8 * NS <= N) {
    const int k = t & (NS - 1);
    if constexpr (NS > 1) {
#pragma unroll
      for (int q = 1; q < 8; ++q) v[q] = cmul(v[q], __ldg(g_stage + kBase(NS) + (q - 1) * NS + k));
    }
    dft8(v);
    if constexpr (NS == 8 && LG >= kTwoScales) {
      const i64 half = down ? (i64)1 << (down - 1) : 0;
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = Z{(v[q].x + half) >> down, (v[q].y + half) >> down};
    }
    if constexpr (8 * NS < N) {
      const int d = (t / NS) * NS * 8 + k;
      if constexpr (NS > 1) __syncthreads();   // the previous stage's reads
#pragma unroll
      for (int q = 0; q < 8; ++q) xb[at<NB>(d + q * NS, c)] = make_longlong2(v[q].x, v[q].y);
      __syncthreads();
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const longlong2 u = xb[at<NB>(t + q * T, c)];
        v[q] = Z{u.x, u.y};
      }
      stages<LG, NB, 8 * NS>(v, xb, t, c, down);
    }
  } else if constexpr (4 * NS == N) {   // butterflies t and t + T over v[0,2,4,6] and v[1,3,5,7]
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int4* w = g_stage + kBase(NS) + t + h * T;   // W_{4 NS}^{r k} = W_{8 NS}^{2 r k}
      Z a1 = cmul(v[h + 2], __ldg(w + NS)), a2 = cmul(v[h + 4], __ldg(w + 3 * NS)), a3 = cmul(v[h + 6], __ldg(w + 5 * NS));
      dft4(v[h], a1, a2, a3);
      v[h + 2] = a1;
      v[h + 4] = a2;
      v[h + 6] = a3;
    }
  } else {                              // 2 NS == N: butterflies t + i T over v[i], v[i + 4]
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const Z b = cmul(v[i + 4], __ldg(g_stage + kBase(NS) + 3 * NS + t + i * T)), a = v[i];
      v[i] = add(a, b);
      v[i + 4] = sub(a, b);
    }
  }
}

// Loads the thread's points p[q T gs] of its transform, finds the transform's
// exponents and converts.  Returns false, for the whole CTA, when a transform is
// outside the fixed-point range.  swap: exchange
// Re and Im (the inverse transform is the forward one of the exchanged parts).
template <int LG, int NB>
__device__ __forceinline__ bool load(const double2* p, int64_t step, bool swap, int c, Z (&v)[8], Scale& sc) {
  using F = Cfg<LG, NB>;
  constexpr int NW = F::kThreads / 32;
  __shared__ float red[NW][NB], redm[NW][NB];
  double2 u[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) u[q] = p[q * step];
  float L = 0.f, M = 0.f;
  unsigned any = 0;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    // |z| <= max + (sqrt(2) - 1) min of the parts' sizes
    const float a = abs_float(u[q].x), b = abs_float(u[q].y);
    const float r = fmaf(0.41422f, fminf(a, b), fmaxf(a, b));
    L += r;
    M = fmaxf(M, r);
    any |= (unsigned)__double2hiint(u[q].x) << 1 | (unsigned)__double2loint(u[q].x) |
           (unsigned)__double2hiint(u[q].y) << 1 | (unsigned)__double2loint(u[q].y);
  }
#pragma unroll
  for (int off = 16; off >= NB; off >>= 1) {
    L += __shfl_xor_sync(0xffffffffu, L, off);
    if (LG >= kTwoScales) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, off));
  }
  if ((threadIdx.x & 31) < NB) {
    red[threadIdx.x >> 5][c] = L;
    if (LG >= kTwoScales) redm[threadIdx.x >> 5][c] = M;
  }
  const int nonzero = __syncthreads_or(any != 0);   // also orders red
  L = 0.f;
#pragma unroll 8
  for (int w = 0; w < NW; ++w) {
    L += red[w][c];
    if (LG >= kTwoScales) M = fmaxf(M, redm[w][c]);
  }
  const bool bad = !(L < 1e30f) || (L < 1e-30f && nonzero);
  // NB transforms share the decision (each thread sees its own transform's L)
  if (__syncthreads_or(bad)) return false;
  L = fmaxf(L * 1.001f, 1e-30f);
  sc.k = 61 - ilogbf(LG >= kTwoScales ? fminf(L, fmaxf(64.064f * M, 1e-30f)) : L);
  sc.down = sc.k - (61 - ilogbf(L));
  const int k = sc.k;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const i64 a = to_fixed(u[q].x, k), b = to_fixed(u[q].y, k);
    v[q] = swap ? Z{b, a} : Z{a, b};
  }
  return true;
}

// The CTA's transforms in double in the same shared memory (element i of
// transform c at i NB + c), for the inputs load() refuses.
template <int LG, int NB>
__device__ __noinline__ void fallback(const double2* p, int64_t step, double2* buf, int t, int c, int sign,
                                      const double2* __restrict__ tc) {
  using F = Cfg<LG, NB>;
#pragma unroll 1
  for (int q = 0; q < 8; ++q) buf[(t + q * F::T) * NB + c] = p[q * step];
  __syncthreads();
  smem_fft<double2, LG, NB, F::kThreads>(buf, sign, tc);
}

// exp(-2 pi i m / 2^22), m < 2^22
__device__ __forceinline__ Z unit(int4 w) { return Z{fx::value(Op{w.x, w.y}), fx::value(Op{w.z, w.w})}; }
__device__ __forceinline__ Z twiddle(uint32_t m) { return cmul(unit(__ldg(g_ta + (m >> 10))), __ldg(g_tb + (m & 1023u))); }
__device__ __forceinline__ int4 pack(Z w) { return pack(w.x, w.y); }

__device__ __forceinline__ double2 out2(Z v, int k, bool swap) {
  const double a = from_fixed(v.x, k), b = from_fixed(v.y, k);
  return swap ? make_double2(b, a) : make_double2(a, b);
}

// Pass 1: NB adjacent columns j1, with the inter-pass twiddle W_n^{j1 k2} on
// the way out: W^{j1 t} of the thread times W^{j1 T q}, one per column and slot.
// 256 threads a CTA (NB = 2, 4, 8 columns of 1024, 512, 256 points), three CTAs
// per SM at 80 registers: one CTA's loads and stores run beside the others'
// stages.
template <int LG, int NB>
__global__ void __launch_bounds__(Cfg<LG, NB>::kThreads, 3)
    k3_pass1_fixed(const double2* zin, double2* zout, int64_t n, int n1, int sign, int shift22, const double2* __restrict__ ta,
                   const double2* __restrict__ tb, const double2* __restrict__ tc) {
  using F = Cfg<LG, NB>;
  extern __shared__ __align__(16) unsigned char smraw[];
  longlong2* xb = reinterpret_cast<longlong2*>(smraw);
  __shared__ int4 sq[8][NB];
  const int c = threadIdx.x % NB, t = threadIdx.x / NB;
  const int j1 = blockIdx.x * NB + c;
  const double2* zw = zin + (int64_t)blockIdx.y * n + j1;
  double2* zo = zout + (int64_t)blockIdx.y * n + j1;
  const bool swap = sign > 0;
  if (threadIdx.x < 8 * NB) sq[t][c] = pack(twiddle((uint32_t)(j1 * F::T * t) << shift22));   // slot t
  Z v[8];
  Scale sc;
  if (!load<LG, NB>(zw + (int64_t)t * n1, (int64_t)F::T * n1, swap, c, v, sc)) {
    double2* buf = reinterpret_cast<double2*>(smraw);
    fallback<LG, NB>(zw + (int64_t)t * n1, (int64_t)F::T * n1, buf, t, c, sign, tc);
#pragma unroll 1
    for (int q = 0; q < 8; ++q) {
      const int k2 = t + q * F::T;
      zo[(int64_t)n1 * k2] =
          ::emri::cmul(buf[k2 * NB + c], twiddle22(ta, tb, (uint32_t)(j1 * k2) << shift22, sign));
    }
    return;
  }
  stages<LG, NB, 1>(v, xb, t, c, sc.down);
  const Z w0 = twiddle((uint32_t)(j1 * t) << shift22);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const Z w = q == 0 ? w0 : cmul(w0, sq[q][c]);
    zo[(int64_t)n1 * (t + q * F::T)] = out2(cmul(v[q], pack(w)), sc.out(), swap);
  }
}

// Pass 2 to natural order, NB adjacent rows k2 (whole 32-byte sectors of the
// output for NB = 2).
template <int LG, int NB>
__global__ void __launch_bounds__(Cfg<LG, NB>::kThreads, Cfg<LG, NB>::kThreads > 256 ? 1 : 2)
    k4_pass2_store_fixed(const double2* __restrict__ y, double2* __restrict__ out, int64_t n, int n2, int sign,
                         const double2* __restrict__ tc) {
  using F = Cfg<LG, NB>;
  extern __shared__ __align__(16) unsigned char smraw[];
  const int c = threadIdx.x % NB, t = threadIdx.x / NB;
  const int k2 = blockIdx.x * NB + c;
  const double2* row = y + (int64_t)blockIdx.y * n + (int64_t)F::N * k2 + t;
  double2* o = out + (int64_t)blockIdx.y * n + k2;
  const bool swap = sign > 0;
  Z v[8];
  Scale sc;
  if (!load<LG, NB>(row, F::T, swap, c, v, sc)) {
    double2* buf = reinterpret_cast<double2*>(smraw);
    fallback<LG, NB>(row, F::T, buf, t, c, sign, tc);
#pragma unroll 1
    for (int q = 0; q < 8; ++q) o[(int64_t)n2 * (t + q * F::T)] = buf[(t + q * F::T) * NB + c];
    return;
  }
  stages<LG, NB, 1>(v, reinterpret_cast<longlong2*>(smraw), t, c, sc.down);
#pragma unroll
  for (int q = 0; q < 8; ++q) o[(int64_t)n2 * (t + q * F::T)] = out2(v[q], sc.out(), swap);
}

// Pass 2 of row k2 fused with the inner products.  dtab: the walker's delay
// factors as (cos.h, cos.l, sin.h, sin.l), Q62 in balanced halves.
//
// The bin, its product with the delay factor and its square modulus stay in
// fixed point, normalised per bin so that small bins keep 60 bits; three
// conversions and five FP64 FMAs per bin remain (twelve in double), and run
// beside the integer work.  FD: the phase's sine and cosine in fixed point too,
// the amplitude's exponential in double (32 walkers x 2^18: 1.64 -> 0.54 ms).
template <int LG, bool FD>
__global__ void __launch_bounds__(Cfg<LG, 1>::kThreads, Cfg<LG, 1>::kThreads > 256 ? 1 : 768 / Cfg<LG, 1>::kThreads)
    k4_pass2_ip_fixed(const double2* __restrict__ y, int64_t n, int n2, const double2* __restrict__ tc,
                      const WalkerC* __restrict__ wcs, const int4* __restrict__ dtab, const double2* __restrict__ rtab,
                      const double2* __restrict__ dperm, const double* __restrict__ wperm,
                      double2* __restrict__ partial, const FdW* __restrict__ fdw) {
  using F = Cfg<LG, 1>;
  extern __shared__ __align__(16) unsigned char smraw[];
  double2* buf = reinterpret_cast<double2*>(smraw);
  const int t = threadIdx.x;
  const int k2 = blockIdx.x, wk = blockIdx.y;
  const int64_t base = (int64_t)k2 * F::N;
  const double2* row = y + (int64_t)wk * n + base + t;
  const double2* ds = dperm + base;
  const double* ws = wperm + base;
  const int4* ts = dtab + (int64_t)wk * F::N;
  Z v[8];
  __shared__ FdRec<double> fd;
  if (FD && t == 0) fd.set(fdw[wk]);   // (read after load()'s barriers)
  Scale sc{0, 0};
  const bool fixed = load<LG, 1>(row, F::T, false, 0, v, sc);
  if (fixed) stages<LG, 1, 1>(v, reinterpret_cast<longlong2*>(smraw), t, 0, sc.down);
  else fallback<LG, 1>(row, F::T, buf, t, 0, -1, tc);
  const int k = sc.out();
  const double2 cnv = make_double2(wcs[wk].cn_re, wcs[wk].cn_im);
  double zr = 0.0, zi = 0.0, shh = 0.0;
  if (fixed) {
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      const int k1 = t + q * F::T;
      const int4 w = __ldg(ts + k1);
      const double2 G = __ldg(ds + k1);
      double wv = __ldg(ws + k1);
      const fx::u64 m = (fx::u64)(v[q].x ^ (v[q].x >> 63)) | (fx::u64)(v[q].y ^ (v[q].y >> 63));
      const int sh = max(__clzll((long long)m) - 3, 0);
      const Z H{v[q].x << sh, v[q].y << sh};
      Sum h2;
      h2.add(fx::op(H.x), fx::op(H.x));
      h2.add(fx::op(H.y), fx::op(H.y));
      Z Pi = cmul(H, w);
      double A = 1.0;
      if (FD) {
        const bool neg = q > 4 || (q == 4 && (t > 0 || k2 > 0));
        const uint32_t kk = (uint32_t)k2 + (uint32_t)n2 * (uint32_t)k1, ak = neg ? (uint32_t)n - kk : kk;
        if (fd.qt > 0) {
          const fx::Trig f = fx::sincos_cycles(0 - fd_phase(fd, ak, neg), g_trig);
          Pi = cmul(Pi, pack(f.c, f.s));
        }
        A = fd_amp(fd, ak);
        wv *= A * A;
      }
      double2 P = make_double2(from_fixed(Pi.x, sh), from_fixed(Pi.y, sh));
      // the one negative bin of this column not in the table: k1 = N/2 = 4 T
      if (q == 4 && t == 0 && k2 > 0) P = ::emri::cmul(P, cnv);
      if (FD) P = make_double2(A * P.x, A * P.y);
      zr = fma(-G.y, P.y, fma(G.x, P.x, zr));
      zi = fma(G.y, P.x, fma(G.x, P.y, zi));
      shh = fma(wv, from_fixed_pos(h2.get(), 2 * sh), shh);
    }
  } else {
#pragma unroll 1
    for (int q = 0; q < 8; ++q) {
      const int k1 = t + q * F::T;
      const double2 H = buf[k1];
      const int4 w = __ldg(ts + k1);
      const double2 G = __ldg(ds + k1);
      double2 P = ::emri::cmul(H, out2(unit(w), 62, false));
      if (2 * k1 == F::N && k2 > 0) P = ::emri::cmul(P, cnv);
      double A2 = 1.0;
      if (FD) {
        const bool neg = 2 * k1 > F::N || (2 * k1 == F::N && k2 > 0);
        const uint32_t kk = (uint32_t)k2 + (uint32_t)n2 * (uint32_t)k1;
        double cf, sf;
        const double A = fd_factor<double>(fd, neg ? (uint32_t)n - kk : kk, neg, cf, sf);
        P = ::emri::cmul(P, make_double2(A * cf, A * sf));
        A2 = A * A;
      }
      zr = fma(-G.y, P.y, fma(G.x, P.x, zr));
      zi = fma(G.y, P.x, fma(G.x, P.y, zi));
      shh += __ldg(ws + k1) * (H.x * H.x + H.y * H.y) * A2;
    }
  }
  // fixed-order sum: every thread's pair to shared memory, then one warp
  // (2 T/32 + 10 FP64 instructions; a shuffle tree in every warp takes 10 T/32)
  const double2 a = rtab[(int64_t)wk * n2 + k2];   // exp(-2 pi i frac(k2 r))
  __syncthreads();
  buf[t] = make_double2(a.x * zr - a.y * zi, shh);
  __syncthreads();
  if (t < 32) {
    double2 r = buf[t];
#pragma unroll
    for (int i = t + 32; i < F::T; i += 32) {
      const double2 b = buf[i];
      r.x += b.x;
      r.y += b.y;
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      r.x += __shfl_xor_sync(0xffffffffu, r.x, off);
      r.y += __shfl_xor_sync(0xffffffffu, r.y, off);
    }
    if (fixed) {   // units of the bins: H 2^k, |H|^2 2^(2 k - 64)
      r.x *= __longlong_as_double((long long)(1023 - k) << 52);
      r.y *= __longlong_as_double((long long)(1087 - 2 * k) << 52);
    }
    if (t == 0) partial[(int64_t)wk * n2 + k2] = r;
  }
}

}  // namespace fxfft
