// emri_internal.h -- host-side declarations shared by the libemri
// translation units (kernel launchers and normalised options).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace emri {

struct WalkerC;
struct Knot;
struct FdW;

// Largest grid y of a launch: the batched kernels put walkers (or
// sequences) on grid y, so a call processes at most this many per launch.
constexpr int kMaxGridY = 65535;

// Options after defaults and validation.
struct OptsN {
  int precision;   // 0 FP64, 1 mixed
  int n_max;
  int doppler;
  int pn_terms;
  int mode;        // 0 forward, 1 backward from LSO
  int ks;          // knot spacing (samples)
  double n_xi, omega_m, h0;
};

// FFT split of n = n1 * n2 (n2 = column length, n1 = row length).
struct FftPlan {
  int64_t n;
  int n1, n2;
  int log2n;
};
// n2 = 0: default split n2 = 2^min(10, log2(n)/2)
FftPlan make_fft_plan(int64_t n, int n2 = 0);

// Twiddle tables: ta[i] = exp(-2 pi i i/4096), i < 4096; tb[i] = exp(-2 pi i i/2^22), i < 1024.
struct Twiddles {
  double2* ta64;   // exp(-2 pi i k / 4096)
  double2* tb64;   // exp(-2 pi i k / 2^22), k < 1024
  float2* ta32;
  float2* tb32;
  double2* tc64;   // (cos, tan) of -2 pi k / 4096, |cos| >= 2^-60
  float2* tt32;    // stage twiddles: tt32[M/2 + k] = exp(-2 pi i k / M), M = 2..4096, k < M/2
};

void launch_twiddle_init(Twiddles t, cudaStream_t s);

// Bessel series tables: c[m * kBesselTerms + k] = (-1)^k m!/(k! (m+k)!),
// f[m] = 1/m!, m < kBesselOrders
constexpr int kBesselOrders = 35;
constexpr int kBesselTerms = 48;
struct BesselTab {
  double* c64;
  float* c32;
  double* f64;
  float* f32;
};
// fills the tables from the host (synchronous); 0 on success
int upload_bessel_tables(const BesselTab& t);
// the FP64 waveform kernel's exp(2 pi i k/512) table on the current device; 0 on success
int upload_exp512();

// the walkers' constants: all of them, all but the delay's (which only the
// delay tables and pass 2 read), or the delay's
enum class ProPart { kAll, kNoDelay, kDelay };
void launch_prologue(const double* theta, int64_t ld, int w, int64_t n, double dt, const OptsN& o,
                     const double* gl, WalkerC* out, cudaStream_t s, ProPart part = ProPart::kAll);
// (FP64 tab with n1 >= 256: (cos.h, cos.l, sin.h, sin.l) in Q62, balanced halves (fx64.cuh), four ints)
// tab[w][n1] = exp(-2 pi i frac(n2 k1 r)), rtab[w][n2] = exp(-2 pi i frac(k2 r))
void launch_delay_table(const WalkerC* wc, int w, int n1, int n2, bool fp32, void* tab, void* rtab, cudaStream_t s);
void launch_prologue_export(const WalkerC* wc, int w, double* out, cudaStream_t s);
// frequency-dependent propagation records fd[w] from theta and coef[qm+qt][ldc]
void launch_fdprop(const double* theta, int64_t ld, int w, int64_t n, double dt, const OptsN& o, int qm, int qt,
                   double fstar, const double* coef, int64_t ldc, FdW* fd, cudaStream_t s);

// orbit: knots[w][nk+1], nk = n / ks
// mcpi_tab: Chebyshev-Picard tables (qn then qk), required; cs: cos, sin of the
// LISA orbital phase at the knots (launch_lisa); orb: solver state of `fit`
// walkers, orbit_bytes(n, ks) each, 16-byte aligned, free again afterwards
// (more walkers than that take turns).  Returns the number of launches.
int launch_orbit(WalkerC* wc, int w, int64_t n, double dt, const double2* cs, const OptsN& o, Knot* knots,
                 const double* mcpi_tab, char* orb, int64_t fit, cudaStream_t s);
size_t orbit_bytes(int64_t n, int ks);

// Memory that only the orbit step uses: the LISA phase table at the knots,
// then the solver state.  It lies where the step's successors write the time
// series; one series of n samples holds the table and one walker's state.
struct OrbScratch {
  double2* cs;
  char* orb;
  int64_t fit;   // walkers whose state fits
  // in the `bytes` at p (alignment as the series': 8 bytes)
  OrbScratch(void* p, size_t bytes, int64_t n, int ks) {
    char* a = (char*)(((uintptr_t)p + 255) & ~(uintptr_t)255);
    const size_t tab = ((size_t)(n / ks + 1) * 16 + 255) & ~(size_t)255;
    cs = (double2*)a;
    orb = a + tab;
    fit = (int64_t)((bytes - (size_t)(orb - (char*)p)) / orbit_bytes(n, ks));
  }
};

// waveform: z[w][n] (double2 or float2); unit_scale multiplies by mu_s c (cm units)
// lisa: LISA orbital phase table (launch_lisa); ivs: mixed
// interval records [w][n/ks] (launch_intervals_mixed; unused for FP64)
void launch_wave(const Knot* knots, const WalkerC* wc, int w, int64_t n, double dt, double t0,
                 const OptsN& o, void* z, bool unit_scale, const BesselTab& bt, const double* lisa, const void* ivs,
                 cudaStream_t s);
void launch_intervals_mixed(const Knot* knots, int w, int64_t n, int ks, double dt, void* ivs, cudaStream_t s);
// cos, sin of the LISA orbital phase at the pattern-fit nodes of each
// 256-sample tile, tiles[n/256][8], and at the knots, knots[n/ks + 1]
inline size_t lisa_len(int64_t n) { return (size_t)(n / 256) * 8; }
void launch_lisa(int64_t n, int ks, double t0, double dt, double* tiles, double2* knots, cudaStream_t s);
constexpr size_t kIvMBytes = 104;

// FFT pass 1 (columns, with the inter-pass twiddle; out may be z); sign -1 forward, +1 inverse
void launch_fft_pass1(const void* z, void* out, int batch, const FftPlan& p, bool fp32, int sign, const Twiddles& t,
                      cudaStream_t s);
// FFT pass 2 to natural order into out (out-of-place)
void launch_fft_pass2_store(const void* y, void* out, int batch, const FftPlan& p, bool fp32, int sign,
                            const Twiddles& t, cudaStream_t s);
// FFT pass 2 fused with the weighted inner products; partial[w][n2] = (dh, hh)
void launch_fft_pass2_ip(const void* y, int w, const FftPlan& p, bool fp32, const Twiddles& t,
                         const WalkerC* wc, const void* delay_tab, const void* row_tab, const void* data_perm,
                         const void* wt_perm, double2* partial, cudaStream_t s, const FdW* fd = nullptr);
// per-walker fixed-order reduction of the partials and lnL
// dh_scale / hh_scale undo the dataset's FP32 scaling (1 for FP64)
void launch_finalize(const double2* partial, int n2, const WalkerC* wc, int w, double dh_scale, double hh_scale,
                     double* lnl, double* dh, double* hh, uint32_t* status, cudaStream_t s);
// shared-memory limits and fixed-point tables on the current device (the tables
// on stream s); false on failure
bool fft_setup(cudaStream_t s);

// dataset preparation: the weighted conjugate spectrum g = w conj(D) and
// the weights w in the pass-2 order (k2-major), plus FP32 copies scaled by
// d_scale w_scale and w_scale
void launch_dataset_permute(const double2* d_nat, const double* w_nat, const FftPlan& p, double2* g_perm,
                            double* w_perm, float2* g_perm32, float* w_perm32, double d_scale,
                            double w_scale, cudaStream_t s);
void launch_weights(const double* psd, int64_t n, double dt, double fmin, double fmax, double* w,
                    cudaStream_t s);
void launch_pack_time_series(const double* d2, int64_t n, double2* z, cudaStream_t s);
void launch_inner_dd(const double2* d, const double* w, int64_t n, double* out, cudaStream_t s);

}  // namespace emri
