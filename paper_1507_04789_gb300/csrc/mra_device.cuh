// mra_device.cuh -- device building blocks shared by the M-RA kernels.
//
// FP64 tile arithmetic for one CTA of NT threads: covariance tiles (Sec. 2.1,
// Eq. mat15), region boxes and knots (Sec. 2.2), a register-blocked tile
// product staged through shared memory, and in-shared-memory Cholesky and
// triangular inversion.  On GB300 the FP64 pipe retires 2 DFMA per clock per
// SM, so every routine here is written to keep DFMA lanes busy with useful
// work; shared-memory bandwidth is never the limit.
#pragma once
#include <cmath>
#include <cstring>
#include <cstdint>
#include <cuda_runtime.h>

namespace mra {

constexpr int NT = 256;          // threads per CTA (the kernels of the emulation engine: EM_NT, mra_emu.cuh);
                                 // helpers used by both take the count as NTH
constexpr int KC = 32;           // k-chunk of the staged tile product
constexpr int MAX_R_DEV = 64;    // largest r (knots per internal region)
constexpr double SQRT3 = 1.7320508075688772935;
constexpr double PI = 3.141592653589793238463;

// ---- error status (device) ------------------------------------------------
// status[0] = first error code, status[1] = level, status[2] = region
enum : int { ST_OK = 0, ST_NOT_PD = 4, ST_LIMIT = 6, ST_ARG = 1, ST_TIMEOUT = 7 };

__device__ __forceinline__ void flag_error(int* status, int code, int level, long region) {
  if (atomicCAS(status, 0, code) == 0) {
    status[1] = level;
    status[2] = (int)region;
  }
}

// ---- covariance function C0 (Sec. 2.1; Eq. mat15; nonstationary variance) --
struct Cov {
  double sigma2, kappa;
  int family;   // 0 exponential, 1 Matern-1.5, 2 Matern of smoothness nu
  int nonstat;
  double ik;    // 1 / kappa (set by make_cov)
  // family 2 (set by make_cov): nu, sqrt(2 nu), log of 2^(1-nu) / Gamma(nu) and
  // its derivative in nu, -log 2 - digamma(nu)
  double nu, snu, lcnu, dlcnu;
};

// digamma(x), x > 0, for the host: psi(x) = psi(x + k) - sum_{j<k} 1/(x + j) with
// x + k >= 8, then the asymptotic series of psi (Abramowitz & Stegun 6.3.18):
// log y - 1/(2y) - sum_{n>=1} B_2n / (2n y^2n), B_2..B_12 = 1/6, -1/30, 1/42,
// -1/30, 5/66, -691/2730 (truncation below 1e-17 at y >= 8).
inline double digamma_host(double x) {
  double acc = 0.0;
  while (x < 8.0) {
    acc -= 1.0 / x;
    x += 1.0;
  }
  const double y2 = 1.0 / (x * x);
  const double series = y2 * (1.0 / 12 - y2 * (1.0 / 120 - y2 * (1.0 / 252 - y2 * (1.0 / 240 - y2 * (1.0 / 132 -
                                                                                                   y2 * 691.0 / 32760)))));
  return acc + std::log(x) - 0.5 / x - series;
}

inline Cov make_cov(double sigma2, double kappa, int family, int nonstat, double nu = 0.0) {
  Cov c{sigma2, kappa, family, nonstat, 1.0 / kappa, nu, 0.0, 0.0, 0.0};
  if (family == 2) {
    c.snu = std::sqrt(2.0 * nu);
    c.lcnu = (1.0 - nu) * std::log(2.0) - std::lgamma(nu);
    c.dlcnu = -std::log(2.0) - digamma_host(nu);
  }
  return c;
}

__device__ __forceinline__ double gvar(double x) { return 1.0 + 0.5 * sin(4.0 * PI * x); }

// ---- e^{-a}, a >= 0, for the covariance evaluations --------------------------
// Table-driven argument reduction (Tang, "Table-driven implementation of the
// exponential function in IEEE floating-point arithmetic", ACM TOMS 15, 1989):
// -a = k ln2/64 + r with k = round(-a 64/ln2), |r| <= ln2/128, so
// e^{-a} = 2^floor(k/64) 2^{(k mod 64)/64} e^r; 2^{j/64} comes from a table built
// at compile time from its Taylor series in long double, e^r - 1 from the
// Taylor polynomial of degree 5 (truncation below 4e-17 relative).  About 11
// FP64 operations; error about 1.5 ulp.  Returns 0 for a > 708 (below 1e-307).
constexpr long double MRA_LN2L = 0.693147180559945309417232121458176568L;

constexpr double exp2_frac(int j) {            // 2^(j/64)
  long double x = (long double)j / 64.0L * MRA_LN2L, term = 1.0L, sum = 1.0L;
  for (int k = 1; k < 40; ++k) {
    term *= x / (long double)k;
    sum += term;
  }
  return (double)sum;
}
#define MRA_EXP2_T8(b)                                                                                      \
  exp2_frac(b), exp2_frac(b + 1), exp2_frac(b + 2), exp2_frac(b + 3), exp2_frac(b + 4), exp2_frac(b + 5), \
      exp2_frac(b + 6), exp2_frac(b + 7)
#define MRA_EXP2_TAB                                                                                           \
  {                                                                                                           \
    MRA_EXP2_T8(0), MRA_EXP2_T8(8), MRA_EXP2_T8(16), MRA_EXP2_T8(24), MRA_EXP2_T8(32), MRA_EXP2_T8(40),         \
        MRA_EXP2_T8(48), MRA_EXP2_T8(56)                                                                      \
  }
static __device__ const double k_exp2_tab[64] = MRA_EXP2_TAB;
constexpr double k_exp2_tab_host[64] = MRA_EXP2_TAB;

constexpr double MRA_EXP_INV = (double)(64.0L / MRA_LN2L);                 // 64 / ln2
constexpr double MRA_EXP_C1 = (double)((long double)(long long)(MRA_LN2L / 64.0L * 4398046511104.0L) /
                                       4398046511104.0L);                  // ln2/64 to 36 bits: k C1 exact
constexpr double MRA_EXP_C2 = (double)(MRA_LN2L / 64.0L - (long double)MRA_EXP_C1);

__host__ __device__ inline double exp_neg_tab(double a, const double* tab) {
  if (!(a <= 708.0)) return 0.0;
  const double t = -a;
  const double magic = 6755399441055744.0;     // 1.5 2^52: adding it rounds to an integer
  const double kd0 = fma(t, MRA_EXP_INV, magic);
  long long kb;
#ifdef __CUDA_ARCH__
  kb = __double_as_longlong(kd0);
#else
  memcpy(&kb, &kd0, 8);
#endif
  const int k = (int)(unsigned)(kb & 0xFFFFFFFFll);
  const double kd = kd0 - magic;
  double r = fma(-kd, MRA_EXP_C1, t);
  r = fma(-kd, MRA_EXP_C2, r);
  double q = fma(r, 1.0 / 120.0, 1.0 / 24.0);
  q = fma(q, r, 1.0 / 6.0);
  q = fma(q, r, 0.5);
  q = fma(q, r, 1.0);
  q *= r;                                      // e^r - 1
  const int j = k & 63, m = k >> 6;            // k <= 0: m = floor(k / 64)
#ifdef __CUDA_ARCH__
  const double tj = __ldg(tab + j);
#else
  const double tj = tab[j];
#endif
  const double v = fma(tj, q, tj);
  const long long sb = (long long)(m + 1023) << 52;
  double s2;
#ifdef __CUDA_ARCH__
  s2 = __longlong_as_double(sb);
#else
  memcpy(&s2, &sb, 8);
#endif
  return v * s2;
}

__device__ __forceinline__ double exp_neg(double a) { return exp_neg_tab(a, k_exp2_tab); }

// Euclidean distance times s, sqrt through the reciprocal square root.
__device__ __forceinline__ double dist_scaled(double dx, double dy, double s) {
  const double u = fma(dx, dx, dy * dy);
  return u > 0.0 ? u * rsqrt(u) * s : 0.0;
}

// ---- Matern correlation of smoothness nu (family 2) --------------------------
// rho(h) = 2^(1-nu) / Gamma(nu) z^nu K_nu(z), z = sqrt(2 nu) h (the scaling of
// Eq. mat15, which is nu = 3/2; nu = 1/2 is the exponential), with the
// modified Bessel function of the second kind from its integral
//     K_nu(z) = int_0^inf exp(-z cosh t) cosh(nu t) dt,
// evaluated by the trapezoidal rule, whose error falls exponentially with
// 1/step for an integrand analytic in a strip around the real axis
// (Trefethen & Weideman, "The exponentially convergent trapezoidal rule",
// SIAM Review 56, 2014): step min(0.2, 0.5/sqrt(z), 0.9/(1+nu)), nodes until
// z (cosh t - 1) - max(nu, 1 - nu) t > 40.  The same nodes give K_{nu-1}, whence
// d(z^nu K_nu)/dz = -z^nu K_{nu-1}, and dK/dnu (integrand t sinh(nu t)).  Relative error below about 1e-13 for
// nu in [0.3, 6] and z in [1e-8, 600] (checked on the host against the
// modified Bessel function of a library); sums are taken relative to e^{-z},
// so rho = c_nu exp(nu log z - z) h S0 never overflows.
struct MaternNu {
  double rho, dh, dnu;   // rho, d rho / d h, d rho / d nu (h fixed)
};

__host__ __device__ inline MaternNu matern_nu(const Cov& c, double h) {
  if (!(h > 0.0)) return MaternNu{1.0, 0.0, 0.0};
  const double nu = c.nu, z = c.snu * h;
#ifdef __CUDA_ARCH__
  const double* tab = k_exp2_tab;
  const double rz = rsqrt(z);
#else
  const double* tab = k_exp2_tab_host;
  const double rz = 1.0 / std::sqrt(z);
#endif
  const double q = fmin(fmin(0.2, 0.5 * rz), 0.9 / (1.0 + nu));
  // e^{t}, e^{nu t} and e^{(nu - 1) t} at the nodes t = k q, by recurrence
  const double e1 = exp(q), e1n = exp(nu * q), e1m = exp((nu - 1.0) * q);
  const double ie1 = 1.0 / e1, ie1n = 1.0 / e1n, ie1m = 1.0 / e1m;
  double E = 1.0, Ei = 1.0, En = 1.0, Eni = 1.0, Em = 1.0, Emi = 1.0;
  double s0 = 0.5, s2 = 0.0, s3 = 0.5;          // t = 0: weight 1/2, cosh = 1, t sinh(nu t) = 0
  for (int k = 1; k < 4096; ++k) {
    E *= e1;
    Ei *= ie1;
    En *= e1n;
    Eni *= ie1n;
    Em *= e1m;
    Emi *= ie1m;
    const double t = k * q;
    const double cm1 = 0.5 * (E + Ei) - 1.0;        // cosh t - 1
    const double ex = z * cm1;
    const double w = exp_neg_tab(ex, tab);
    s0 = fma(w, 0.5 * (En + Eni), s0);              // cosh(nu t)
    s2 = fma(w * t, 0.5 * (En - Eni), s2);          // t sinh(nu t)
    s3 = fma(w, 0.5 * (Em + Emi), s3);              // cosh((nu - 1) t)
    if (ex - fmax(nu, 1.0 - nu) * t > 40.0) break;   // (the order-(nu - 1) integrand decays at 1 - nu)
  }
  const double lz = log(z);
  const double rho = exp(c.lcnu + nu * lz - z) * q * s0;
  const double r2 = s2 / s0, r3 = s3 / s0;         // (dK_nu/dnu) / K_nu and K_{nu-1} / K_nu
  // d(z^nu K_nu(z))/dz = -z^nu K_{nu-1}(z), so d rho / d z = -rho K_{nu-1}/K_nu; d z / d h = sqrt(2 nu)
  const double dh = -rho * r3 * c.snu;
  // d log rho / d nu = d log c_nu + log z + (dK/dnu)/K + (dz/dnu) (nu/z + K'/K), dz/dnu = z / (2 nu),
  // and nu/z + K'/K = -K_{nu-1}/K
  const double dnu = rho * (c.dlcnu + lz + r2 - 0.5 * z / nu * r3);
  return MaternNu{rho, dh, dnu};
}

__device__ __forceinline__ double cov0(const Cov& c, double x1, double y1, double x2, double y2) {
  double rho;
  if (c.family == 2) {
    rho = matern_nu(c, dist_scaled(x1 - x2, y1 - y2, c.ik)).rho;
  } else if (c.family == 0) {
    rho = exp_neg(dist_scaled(x1 - x2, y1 - y2, c.ik));
  } else {
    const double a = dist_scaled(x1 - x2, y1 - y2, SQRT3 * c.ik);
    const double e = exp_neg(a);
    rho = fma(a, e, e);                        // (1 + a) e^{-a}
  }
  double v = c.sigma2 * rho;
  if (c.nonstat) v *= sqrt(gvar(x1) * gvar(x2));
  return v;
}

// The same with the free-smoothness family's quadrature as a call, for the kernels
// of the emulation engine: inlined its loop shared their 128 registers a thread with
// the engine's state (n = 60,000, r = 36: prior 13.9 -> 12.1 ms, chain 29.5 -> 24.9 ms;
// the kernels of 256 threads and 255 registers took 12.4 and 24.9).
static __device__ __noinline__ double matern_rho(double nu, double snu, double lcnu, double h) {
  Cov c{};
  c.nu = nu;
  c.snu = snu;
  c.lcnu = lcnu;
  return matern_nu(c, h).rho;
}
__device__ __forceinline__ double cov0_em(const Cov& c, double x1, double y1, double x2, double y2) {
  if (c.family != 2) return cov0(c, x1, y1, x2, y2);
  double v = c.sigma2 * matern_rho(c.nu, c.snu, c.lcnu, dist_scaled(x1 - x2, y1 - y2, c.ik));
  if (c.nonstat) v *= sqrt(gvar(x1) * gvar(x2));
  return v;
}

// ---- C0 with few FP64 operations (families 0 and 1) -------------------------
// GB300 retires about 2 FP64 FMA per clock per SM against 128 FP32 operations,
// and the emulated form's kernels evaluate n M r covariances per evaluation,
// so these form C0 from the squared scaled distance u = (s dx)^2 + (s dy)^2
// (s = 1/kappa for the exponential, sqrt(3)/kappa for Matern-1.5) and a
// variance factor sc with 8 (exponential) or 9 (Matern-1.5) FP64 operations,
// the rest on the FP32 and integer pipes:
//  * a = sqrt(u): an FP32 reciprocal square root corrected once in
//    double-float arithmetic (Dekker, "A floating-point technique for
//    extending the available precision", Numer. Math. 18, 1971), which is
//    good to about 2^-44, then one FP64 Newton step;
//  * e^{-a} = 2^{-m} 2^{-j/4096} e^{-r} with k = 4096 m + j the nearest
//    integer to a 4096/ln2 (from the double-float seed), r = a - k ln2/4096 in
//    FP64 with ln2/4096 split so that k C1 is exact (Cody & Waite), and
//    e^{-r} - 1 = -r + r^2/2 - r^3/6 + r^4/24 in double-float (|r| <= 8.5e-5:
//    truncation below 2^-70); 2^{-j/4096} from a 4096-entry table and 2^{-m}
//    folded into sc through the exponent field.
// Error within a few ulp of the exactly rounded value, plus a 2^-53 relative
// (as for any evaluation from a rounded distance); a > 708 gives 0, as
// exp_neg does.
constexpr int C0_GMAX = 16;                    // knot-grid sides whose squared offsets the kernels tabulate

constexpr long double exp2n_frac(int j, int den) {   // 2^{-j/den} by its Taylor series
  long double x = -(long double)j / (long double)den * MRA_LN2L, term = 1.0L, sum = 1.0L;
  for (int k = 1; k < 40; ++k) {
    term *= x / (long double)k;
    sum += term;
  }
  return sum;
}
struct C0Tab {
  double v[4096];
};
constexpr C0Tab make_c0_tab() {              // 2^{-j/4096} = 2^{-(j>>6)/64} 2^{-(j&63)/4096}
  C0Tab t{};
  for (int j = 0; j < 4096; ++j) t.v[j] = (double)(exp2n_frac(j >> 6, 64) * exp2n_frac(j & 63, 4096));
  return t;
}
static __device__ const C0Tab k_c0_tab = make_c0_tab();
constexpr long double MRA_C0_L = MRA_LN2L / 4096.0L;
constexpr double MRA_C0_C1 = (double)((long double)(long long)(MRA_C0_L * 8796093022208.0L) /
                                      8796093022208.0L);          // ln2/4096 to 2^-43: k C1 exact for k < 2^22
constexpr double MRA_C0_C2 = (double)(MRA_C0_L - (long double)MRA_C0_C1);
constexpr float MRA_C0_I1 = (float)(1.0L / MRA_C0_L);                // 4096/ln2 as two floats
constexpr float MRA_C0_I2 = (float)(1.0L / MRA_C0_L - (long double)MRA_C0_I1);

__host__ __device__ inline uint64_t c0_dbits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
__host__ __device__ inline double c0_bitsd(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
__host__ __device__ inline uint32_t c0_bitsf(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  uint32_t b;
  memcpy(&b, &f, 4);
  return b;
#endif
}
__host__ __device__ inline float c0_fbits(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(b);
#else
  float f;
  memcpy(&f, &b, 4);
  return f;
#endif
}
// Exact float -> double by bit moves (0 for zero and subnormal floats).
__host__ __device__ inline double c0_widen(float f) {
  const uint32_t u = c0_bitsf(f);
  const uint32_t e = (u >> 23) & 0xFFu;
  if (e == 0) return 0.0;
  return c0_bitsd(((uint64_t)(u & 0x80000000u) << 32) | ((uint64_t)(e + 896u) << 52) |
                  ((uint64_t)(u & 0x7FFFFFu) << 29));
}
// x = hi + lo: hi the leading 24 bits of x, lo the other 29 rounded to 24, for
// 2^-70 <= |x| < 2^127 (both 0 below).
__host__ __device__ inline void c0_split(double x, float& hi, float& lo) {
  const uint64_t b = c0_dbits(x);
  const uint32_t h = (uint32_t)(b >> 32);
  const int be = (int)((h >> 20) & 0x7FFu);
  if (be < 953) {
    hi = lo = 0.f;
    return;
  }
  const uint32_t sg = h & 0x80000000u;
  hi = c0_fbits(sg | ((uint32_t)(be - 896) << 23) | ((uint32_t)(b >> 29) & 0x7FFFFFu));
  const float rem = (float)(uint32_t)(b & 0x1FFFFFFFu) * c0_fbits((uint32_t)(be - 948) << 23);   // x 2^(be-1075)
  lo = sg ? -rem : rem;
}

// C0 (v), sc e^{-a} (e) and a = sqrt(u), from which the gradient's derivative
// pairs follow: dC0/dsigma2 = v / sigma2, dC0/dkappa = e a / kappa
// (exponential) or e a^2 / kappa (Matern-1.5).
struct C0Val {
  double v, e, a;
};

__host__ __device__ inline C0Val c0_eval(int family, double u, double sc) {
  float uh, ul;
  c0_split(u, uh, ul);
  if (!(uh >= 0x1p-60f)) {                     // zero or tiny distance: the plain evaluation
#ifdef __CUDA_ARCH__
    const double a = u > 0.0 ? sqrt(u) : 0.0;
    const double e = sc * exp_neg_tab(a, k_exp2_tab);
#else
    const double a = u > 0.0 ? std::sqrt(u) : 0.0;
    const double e = sc * exp_neg_tab(a, k_exp2_tab_host);
#endif
    return C0Val{family == 0 ? e : fma(a, e, e), e, a};
  }
  if (uh > 501264.0f) return C0Val{0.0, 0.0, 708.0};   // a > 708
#ifdef __CUDA_ARCH__
  const float y = rsqrtf(uh);
  const double* tab = k_c0_tab.v;
#else
  const float y = 1.0f / std::sqrt(uh);
  static constexpr C0Tab tabh = make_c0_tab();
  const double* tab = tabh.v;
#endif
  // a = sqrt(u): double-float seed (ah, al), then one FP64 Newton step
  const float ah = uh * y, hy = 0.5f * y;
  const float p = ah * ah, pe = fmaf(ah, ah, -p);
  const float al = (((uh - p) - pe) + ul) * hy;
  const double a0 = c0_widen(ah) + c0_widen(al);
  const double a = fma(c0_widen(hy), fma(-a0, a0, u), a0);
  // k = nearest integer to a 4096/ln2, from the seed in double-float
  const float th = ah * MRA_C0_I1;
  const float tl = fmaf(ah, MRA_C0_I1, -th) + fmaf(ah, MRA_C0_I2, al * MRA_C0_I1);
  float kf = rintf(th);
  const float fr = (th - kf) + tl;
  kf += fr > 0.5f ? 1.0f : (fr < -0.5f ? -1.0f : 0.0f);
  const int k = (int)kf;
  const double kd = c0_widen(kf);
  double rr = fma(kd, -MRA_C0_C1, a);
  rr = fma(kd, -MRA_C0_C2, rr);
  // g = e^{-r} - 1 = -r + r^2/2 - r^3/6 + r^4/24, r = rh + rl, as gh + gl
  float rh, rl;
  c0_split(rr, rh, rl);
  const float p2 = rh * rh, e2 = fmaf(rh, rh, -p2);
  const float hp = 0.5f * p2;
  const float gh = hp - rh;                    // two-sum of -rh and hp
  const float bb = gh - hp;
  const float er = (hp - (gh - bb)) + (-rh - bb);
  const float small = fmaf(0.5f, e2, fmaf(rh, rl, -rl)) + p2 * fmaf(p2, 1.0f / 24.0f, -rh * (1.0f / 6.0f));
  const double gd = c0_widen(gh) + c0_widen(er + small);
  // sc 2^{-m} by the exponent field (sc > 0 normal), then sc e^{-a}
  const int j = k & 4095, m = k >> 12;
  const uint64_t sb = c0_dbits(sc);
  if ((int)(sb >> 52) <= m) return C0Val{0.0, 0.0, a};   // below 2^-1022
#ifdef __CUDA_ARCH__
  const double tj = __ldg(tab + j);
#else
  const double tj = tab[j];
#endif
  const double tw = tj * c0_bitsd(sb - ((uint64_t)m << 52));
  const double E = fma(tw, gd, tw);
  return C0Val{family == 0 ? E : fma(a, E, E), E, a};   // Matern-1.5: (1 + a) e^{-a}
}

__host__ __device__ inline double c0_fast(int family, double u, double sc) { return c0_eval(family, u, sc).v; }

// Variance factor of C0 at a point: sqrt(1 + 0.5 sin(4 pi x)) for the
// nonstationary variance (so that C0's factor is the product at the two
// points), else 1.
__device__ __forceinline__ double c0_vfac(const Cov& c, double x) { return c.nonstat ? sqrt(gvar(x)) : 1.0; }

// Scale s of the squared distance c0_fast takes.
__host__ __device__ inline double c0_scale(const Cov& c) { return c.family == 0 ? c.ik : SQRT3 * c.ik; }

// Whether the kernels may use c0_fast on a knot grid of gx x gy.
__host__ __device__ inline bool c0_fast_ok(const Cov& c, int gx, int gy) {
  return c.family != 2 && gx <= C0_GMAX && gy <= C0_GMAX;
}

// Binary exponent e with |x| < 2^e (-2000 for zero): the row and column
// scales of the FP64-emulation engine.
__device__ __forceinline__ int xexp_of(double x) {
  const int be = (int)(((unsigned long long)__double_as_longlong(x) >> 52) & 0x7FF);
  return be == 0 ? -2000 : be - 1022;
}

// ---- partition and knots (Sec. 2.2) -----------------------------------------
// Every level-(m-1) region splits the same way: into an s_x x s_y grid of equal
// children, s_x = 2^hx_m, s_y = 2^hy_m (J_m = s_x s_y; the midpoint quadtree is
// hx_m = hy_m = 1), each side cut by repeated midpoint halving, half-open with
// the last cell closed.  Child digit j = c_x + s_x c_y; region i of level m
// holds its digits from the top level down, level t's in the hx_t + hy_t bits
// below those of the levels above.  hx_m and hy_m sit in bits 4m..4m+3 of two
// packed words (levels 1..12).
struct Box { double x0, x1, y0, y1; };

__host__ __device__ __forceinline__ int lvl_hx(unsigned long long hx, int m) { return (int)((hx >> (4 * m)) & 15ull); }
__host__ __device__ __forceinline__ int lvl_bits(unsigned long long hx, unsigned long long hy, int m) {
  return lvl_hx(hx, m) + lvl_hx(hy, m);
}
// bits of a level-m region id: hx_1 + hy_1 + ... + hx_m + hy_m
__host__ __device__ __forceinline__ int lvl_depth(unsigned long long hx, unsigned long long hy, int m) {
  int d = 0;
  for (int t = 1; t <= m; ++t) d += lvl_bits(hx, hy, t);
  return d;
}

__device__ __forceinline__ Box region_box(const double* bbox, unsigned long long hx, unsigned long long hy, int m,
                                          long i) {
  Box b{bbox[0], bbox[1], bbox[2], bbox[3]};
  int sh = lvl_depth(hx, hy, m);
  for (int t = 1; t <= m; ++t) {
    const int a = lvl_hx(hx, t), c = lvl_hx(hy, t);
    sh -= a + c;
    const long j = (i >> sh) & ((1L << (a + c)) - 1);
    const long cx = j & ((1L << a) - 1), cy = j >> a;
    for (int q = a - 1; q >= 0; --q) {
      const double xm = 0.5 * (b.x0 + b.x1);
      if ((cx >> q) & 1) b.x0 = xm; else b.x1 = xm;
    }
    for (int q = c - 1; q >= 0; --q) {
      const double ym = 0.5 * (b.y0 + b.y1);
      if ((cy >> q) & 1) b.y0 = ym; else b.y1 = ym;
    }
  }
  return b;
}

// Knot q = a + gx * b of a gx x gy cell-centred grid in box.
__device__ __forceinline__ void knot_xy(const Box& b, int gx, int gy, int q, double& x, double& y) {
  int a = q % gx, c = q / gx;
  x = b.x0 + ((a + 0.5) * (b.x1 - b.x0)) / gx;
  y = b.y0 + ((c + 0.5) * (b.y1 - b.y0)) / gy;
}

// ---- register-blocked tile product ------------------------------------------
// acc(i, j) += sum_k A(i, k) * B(j, k) for i < na, j < nb (both <= TILE).
// A(i, k) = A[i * sai + k * sak] and B(j, k) = B[j * sbj + k * sbk]: either
// operand may be row-major (sak = 1) or k-major (sai = 1).  Operands are staged
// k-major through shared memory in chunks of KC; the 16 x 16 thread grid gives
// every thread an RM x RM block of the TILE x TILE output (RM = TILE / 16).
template <int TILE>
struct TileAcc {
  static constexpr int RM = TILE / 16;
  double v[RM][RM];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int a = 0; a < RM; ++a)
#pragma unroll
      for (int b = 0; b < RM; ++b) v[a][b] = 0.0;
  }
  __device__ __forceinline__ int row(int a) const { return (threadIdx.x >> 4) * RM + a; }
  __device__ __forceinline__ int col(int b) const { return (threadIdx.x & 15) * RM + b; }
};

template <int TILE>
constexpr int tile_smem_doubles() { return 2 * KC * (TILE + 2); }

template <int TILE>
__device__ __forceinline__ void stage(double* s, const double* X, long sxi, long sxk, int nx,
                                      int k0, int kn) {
  constexpr int LD = TILE + 2;
  if (sxk == 1) {          // row-major source: threads along k for coalescing
    for (int t = threadIdx.x; t < TILE * KC; t += NT) {
      int i = t / KC, k = t - i * KC;
      s[k * LD + i] = (i < nx && k < kn) ? X[i * sxi + (long)(k0 + k)] : 0.0;
    }
  } else {                 // k-major source: threads along i
    for (int t = threadIdx.x; t < TILE * KC; t += NT) {
      int k = t / TILE, i = t - k * TILE;
      s[k * LD + i] = (i < nx && k < kn) ? X[(long)(k0 + k) * sxk + i * sxi] : 0.0;
    }
  }
}

template <int TILE>
__device__ void tile_mma(TileAcc<TILE>& acc, const double* A, long sai, long sak, int na,
                         const double* B, long sbj, long sbk, int nb, int K, double* smem) {
  constexpr int LD = TILE + 2;
  constexpr int RM = TILE / 16;
  double* sA = smem;
  double* sB = smem + KC * LD;
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  for (int k0 = 0; k0 < K; k0 += KC) {
    int kn = min(KC, K - k0);
    __syncthreads();
    stage<TILE>(sA, A, sai, sak, na, k0, kn);
    stage<TILE>(sB, B, sbj, sbk, nb, k0, kn);
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < kn; ++k) {
      double a[RM], b[RM];
#pragma unroll
      for (int q = 0; q < RM; ++q) {
        a[q] = sA[k * LD + ty * RM + q];
        b[q] = sB[k * LD + tx * RM + q];
      }
#pragma unroll
      for (int p = 0; p < RM; ++p)
#pragma unroll
        for (int q = 0; q < RM; ++q) acc.v[p][q] = fma(a[p], b[q], acc.v[p][q]);
    }
  }
  __syncthreads();
}

// The same product on a TR x TC output tile (TR, TC multiples of 16): the 16 x
// 16 thread grid gives every thread an (TR / 16) x (TC / 16) block, so a tile
// of few rows (prediction points) against TC columns wastes no FMA lanes on
// empty rows.
template <int TR, int TC>
struct TileAccR {
  static constexpr int RR = TR / 16, RC = TC / 16;
  double v[RR][RC];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int a = 0; a < RR; ++a)
#pragma unroll
      for (int b = 0; b < RC; ++b) v[a][b] = 0.0;
  }
  __device__ __forceinline__ int row(int a) const { return (threadIdx.x >> 4) * RR + a; }
  __device__ __forceinline__ int col(int b) const { return (threadIdx.x & 15) * RC + b; }
};

template <int TR, int TC>
__device__ void tile_mma_r(TileAccR<TR, TC>& acc, const double* A, long sai, long sak, int na, const double* B,
                           long sbj, long sbk, int nb, int K, double* smem) {
  constexpr int LDA = TR + 2, LDB = TC + 2;
  constexpr int RR = TR / 16, RC = TC / 16;
  double* sA = smem;
  double* sB = smem + KC * LDA;
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
  for (int k0 = 0; k0 < K; k0 += KC) {
    int kn = min(KC, K - k0);
    __syncthreads();
    stage<TR>(sA, A, sai, sak, na, k0, kn);
    stage<TC>(sB, B, sbj, sbk, nb, k0, kn);
    __syncthreads();
#pragma unroll 4
    for (int k = 0; k < kn; ++k) {
      double a[RR], b[RC];
#pragma unroll
      for (int q = 0; q < RR; ++q) a[q] = sA[k * LDA + ty * RR + q];
#pragma unroll
      for (int q = 0; q < RC; ++q) b[q] = sB[k * LDB + tx * RC + q];
#pragma unroll
      for (int p = 0; p < RR; ++p)
#pragma unroll
        for (int q = 0; q < RC; ++q) acc.v[p][q] = fma(a[p], b[q], acc.v[p][q]);
    }
  }
  __syncthreads();
}

// f(i, j, sum_k A(i, k) B(j, k)) for i < na <= 64, j < nb <= TC, in a tile of na
// rows rounded up to 16.  The FP64 unit takes 64 cycles for a DFMA instruction
// whatever its lanes do, so rows that only fill a tile cost as much as kept ones,
// while a thread's loads (one or two a DFMA even at one output row a thread)
// stay far below the shared-memory rate: leaves of 66 observations on 64-row
// tiles paid for 128.  Opens and ends with a barrier; smem: KC (64 + TC + 4) doubles.
template <int TR, int TC, typename F>
__device__ __forceinline__ void mma_rows_tile(const double* A, long sai, long sak, int na, const double* B, long sbj,
                                              long sbk, int nb, int K, double* smem, F&& f) {
  TileAccR<TR, TC> acc;
  acc.zero();
  tile_mma_r<TR, TC>(acc, A, sai, sak, na, B, sbj, sbk, nb, K, smem);
#pragma unroll
  for (int p = 0; p < TileAccR<TR, TC>::RR; ++p)
#pragma unroll
    for (int q = 0; q < TileAccR<TR, TC>::RC; ++q) {
      const int row = acc.row(p), col = acc.col(q);
      if (row < na && col < nb) f(row, col, acc.v[p][q]);
    }
}
// (RMAX: the most rows the caller has; the wider tiles would only cost the kernel registers)
template <int TC, int RMAX = 64, typename F>
__device__ __forceinline__ void mma_rows(const double* A, long sai, long sak, int na, const double* B, long sbj,
                                         long sbk, int nb, int K, double* smem, F&& f) {
  static_assert(RMAX == 16 || RMAX == 32 || RMAX == 64, "rows of a tile");
  if (RMAX == 16 || na <= 16) mma_rows_tile<16, TC>(A, sai, sak, na, B, sbj, sbk, nb, K, smem, f);
  else if (RMAX == 32 || na <= 32) mma_rows_tile<RMAX == 16 ? 16 : 32, TC>(A, sai, sak, na, B, sbj, sbk, nb, K, smem, f);
  else if (na <= 48) mma_rows_tile<RMAX == 64 ? 48 : 16, TC>(A, sai, sak, na, B, sbj, sbk, nb, K, smem, f);
  else mma_rows_tile<RMAX == 64 ? 64 : 16, TC>(A, sai, sak, na, B, sbj, sbk, nb, K, smem, f);
}
constexpr int mma_rows_smem(int tc) { return KC * (64 + 2 + tc + 2); }

// f(i, j, sum_k X(i, k) L(j, k)) for i < na <= 64, j < n <= 64 with L lower
// triangular (L(j, k) = 0 for k > j): 16 columns at a time over the k they have,
// 5/8 of the full product at n = 64.  The columns are taken from the last, so f
// may overwrite X(i, j): the columns still to come read X(., k <= j) only.
template <int RMAX = 64, typename F>
__device__ __forceinline__ void mma_lower_t(const double* X, long sxi, long sxk, int na, const double* L, long slj,
                                            long slk, int n, double* smem, F&& f) {
  for (int c0 = ((n - 1) >> 4) << 4; c0 >= 0; c0 -= 16) {
    const int nb = min(16, n - c0);
    mma_rows<16, RMAX>(X, sxi, sxk, na, L + c0 * slj, slj, slk, nb, c0 + nb, smem,
                 [&](int i, int j, double v) { f(i, c0 + j, v); });
  }
}

// f(i, j, sum_{k0 <= k < k1} A(i, k) B(j, k)) for i < na, j < nb, any sizes, in
// TR-row tiles (16: k0 = lo(first row), k1 = hi(first row + rows) trim the sum to
// the k a triangular A has in those rows; 64: rows rounded up to 16 per tile).
template <int TR, int TC, typename LO, typename HI, typename F>
__device__ __forceinline__ void mma_tiles(const double* A, long sai, long sak, int na, const double* B, long sbj,
                                          long sbk, int nb, LO&& lo, HI&& hi, double* smem, F&& f) {
  static_assert(TR == 16 || TR == 64, "row tiles of 16, or of up to 64");
  for (int r0 = 0; r0 < na; r0 += TR) {
    const int nr = min(TR, na - r0), k0 = lo(r0), k1 = hi(r0 + nr);
    for (int c0 = 0; c0 < nb; c0 += TC) {
      auto g = [&](int i, int j, double v) { f(r0 + i, c0 + j, v); };
      const double *a = A + r0 * sai + k0 * sak, *b = B + c0 * sbj + k0 * sbk;
      if constexpr (TR == 16) mma_rows_tile<16, TC>(a, sai, sak, nr, b, sbj, sbk, min(TC, nb - c0), k1 - k0, smem, g);
      else mma_rows<TC>(a, sai, sak, nr, b, sbj, sbk, min(TC, nb - c0), k1 - k0, smem, g);
    }
  }
}

// f(i, j, sum_k A(i, k) A(j, k)) for j <= i < n: the lower triangle of a Gram
// product, 16 columns at a time over the rows from their first on.
template <typename F>
__device__ __forceinline__ void mma_gram_lower(const double* A, long si, long sk, int n, int K, double* smem, F&& f) {
  for (int c0 = 0; c0 < n; c0 += 16)
    for (int r0 = c0; r0 < n; r0 += 64)
      mma_rows<16>(A + r0 * si, si, sk, min(64, n - r0), A + c0 * si, si, sk, min(16, n - c0), K, smem,
                   [&](int i, int j, double v) {
                     if (c0 + j <= r0 + i) f(r0 + i, c0 + j, v);
                   });
}

// ---- factorisations in shared memory ----------------------------------------
// Packed lower-triangle index t -> (i, k), k <= i, t = i (i + 1) / 2 + k.
__device__ __forceinline__ void tri_decode(int t, int& i, int& k) {
  int ii = (int)((sqrtf(8.0f * (float)t + 1.0f) - 1.0f) * 0.5f);
  while (ii * (ii + 1) / 2 > t) --ii;
  while ((ii + 1) * (ii + 2) / 2 <= t) ++ii;
  i = ii;
  k = t - ii * (ii + 1) / 2;
}

// A DFMA instruction holds an SM sub-partition's FP64 unit for 64 cycles however
// few of its lanes are active, dependent or not (measured), and a double rsqrt
// for about five of them.  What these routines can save is therefore the
// serial chain around the FP64 work, not the work: with one column at a time
// (scale, barrier, rank-1 update with every element's index decoded again,
// barrier) a 64 x 64 Cholesky factor took 64 us and its inverse 55 us, against
// 11 us each of FP64 time on four units.  They go by panels of FB = 4 columns:
// two barriers and one index decoding per four columns, and the next panel's
// diagonal block is updated and factorised by one warp while the others update
// the rest.  Every entry sees the same operations in the same order as with one
// column at a time, so the factors are the same to the bit.
constexpr int FB = 4;
constexpr int LGRP_MAX = 4;        // blocks of one block-diagonal matrix (leaves or regions of one group)
constexpr int FAC_MAX_N = 128;     // largest order (of all blocks together)
constexpr int FAC_SCRATCH = FAC_MAX_N * (1 + 2 * FB);   // doubles of shared scratch of the inverse (idle staging)

// The nb diagonal blocks of A start at rows seg[0] = 0 <= seg[1] <= ... <=
// seg[nb] (= the order of A); ONE: a single block of order n1.  The panels of
// all blocks run together.  STK (stacked storage): row i holds only its
// block's columns, entry (i, k) of block b at A[i lda + k - seg[b]], lda >= the
// largest block.
template <bool STK, bool ONE>
struct Blocks {
  double* A;
  int lda;
  const int* seg;
  int nb, n1;
  __device__ __forceinline__ int count() const { return ONE ? 1 : nb; }
  __device__ __forceinline__ int start(int b) const { return ONE ? 0 : seg[b]; }
  __device__ __forceinline__ int len(int b) const { return ONE ? n1 : seg[b + 1] - seg[b]; }
  __device__ __forceinline__ int longest() const {
    int n = 0;
    for (int b = 0; b < count(); ++b) n = max(n, len(b));
    return n;
  }
  // entry (i, k) of block b, both counted from the block's start
  __device__ __forceinline__ double* at(int b, int i, int k) const {
    const int s0 = start(b);
    return A + (s0 + i) * lda + k + (STK ? 0 : s0);
  }
  // item t of the concatenated per-block counts cnt(b): its block, t becomes the item within it
  template <typename F>
  __device__ __forceinline__ int find(int& t, F&& cnt) const {
    int b = 0;
    if (!ONE)
      for (int c = cnt(0); t >= c; c = cnt(b)) {
        t -= c;
        ++b;
      }
    return b;
  }
  template <typename F>
  __device__ __forceinline__ int total(F&& cnt) const {
    int s = 0;
    for (int b = 0; b < count(); ++b) s += cnt(b);
    return s;
  }
};

// Lower Cholesky factor of every block in place; a non-positive (or NaN) pivot
// sets *bad and is replaced by 1 so the factorisation stays finite.
template <bool STK, bool ONE, int NTH>
__device__ inline void chol_panels(const Blocks<STK, ONE> M, int* bad) {
  __shared__ double pinv[LGRP_MAX][FB];        // reciprocal square roots of the panel's pivots
  static_assert(FB == 4, "the diagonal block's lanes and the solve below are written for four columns");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nb = M.count();
  // lane e < 10 holds entry (er, ec) of a 4 x 4 lower triangle, e = er (er + 1) / 2 + ec
  const int er = lane < 1 ? 0 : (lane < 3 ? 1 : (lane < 6 ? 2 : 3)), ec = lane - er * (er + 1) / 2;
  // one warp: the diagonal block at row j of block b, first (upd) updated with the panel before it
  auto diagonal = [&](int b, int j, bool upd) {
    const int w = min(FB, M.len(b) - j);
    const bool in = lane < 10 && er < w;
    double* const p = M.at(b, j + er, j + ec);
    double x = in ? *p : 1.0;
    if (upd && in)
      for (int q = j - FB; q < j; ++q) x = fma(-*M.at(b, j + er, q), *M.at(b, j + ec, q), x);
    __syncwarp();
#pragma unroll
    for (int c = 0; c < FB; ++c) {
      const double d = __shfl_sync(0xffffffffu, x, c * (c + 1) / 2 + c);
      const bool ok = d > 0.0;
      const double rs = ok ? rsqrt(d) : 1.0;
      if (c < w && lane == 0) {
        if (!ok) *bad = 1;
        pinv[b][c] = rs;
      }
      if (ec == c) x = ok || er != c ? x * rs : 1.0;
      const double xr = __shfl_sync(0xffffffffu, x, (er * (er + 1) / 2 + c) & 31);
      const double xc = __shfl_sync(0xffffffffu, x, (ec * (ec + 1) / 2 + c) & 31);
      if (ec > c) x = fma(-xr, xc, x);
    }
    if (in) *p = x;
  };
  __syncthreads();
  if (warp < nb && M.len(warp) > 0) diagonal(warp, 0, false);
  __syncthreads();
  const int nmax = M.longest();
  for (int j = 0; j + FB < nmax; j += FB) {
    auto below = [&](int b) { return max(0, M.len(b) - j - FB); };
    // the panel's rows below its diagonal block
    const int rows = M.total(below);
    for (int t = threadIdx.x; t < rows; t += NTH) {
      int u = t;
      const int b = M.find(u, below);
      const double *L1 = M.at(b, j + 1, j), *L2 = M.at(b, j + 2, j), *L3 = M.at(b, j + 3, j);
      double* a = M.at(b, j + FB + u, j);
      const double l0 = a[0] * pinv[b][0];
      const double l1 = fma(-l0, L1[0], a[1]) * pinv[b][1];
      const double l2 = fma(-l1, L2[1], fma(-l0, L2[0], a[2])) * pinv[b][2];
      const double l3 = fma(-l2, L3[2], fma(-l1, L3[1], fma(-l0, L3[0], a[3]))) * pinv[b][3];
      a[0] = l0;
      a[1] = l1;
      a[2] = l2;
      a[3] = l3;
    }
    __syncthreads();
    // the trailing lower triangles; their first rows (the next diagonal blocks) by warp b, and while the
    // rest is less than that chain takes, the other warps of its sub-partition leave it the FP64 unit
    // (log-likelihood at n = 2^14, emulated: 3.023 ms; 3.027 never leaving it, 3.038 always; n = 4096, FP64:
    // 0.648, 0.648, 0.650)
    auto rest = [&](int b) {
      const int m = below(b);
      return m < FB ? 0 : m * (m + 1) / 2 - FB * (FB + 1) / 2;
    };
    const int tot = M.total(rest);
    const bool leave = nb < 4 && tot < 900;
    if (warp < nb) {
      if (below(warp) > 0) diagonal(warp, j + FB, true);
    } else if (!leave || (warp & 3) >= nb) {
      const int id = leave ? (warp >> 2) * (4 - nb) + (warp & 3) - nb : warp - nb;
      const int cnt = leave ? (NTH / 128) * (4 - nb) : NTH / 32 - nb;
      for (int t = id * 32 + lane; t < tot; t += cnt * 32) {
        int u = t, ii, kk;
        const int b = M.find(u, rest);
        tri_decode(u + FB * (FB + 1) / 2, ii, kk);
        const double *x = M.at(b, j + FB + ii, j), *y = M.at(b, j + FB + kk, j);
        double* p = M.at(b, j + FB + ii, j + FB + kk);
        double v = *p;
#pragma unroll
        for (int q = 0; q < FB; ++q) v = fma(-x[q], y[q], v);
        *p = v;
      }
    }
    __syncthreads();
  }
}

// Lower-triangular L of every block in place -> L^{-1}, by forward substitution
// on the rows of the identity, four rows at a time: the panel's rows are
// finished column by column (one thread a column), then their multiples are
// subtracted from every row below.
template <bool STK, bool ONE, int NTH>
__device__ inline void trinv_panels(const Blocks<STK, ONE> M, double* scr) {
  double* const rinv = scr;                            // 1 / L_ii
  double* const lps = scr + FAC_MAX_N;                 // the panel's columns of L, before they are overwritten: two panels
  auto save = [&](int j, int buf) {                    // rows j .. of columns j .. j + 3 of every block
    auto cnt = [&](int b) { return max(0, M.len(b) - j) * FB; };
    const int n = M.total(cnt);
    for (int t = threadIdx.x; t < n; t += NTH) {
      int u = t;
      const int b = M.find(u, cnt);
      const int i = j + u / FB, q = u % FB;
      lps[buf * FAC_MAX_N * FB + (M.start(b) + i) * FB + q] = j + q <= i ? *M.at(b, i, j + q) : 0.0;
    }
  };
  __syncthreads();
  {
    auto cnt = [&](int b) { return M.len(b); };
    const int n = M.total(cnt);
    for (int t = threadIdx.x; t < n; t += NTH) {
      int u = t;
      const int b = M.find(u, cnt);
      rinv[t] = 1.0 / *M.at(b, u, u);
    }
  }
  save(0, 0);
  __syncthreads();
  const int nmax = M.longest();
  for (int j = 0, buf = 0; j < nmax; j += FB, buf ^= 1) {
    // rows j .. j + w - 1: X_ik = (X_ik - sum_{s < i} L_is X_sk) / L_ii, one thread a column
    auto width = [&](int b) { return min(FB, max(0, M.len(b) - j)); };
    auto cols = [&](int b) { return width(b) ? j + width(b) : 0; };
    const int nc = M.total(cols);
    for (int t = threadIdx.x; t < nc; t += NTH) {
      int k = t;
      const int b = M.find(k, cols), w = width(b);
      const double *l = lps + buf * FAC_MAX_N * FB + (M.start(b) + j) * FB, *ri = rinv + M.start(b) + j;
      double x[FB];
#pragma unroll
      for (int q = 0; q < FB; ++q)
        if (q < w) {
          double* p = M.at(b, j + q, k);
          double v = k < j ? *p : 0.0;
#pragma unroll
          for (int s = 0; s < q; ++s)
            if (k <= j + s) v = fma(-l[q * FB + s], x[s], v);
          x[q] = k < j + q ? v * ri[q] : ri[q];
          if (k <= j + q) *p = x[q];
        }
    }
    __syncthreads();
    // X_ik -= sum_q L_iq X_qk for the rows below (the panel's own columns start from 0)
    auto upd = [&](int b) { return max(0, M.len(b) - j - FB) * (j + FB); };
    const int tot = M.total(upd), w = j + FB;
    for (int t = threadIdx.x; t < tot; t += NTH) {
      int u = t;
      const int b = M.find(u, upd);
      const int ii = u / w, k = u - ii * w, i = j + FB + ii;
      const double* l = lps + buf * FAC_MAX_N * FB + (M.start(b) + i) * FB;
      double* p = M.at(b, i, k);
      double v = k < j ? *p : 0.0;
#pragma unroll
      for (int q = 0; q < FB; ++q)
        if (k <= j + q) v = fma(-l[q], *M.at(b, j + q, k), v);
      *p = v;
    }
    save(j + FB, buf ^ 1);
    __syncthreads();
  }
}

// Lower Cholesky factor in place (A = L L'); the strict upper triangle is set
// to zero.  Ends with a barrier.
template <int NTH = NT>
__device__ inline void chol_smem(double* A, int n, int lda, int* bad) {
  chol_panels<false, true, NTH>(Blocks<false, true>{A, lda, nullptr, 1, n}, bad);
  for (int t = threadIdx.x; t < n * n; t += NTH) {
    int i = t / n, k = t - i * n;
    if (k > i) A[i * lda + k] = 0.0;
  }
  __syncthreads();
}

// L^{-1} of the lower triangle in place (n <= FAC_MAX_N; scr: FAC_SCRATCH doubles).
template <int NTH = NT>
__device__ inline void trinv_smem(double* A, int n, int lda, double* scr) {
  trinv_panels<false, true, NTH>(Blocks<false, true>{A, lda, nullptr, 1, n}, scr);
}

// ---- block-diagonal factorisations (a group of leaves in one CTA) ---------
// chol_seg factorises every block in place as chol_smem factorises one matrix
// and leaves every entry outside the blocks' lower triangles zero; trinv_seg
// inverts every block's lower triangle as trinv_smem does.
__device__ __forceinline__ int seg_block(const int* seg, int nb, int i) {   // block of row i
  int b = 0;
  while (b + 1 < nb && i >= seg[b + 1]) ++b;
  return b;
}

template <bool STK = false, int NTH = NT>
__device__ inline void chol_seg(double* A, int lda, const int* seg, int nb, int* bad) {
  chol_panels<STK, false, NTH>(Blocks<STK, false>{A, lda, seg, nb, 0}, bad);
  const int n = seg[nb];
  if (STK) {                                   // (stacked: row i holds its block's columns only, lda of them)
    for (int t = threadIdx.x; t < n * lda; t += NTH) {
      const int i = t / lda, k = t - i * lda;
      if (k > i - seg[seg_block(seg, nb, i)]) A[t] = 0.0;
    }
  } else {
    for (int t = threadIdx.x; t < n * n; t += NTH) {
      const int i = t / n, k = t - i * n;
      if (k > i || k < seg[seg_block(seg, nb, i)]) A[i * lda + k] = 0.0;
    }
  }
  __syncthreads();
}

template <bool STK = false, int NTH = NT>
__device__ inline void trinv_seg(double* A, int lda, const int* seg, int nb, double* scr) {
  trinv_panels<STK, false, NTH>(Blocks<STK, false>{A, lda, seg, nb, 0}, scr);
}

// ---- reductions --------------------------------------------------------------
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// d C0 / d sigma2, d C0 / d kappa and (family 2) d C0 / d nu at one pair of points.
__device__ __forceinline__ void dcov0(const Cov& c, double x1, double y1, double x2, double y2, double& ds2,
                                      double& dk, double& dnu) {
  double rho, drho;   // rho(h/kappa) and kappa * d rho / d kappa (= -h rho'(h))
  dnu = 0.0;
  if (c.family == 2) {
    const double h = dist_scaled(x1 - x2, y1 - y2, c.ik);
    const MaternNu mv = matern_nu(c, h);
    rho = mv.rho;
    drho = -h * mv.dh;
    dnu = c.sigma2 * mv.dnu;
  } else if (c.family == 0) {
    const double h = dist_scaled(x1 - x2, y1 - y2, c.ik);
    rho = exp_neg(h);
    drho = rho * h;
  } else {
    const double a = dist_scaled(x1 - x2, y1 - y2, SQRT3 * c.ik);
    const double e = exp_neg(a);
    rho = fma(a, e, e);
    drho = a * a * e;
  }
  double gg = c.nonstat ? sqrt(gvar(x1) * gvar(x2)) : 1.0;
  ds2 = rho * gg;
  dk = c.sigma2 * drho * gg * c.ik;
  dnu *= gg;
}

// The same two derivatives for families 0 and 1 with c0_eval's few FP64
// operations (10 instead of about 35): u the squared scaled distance
// (c0_scale), sc the variance factor with sigma2, is2 = 1 / sigma2.
__device__ __forceinline__ void dcov_fast(const Cov& c, double u, double sc, double is2, double& ds2, double& dk) {
  const C0Val z = c0_eval(c.family, u, sc);
  const double ea = z.e * z.a * c.ik;
  ds2 = z.v * is2;
  dk = c.family == 0 ? ea : ea * z.a;
}

// C0 at one pair of points (rounded exactly as cov0) and, from the same
// exponential, dcov0's two derivatives (rounded exactly as dcov0).
__device__ __forceinline__ double cov0_d(const Cov& c, double x1, double y1, double x2, double y2, double& ds2,
                                         double& dk) {
  double rho, drho;
  if (c.family == 2) {   // (the gradient keeps no derivative cache for this family: it also needs d/dnu)
    const double h = dist_scaled(x1 - x2, y1 - y2, c.ik);
    const MaternNu mv = matern_nu(c, h);
    rho = mv.rho;
    drho = -h * mv.dh;
  } else if (c.family == 0) {
    const double h = dist_scaled(x1 - x2, y1 - y2, c.ik);
    rho = exp_neg(h);
    drho = rho * h;
  } else {
    const double a = dist_scaled(x1 - x2, y1 - y2, SQRT3 * c.ik);
    const double e = exp_neg(a);
    rho = fma(a, e, e);
    drho = a * a * e;
  }
  const double gg = c.nonstat ? sqrt(gvar(x1) * gvar(x2)) : 1.0;
  ds2 = rho * gg;
  dk = c.sigma2 * drho * gg * c.ik;
  double v = c.sigma2 * rho;
  if (c.nonstat) v *= gg;
  return v;
}

// Sum over the CTA; every thread gets the result.  red: 32 doubles of shared.
template <int NTH = NT>
__device__ __forceinline__ double block_sum(double v, double* red) {
  v = warp_sum(v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  for (int w = 0; w < NTH / 32; ++w) s += red[w];
  __syncthreads();
  return s;
}

// Lower-tile index of block (k, l), k >= l, in a packed block-lower store.
__host__ __device__ __forceinline__ int tri_index(int k, int l) { return k * (k + 1) / 2 + l; }

}  // namespace mra
