// fx64.cuh -- 2^x and log2 x of FP64 arguments in 64-bit fixed-point integer arithmetic, and the bond order on
// top of them.
//
// The device's FP64 unit takes 16 cycles for a warp instruction of a multiprocessor, its integer units about
// half a cycle: CUDA's exp2 and log2 made up two thirds of the FP64 kernels' time. Here a bond's 2^x chain runs on the
// integer units and the FP64 unit sees none of it. Measured against 113-bit arithmetic over the potential's ranges:
// f_R, b f_A and the coefficient cc within 2.1e-16 relative, 5.3e-17 to 5.7e-17 rms (the library's functions one after
// the other: within 6e-16 to 7e-15, 1.3e-16 to 6.8e-16 rms).
//
// Method: table-driven argument reduction and a short polynomial (P. T. P. Tang, "Table-driven implementation of
// the exponential function in IEEE floating-point arithmetic", ACM TOMS 15 (1989), and the same for the logarithm,
// ACM TOMS 16 (1990)), carried in fixed point. 2^x = 2^k 2^(j/256) (1 + p), with p = e^y - 1 a degree-5 Taylor
// polynomial on y < 2^-8.5 (remainder below 2^-60); log2 m = -log2 c_j + log2(1 + r), c_j an 11-bit reciprocal so
// that r = m c_j - 1 is formed without rounding and |r| < 2^-8.6, log2(1 + r) a degree-6 polynomial (remainder
// below 2^-61). Errors: 2^x within 2^-57 relative of the exact value for its fixed-point argument, before one
// rounding to FP64; log2 within 2^-53.9 absolute (fixed point with 54 fraction bits). See fx_bond for
// what is made of them.
#pragma once

#include <stdint.h>

#ifdef __CUDA_ARCH__
#define TSF_UMULHI64(a, b) __umul64hi((a), (b))
#define TSF_SMULHI64(a, b) __mul64hi((a), (b))
#define TSF_UMULHI32(a, b) __umulhi((a), (b))
#define TSF_SMULHI32(a, b) __mulhi((a), (b))
#else   // host form, for tests of the arithmetic on the CPU
#define TSF_UMULHI64(a, b) ((uint64_t)(((unsigned __int128)(uint64_t)(a) * (uint64_t)(b)) >> 64))
#define TSF_SMULHI64(a, b) ((int64_t)(((__int128)(int64_t)(a) * (int64_t)(b)) >> 64))
#define TSF_UMULHI32(a, b) ((uint32_t)(((uint64_t)(uint32_t)(a) * (uint32_t)(b)) >> 32))
#define TSF_SMULHI32(a, b) ((int32_t)(((int64_t)(int32_t)(a) * (int32_t)(b)) >> 32))
#endif

namespace tsf {

// Tables in the caller's memory (shared memory in the kernels; filled from fx64_tables.inc).
struct alignas(16) FxTables {
  unsigned long long exp2[256];     // 2^(j/256), 63 fraction bits
  unsigned long long log_inv[256];  // -log2(c_j), 62 fraction bits
  unsigned inv[256];                // c_j, 11 fraction bits
};

// A positive number m 2^-63 2^k, m in [2^63, 2^64).
struct FxNum {
  uint64_t m;
  int k;
};

// 2^Y for Y with 54 fraction bits, |Y| < 2^62.
__host__ __device__ __forceinline__ FxNum fx_exp2(int64_t Y, const FxTables &t) {
  const uint64_t f = (uint64_t)Y & ((1ull << 54) - 1);
  const uint64_t T = t.exp2[f >> 46];
  // y = ln2 times the low 46 bits, 72 fraction bits (y < 2^-8.5)
  const uint64_t y = TSF_UMULHI64((f & ((1ull << 46) - 1)) << 18, 0xb17217f7d1cf79acull);
  const uint32_t yh = (uint32_t)(y >> 32);         // 40 fraction bits
  uint32_t h = 0xaaaaaabu + (TSF_UMULHI32(yh, 0x2222222u) >> 8);   // 1/24 + y/120, 32 fraction bits
  h = 0x2aaaaaabu + (TSF_UMULHI32(yh, h) >> 8);                     // 1/6 + y h
  const uint64_t i1 = (1ull << 39) + TSF_UMULHI32(yh, h);           // 1/2 + y h, 40 fraction bits
  const uint64_t c = TSF_UMULHI64(y, i1 << 24);    // y (1/2 + ...), 72 fraction bits
  const uint64_t p = y + (TSF_UMULHI64(y, c) >> 8);
  FxNum r;
  r.m = T + (TSF_UMULHI64(T, p) >> 8);
  if (r.m < T) r.m = ~0ull;                        // just below 2: the polynomial's error must not carry out
  r.k = (int)(Y >> 54);
  return r;
}

// log2 of a number, 54 fraction bits.
__host__ __device__ __forceinline__ int64_t fx_log2(const FxNum &z, const FxTables &t) {
  const unsigned j = (unsigned)(z.m >> 55) & 255u;
  const int64_t R = (int64_t)((z.m >> 3) * (uint64_t)t.inv[j]);    // r = m c - 1, 71 fraction bits (mod 2^64)
  const int32_t r = (int32_t)(R >> 32);            // 39 fraction bits
  int32_t w = 0x1999999a - (TSF_SMULHI32(r, 0x15555555) >> 7);      // 1/5 - r/6, 31 fraction bits
  w = 0x20000000 - (TSF_SMULHI32(r, w) >> 7);                       // 1/4 - r w
  w = 0x2aaaaaab - (TSF_SMULHI32(r, w) >> 7);                       // 1/3 - r w
  const uint64_t q = (uint64_t)((1ll << 37) - (int64_t)TSF_SMULHI32(r, w));   // 1/2 - r w, 38 fraction bits
  const uint64_t a = (uint64_t)(R < 0 ? -R : R) << 1;
  const uint64_t r2q = TSF_UMULHI64(TSF_UMULHI64(a, a), q << 26);   // r^2 q, 80 fraction bits
  const int64_t ln = R - (int64_t)(r2q >> 9);                       // ln(1 + r), 71 fraction bits
  const int64_t l = TSF_SMULHI64(ln, 0x5c551d94ae0bf85ell) >> 7;    // log2(1 + r), 62 fraction bits
  return ((int64_t)z.k << 54) + (((int64_t)t.log_inv[j] + l + 128) >> 8);
}

// 1 + z for z = 2^Y's number.
__host__ __device__ __forceinline__ FxNum fx_one_plus(const FxNum &z) {
  FxNum w;
  if (z.k < 0) {
    w.k = 0;
    w.m = (1ull << 63) + (z.k > -64 ? z.m >> -z.k : 0ull);   // below 2: the sum of 1 and a number below 1
  } else {
    const uint64_t one = z.k < 64 ? (1ull << 63) >> z.k : 0ull;
    w.k = z.k;
    w.m = z.m + one;
    if (w.m < one) {                               // carry: the sum is at least 2^(k + 1)
      w.m = (w.m >> 1) | (1ull << 63);
      ++w.k;
    }
  }
  return w;
}

__host__ __device__ __forceinline__ uint64_t fx_bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  __builtin_memcpy(&u, &x, 8);
  return u;
#endif
}
__host__ __device__ __forceinline__ double fx_from_bits(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  __builtin_memcpy(&x, &u, 8);
  return x;
#endif
}

// A number as FP64, rounded to nearest (|k| < 1000).
__host__ __device__ __forceinline__ double fx_to_double(const FxNum &z) {
  // the carry of the rounding runs into the exponent field, as it should
  return fx_from_bits(((uint64_t)(z.k + 1022) << 52) + (z.m >> 11) + ((z.m >> 10) & 1ull));
}

// x as fixed point with S fraction bits, truncated toward zero below them; false (and no value) where |x| >= 2^L or
// x is not finite. S + L <= 62.
template <int S, int L>
__host__ __device__ __forceinline__ bool fx_from_double(double x, int64_t &out) {
  const uint64_t b = fx_bits(x);
  const int e = (int)((b >> 52) & 0x7ffu) - 1023;
  if (e >= L) return false;
  const uint64_t m = (b & 0xfffffffffffffull) | (1ull << 52);      // value m 2^(e - 52)
  const int sh = e - 52 + S;
  const uint64_t v = sh >= 0 ? m << sh : (sh > -64 ? m >> -sh : 0ull);   // zeros and subnormals give 0 (sh far below)
  out = (b >> 63) ? -(int64_t)v : (int64_t)v;
  return true;
}

// log2 of a positive normal FP64 number between 2^-200 and 2^200, 54 fraction bits; false otherwise.
__host__ __device__ __forceinline__ bool fx_log2_double(double x, const FxTables &t, int64_t &L) {
  const uint64_t u = fx_bits(x);
  const int e = (int)(u >> 52) - 1023;             // a negative x has the sign bit in here: far above 200
  L = 0;
  if (e < -200 || e > 200) return false;
  FxNum z;
  z.m = (u << 11) | (1ull << 63);
  z.k = e;
  L = fx_log2(z, t);
  return true;
}

// a b for a with FA and b with FB fraction bits, to 54 fraction bits (10 <= FA + FB - 54 <= 63).
template <int FA, int FB>
__host__ __device__ __forceinline__ int64_t fx_mul(int64_t a, int64_t b) {
  constexpr int S = FA + FB - 54;
  return (int64_t)(((uint64_t)TSF_SMULHI64(a, b) << (64 - S)) | (((uint64_t)a * (uint64_t)b) >> S));
}

__host__ __device__ __forceinline__ int64_t fx_add(int64_t a, int64_t b) { return (int64_t)((uint64_t)a + (uint64_t)b); }

// The pair functions and the bond order of one parameter set in fixed point:
//   f_R = 2^(lR + kR (r - r0)),   f_A / 2 = 2^(lA + kA (r - r0)),   zeta = 2^lB S,   b = (1 + zeta^n)^(-1/(2n)).
// The minimal form has lR = lA = log2 D0, kR = 2 kA and lB = log2 beta (S the angular sum without beta). ok: every
// constant is within the fixed-point ranges (positive prefactors, r0 < 16, |k| < 16, 1/64 <= n < 4).
struct FxLane {
  int64_t r0, kA, kR;        // 58, 58 and 58 fraction bits
  int64_t lA, lR, lB;        // 54 fraction bits
  int64_t n, inv2n;          // 60 and 56 fraction bits
  bool ok;
};
__host__ __device__ __forceinline__ FxLane fx_lane(double r0, double kA, double kR, double pA, double pR, double zB,
                                                   double n, double minus_inv2n, const FxTables &t) {
  FxLane o;
  o.r0 = o.kA = o.kR = o.n = o.inv2n = 0;
  o.ok = fx_log2_double(pA, t, o.lA);
  o.ok = fx_log2_double(pR, t, o.lR) && o.ok;
  o.ok = fx_log2_double(zB, t, o.lB) && o.ok;
  o.ok = fx_from_double<58, 4>(r0, o.r0) && fx_from_double<58, 4>(kA, o.kA) && fx_from_double<58, 4>(kR, o.kR) &&
         n >= 0.015625 && n < 4.0 && fx_from_double<60, 2>(n, o.n) && fx_from_double<56, 6>(-minus_inv2n, o.inv2n) && o.ok;
  return o;
}

// One bond: f_R, b f_A / 2 and cc = 2^lB dU/dzeta-type coefficient zeta^n / (2 zeta (1 + zeta^n)) b f_A / 2 (the
// angular factor 2^lB included, so that it multiplies derivatives of S), from the bond length and the angular sum S.
// zeta is clamped to 1e-30 from below. Each value is one exponential of a sum of exponents: the FP64 unit does none of
// the products. False where something leaves the fixed-point ranges (the caller takes the library functions).
__host__ __device__ __forceinline__ bool fx_bond(double r, double S, const FxLane &o, const FxTables &t, double &fR,
                                                 double &bh, double &cc) {
  int64_t R, LS;
  const uint64_t us = fx_bits(S);
  if (!o.ok || !fx_from_double<58, 4>(r, R) || (us >> 52) > 1023u + 200u) return false;
  const int64_t lmin = -1795276095634356808ll;     // log2(1e-30) with 54 fraction bits
  int64_t L = lmin;
  if (fx_log2_double(S, t, LS)) L = LS + o.lB > lmin ? LS + o.lB : lmin;
  else if (us != 0) return false;                  // below 2^-200; S = 0 is clamped
  if (L >= 125ll << 54) return false;              // so that n L stays below 512, which is all that fits
  const int64_t dr = R - o.r0;                     // |dr| < 32
  // sums of two exponents may wrap (at 512), from at most 200 + 512, to something beyond lim
  const int64_t YA = fx_add(o.lA, fx_mul<58, 58>(dr, o.kA)), YR = fx_add(o.lR, fx_mul<58, 58>(dr, o.kR));
  const int64_t Y = fx_mul<54, 60>(L, o.n);        // n L
  const int64_t lim = 250ll << 54;
  if (Y >= lim || Y <= -lim || YA >= lim || YA <= -lim || YR >= lim || YR <= -lim) return false;
  const FxNum w = fx_one_plus(fx_exp2(Y, t));
  const int64_t L2 = fx_log2(w, t);                // 0 <= L2 < 251
  const int64_t H = YA - fx_mul<54, 56>(L2, o.inv2n);              // log2 of b f_A / 2 (0 <= L2/(2n) < 95)
  const int64_t C = fx_add(H, Y - L - L2 - (1ll << 54) + o.lB);    // between -640 and 550 where H is above -lim
  if (H <= -lim || C >= lim || C <= -lim) return false;
  fR = fx_to_double(fx_exp2(YR, t));
  bh = fx_to_double(fx_exp2(H, t));
  cc = fx_to_double(fx_exp2(C, t));
  return true;
}

}  // namespace tsf
