// FP64 values as 64-bit fixed-point numbers, for the FP64 step's sums,
// differences and convection increments.
//
// GB300 starts one warp-wide FP64 operation per quarter SM every 64-76
// cycles (measured), while 64-bit integer sums take 4, 32 x 32 -> 64-bit
// products 5 and float operations about 1.  A distribution value f is held as
// x = f 2^(1081 - ek), |x| < 2^59, with ek the largest biased exponent of its
// shell in the tile's window: one unit is at most 2^-58 of the largest value,
// finer than the double's own spacing for every value within 2^-5 of it, where
// the conversion is exact.  Sums and differences of these numbers are exact;
// conversions and products round to the nearest unit.  (Both used to drop what is
// below a unit: next to gas 20 times as dense, thin gas then lost 1e-16 of its
// mass in every step.)
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "device_common.cuh"
#include "pclb_internal.h"

namespace pclb {

constexpr int kHalfDirs = kNDirs / 2;

// Exponents for which fx_to_double stays inside the normal range; NaN and
// infinity (0x7ff) are outside.
constexpr int kFxMinExp = 128, kFxMaxExp = 1900;

// f as fixed point, rounded to the nearest (ties to even, decided on five bits
// below the unit); its biased exponent must not exceed ek.
__device__ __forceinline__ int64_t fx_from_double(double f, int ek) {
  const int hi = __double2hiint(f);
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
  uint64_t m = ((uint64_t)mh << 32 | (uint32_t)__double2loint(f)) << 11;
  m >>= min(ek - ((hi >> 20) & 0x7ff), 63);
  m = (m + (15u + (((uint32_t)m >> 5) & 1u))) >> 5;
  const int64_t s = hi >> 31;
  return (int64_t)(m ^ s) - s;
}

// The double nearest x 2^(ek - 1081) (|x| < 2^63), ties to even: of the few bits
// that drop out, every fourth pattern or so is a tie.
__device__ __forceinline__ double fx_to_double(int64_t x, int ek) {
  const int64_t s = x >> 63;
  uint64_t u = (uint64_t)((x ^ s) - s);
  const int lz = __clzll((long long)u);
  u <<= lz & 63;                                        // leading bit at 63
  const uint32_t ul = (uint32_t)u;
  const uint64_t r = (u >> 11) + ((ul & 0x7ffu) + ((ul >> 11) & 1u) > 0x400u ? 1 : 0);   // 53 bits, the carry runs into the exponent
  const uint32_t hi = (uint32_t)(r >> 32) + ((uint32_t)(ek + 4 - lz) << 20) + ((uint32_t)s & 0x80000000u);
  return u == 0 ? 0.0 : __hiloint2double((int)hi, (int)(uint32_t)r);
}

// c in [0, 1] as a fraction in units of 2^-63, rounded (c < 2^-960 counts as 0).
__device__ __forceinline__ uint64_t fx_fraction(double c) {
  const int hi = __double2hiint(c);
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
  const uint64_t m = ((uint64_t)mh << 32 | (uint32_t)__double2loint(c)) << 11;   // 2^63 <= m < 2^64
  const int sh = 1023 - (hi >> 20);                     // c = m 2^-63 2^-sh
  const uint64_t one = 1ull << 63, x = sh > 63 ? 0 : (sh < 1 ? m : ((m >> (sh - 1)) + 1) >> 1);
  return x < one ? x : one;
}

// a c 2^-63 for a < 2^61, c <= 2^63, to the nearest (the error is below 1/2 + 2^-31).
__device__ __forceinline__ uint64_t fx_mul(uint64_t a, uint64_t c) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), cl = (uint32_t)c, ch = (uint32_t)(c >> 32);
  // in units of 2^32, with half a unit of the result: < 2^63 + 2^61 + 2^33
  const uint64_t mid = (uint64_t)al * ch + ((uint64_t)ah * cl + 0x40000000u) + __umulhi(al, cl);
  return (uint64_t)(2u * ah) * ch + (mid >> 31);
}

// a c 2^-64, else as fx_mul.
__device__ __forceinline__ uint64_t fx_mul_half(uint64_t a, uint64_t c) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), cl = (uint32_t)c, ch = (uint32_t)(c >> 32);
  const uint64_t mid = (uint64_t)al * ch + ((uint64_t)ah * cl + 0x80000000u) + __umulhi(al, cl);
  return (uint64_t)ah * ch + (mid >> 32);
}

// a c 2^-63 for fractions a, c <= 2^63, to the nearest.
__device__ __forceinline__ uint64_t fx_mul_frac(uint64_t a, uint64_t c) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), cl = (uint32_t)c, ch = (uint32_t)(c >> 32);
  // < 2^64: a high word is 2^31 only where the low word is 0
  const uint64_t mid = (uint64_t)al * ch + ((uint64_t)ah * cl + 0x40000000u) + __umulhi(al, cl);
  return 2 * ((uint64_t)ah * ch) + (mid >> 31);
}

__device__ __forceinline__ uint64_t fx_abs(int64_t x) {
  const int64_t s = x >> 63;
  return (uint64_t)((x ^ s) - s);
}
__device__ __forceinline__ int64_t fx_signed(uint64_t a, int64_t s) { return ((int64_t)a ^ s) - s; }   // s: 0 or -1

// x / sqrt 2 for |x| < 2^61.
__device__ __forceinline__ int64_t fx_diagonal(int64_t x) {
  return fx_signed(fx_mul(fx_abs(x), 0x5a827999fcef3242ull), x >> 63);   // 2^63 / sqrt 2
}

__device__ __forceinline__ float fx_float(uint64_t u) {
  return fmaf(__uint2float_rn((uint32_t)(u >> 32)), 4294967296.0f, __uint2float_rn((uint32_t)u));
}
__device__ __forceinline__ float fx_float(int64_t x) {
  return fmaf(__int2float_rn((int32_t)(x >> 32)), 4294967296.0f, __uint2float_rn((uint32_t)x));
}

// Courant data of one direction, alpha = |C|: M(D, Dp) = D (alpha^2 + 2 K v)
// with K = alpha (1 - alpha) and v = |D| / (|D| + |Dp|) where D and Dp have one
// sign, v = 1 where they have not (Eq. 28: a D + K |D| (D - Dp)/(|D| + |Dp|)).
struct FxCourant {
  uint64_t a2;    // alpha^2, units 2^-63
  uint64_t k40;   // 2 K rounded down to units of 2^-40
  float k2, klo;  // 2 K 2^29, and what k40 leaves off, times 2^52
};

__device__ __forceinline__ FxCourant fx_courant(uint64_t alpha) {
  FxCourant c;
  c.a2 = fx_mul_frac(alpha, alpha);
  const uint64_t k = 2 * (alpha - c.a2);
  c.k40 = k >> 23;
  c.k2 = __uint2float_rn((uint32_t)(k >> 32)) * 0.25f;
  c.klo = __uint2float_rn((uint32_t)k & 0x7fffffu) * 0.00048828125f;
  return c;
}

// M of Eq. (28) in upwind form, |D|, |Dp| < 2^60.  v is formed to ~2^-46: a
// float quotient rounded to i0 2^-23, its exact integer remainder, and the
// remainder's float quotient; 2 K v is then good to K 2^-45 + 2^-62.  Where D = 0
// the quotients may be anything (0 / 0): the result is c |D| = 0 in integers.
__device__ __forceinline__ int64_t fx_mwb(int64_t D, int64_t Dp, const FxCourant& c) {
  const int64_t s = D >> 63;
  const uint64_t a = (uint64_t)((D ^ s) - s), n = a + fx_abs(Dp);
  const uint64_t num = (int32_t)((uint32_t)(D >> 32) ^ (uint32_t)(Dp >> 32)) < 0 ? n : a;
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fx_float(n)));
  const float v0 = fx_float(num) * r;
  const uint32_t i0 = __float_as_uint(__fadd_rn(v0, 1.0f)) - 0x3f800000u;   // v0 in units of 2^-23, rounded
  const int64_t rem = (int64_t)((num << 23) - n * (uint64_t)i0);            // |rem| <= 4 n < 2^63
  const float q = fx_float(rem) * r;                                        // the rest of v, units of 2^-23
  const float k = fmaf(c.k2, q, c.klo * v0);                                // the rest of 2 K v, units of 2^-52
  const int32_t i1 = __float2int_rn(k);
  // and what i1 rounds off, units of 2^-63 (2^-53 of a D far larger than the node's own value is not small beside it)
  const int32_t i2 = __float_as_int(fmaf(k - __int2float_rn(i1), 2048.0f, 12582912.0f)) - 0x4b400000;
  const uint64_t coef = c.a2 + c.k40 * (uint64_t)i0 + (uint64_t)((int64_t)i1 * 2048 + i2);
  return fx_signed(fx_mul(a, coef), s);
}

// Largest biased exponent of the values, and whether fixed point with that
// exponent stays clear of the ends of the double range (NaN and infinity do not).
__device__ __forceinline__ int fx_exponent(int h0) { return (h0 >> 20) & 0x7ff; }
template <class... H>
__device__ __forceinline__ int fx_exponent(int h0, int h1, H... rest) {
  return fx_exponent(max(h0 & 0x7fffffff, h1 & 0x7fffffff), rest...);
}
__device__ __forceinline__ bool fx_range(int e) { return e >= kFxMinExp && e <= kFxMaxExp; }

// c in [0, 1] as a 2^-(63 + s), with 61 leading bits or more in a (subnormal c: 0).
struct FxScaled {
  uint64_t a;
  int s;
};
__device__ __forceinline__ FxScaled fx_scaled(double c) {
  const int hi = __double2hiint(c), sh = 1023 - (hi >> 20);   // c = m 2^-63 2^-sh
  const uint32_t mh = ((uint32_t)hi & 0xfffffu) | 0x100000u;
  const uint64_t m = ((uint64_t)mh << 32 | (uint32_t)__double2loint(c)) << 11;
  if (sh >= 1023) return FxScaled{0, 0};
  if (sh < 1) return FxScaled{1ull << 63, 0};
  return sh < 2 ? FxScaled{m >> 1, 0} : FxScaled{m >> 2, sh - 2};
}

// u 2^-(63 + s) as a double; 0 below its normal range.
__device__ __forceinline__ double fx_fraction_to_double(uint64_t u, int s) {
  const int lz = __clzll((long long)u), e = 1022 - lz - s;
  const uint64_t m = u << (lz & 63), r = (m >> 11) + ((m >> 10) & 1);
  const uint32_t hi = (uint32_t)(r >> 32) + ((uint32_t)e << 20);
  return u == 0 || e < 1 ? 0.0 : __hiloint2double((int)hi, (int)(uint32_t)r);
}

// |D| / (|D| + |Dp|) = v 2^-(63 + s), to ~2^-62 of it: three float quotient digits
// with exact remainders, on integer mantissas aligned to the larger of the two.
// e: the larger biased exponent (0: both below the normal range, v may be anything).
__device__ __forceinline__ FxScaled fx_switch(double D, double Dp, int& e) {
  const int hD = __double2hiint(D), hP = __double2hiint(Dp);
  const int eD = (hD >> 20) & 0x7ff, eP = (hP >> 20) & 0x7ff;
  e = max(eD, eP);
  auto mantissa = [](int h, double x, int ex) -> uint64_t {
    const uint64_t m = ((uint64_t)(((uint32_t)h & 0xfffffu) | 0x100000u) << 32 | (uint32_t)__double2loint(x)) << 6;
    return ex == 0 ? 0 : m;
  };
  const uint64_t mD = mantissa(hD, D, eD);
  const uint64_t n = (mD >> min(e - eD, 63)) + (mantissa(hP, Dp, eP) >> min(e - eP, 63));   // < 2^60
  // |D| below |Dp| by whole powers of two: they go into s, so that v keeps its bits
  const uint64_t a = e > eD ? mD >> 1 : mD;
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(fx_float(n)));
  const uint32_t i0 = __float_as_uint(__fadd_rn(fx_float(a) * r, 1.0f)) - 0x3f800000u;   // units of 2^-23
  const int64_t rem0 = (int64_t)((a << 23) - n * (uint64_t)i0);
  const int32_t i1 = __float2int_rn(fx_float(rem0) * r * 4194304.0f);                    // units of 2^-45
  const int64_t rem1 = (int64_t)(((uint64_t)rem0 << 22) - n * (uint64_t)(int64_t)i1);
  const int32_t i2 = __float2int_rn(fx_float(rem1) * r * 262144.0f);                     // units of 2^-63
  return FxScaled{((uint64_t)i0 << 40) + (uint64_t)((int64_t)i1 * 262144) + (uint64_t)(int64_t)i2, max(e - eD - 1, 0)};
}

// alpha^2 and 2 alpha (1 - alpha) of alpha = c.a 2^-(63 + c.s), in units of 2^-(63 + c.s):
// they keep their digits however small alpha is.
__device__ __forceinline__ void fx_partial_coefs(FxScaled c, uint64_t& a2, uint64_t& k2) {
  a2 = fx_mul_frac(c.a, c.a >> min(c.s, 63));
  k2 = 2 * (c.a - a2);
}

// M of Eq. (28) from doubles, good to the last places of D times the coefficient
// whatever the sizes of D, Dp and alpha: four FP64 operations with the differences.
__device__ __forceinline__ double mwb64(double alpha, double D, double Dp) {
  const FxScaled c = fx_scaled(alpha);
  uint64_t a2, k2;
  fx_partial_coefs(c, a2, k2);
  auto big = [](double x) { return ((__double2hiint(x) >> 20) & 0x7ff) >= 500; };
  const bool small = !big(D) && !big(Dp);   // scaled up: a difference may be subnormal
  if (small) { D *= 0x1p+500; Dp *= 0x1p+500; }
  int e;
  const FxScaled v = fx_switch(D, Dp, e);
  const bool opposite = (__double2hiint(D) ^ __double2hiint(Dp)) < 0;
  const uint64_t w = opposite ? k2 : fx_mul_frac(k2, v.a) >> min(v.s, 63);
  const double M = e < 0x7ff ? D * fx_fraction_to_double(a2 + w, c.s) : __hiloint2double(0x7ff80000, 0);
  return small ? M * 0x1p-500 : M;
}

// The compared schemes (Sec. II B 3) in upwind form: M = alpha D + c/2 ((D' or D)
// - (D or Dp)), c = alpha (1 - alpha) (Warming-Beam, Lax-Wendroff) or alpha
// (second-order upwind), D' = f(downwind) - f of Lax-Wendroff.
struct FxLinear {
  uint64_t a, c;   // units of 2^-63
};
template <int SCH>
using FxCoef = std::conditional_t<SCH == PCLB_SCHEME_MWB, FxCourant, FxLinear>;

template <int SCH>
__device__ __forceinline__ FxCoef<SCH> fx_coef(uint64_t alpha) {
  if constexpr (SCH == PCLB_SCHEME_MWB) return fx_courant(alpha);
  else return FxLinear{alpha, SCH == PCLB_SCHEME_UPWIND2 ? alpha : alpha - fx_mul_frac(alpha, alpha)};
}

// M of node value x0, upwind values u1, u2 and (Lax-Wendroff) downwind value d1,
// all below 2^59.
template <int SCH>
__device__ __forceinline__ int64_t fx_increment(int64_t x0, int64_t u1, int64_t u2, int64_t d1, const FxCoef<SCH>& c) {
  const int64_t D = x0 - u1;
  if constexpr (SCH == PCLB_SCHEME_MWB) {
    return fx_mwb(D, u1 - u2, c);
  } else {
    const int64_t E = SCH == PCLB_SCHEME_LW ? d1 - x0 - D : D - (u1 - u2);
    return fx_signed(fx_mul(fx_abs(D), c.a), D >> 63) + fx_signed(fx_mul_half(fx_abs(E), c.c), E >> 63);
  }
}

// The same from doubles; a = |C|.
template <int SCH>
__device__ __forceinline__ double increment64(double a, double x0, double u1, double u2, double d1) {
  const double D = x0 - u1, Dp = u1 - u2;
  if constexpr (SCH == PCLB_SCHEME_MWB) return mwb64(a, D, Dp);
  const double K = a - a * a;
  if (SCH == PCLB_SCHEME_LW) return a * D + 0.5 * K * ((d1 - x0) - D);
  return a * D + 0.5 * (SCH == PCLB_SCHEME_WB ? K : a) * (D - Dp);
}

// fx_carried from doubles; a call, as it is rare and long (within the loop, N_i =
// 24 on 1024 x 1024 took 2.09 ms a step against 2.02).
template <int SCH>
__device__ __noinline__ double carried64(double x0, double u1, double u2, double v1, double v2, double decay, double ar,
                                         double at) {
  return fma(decay, x0, -increment64<SCH>(ar, x0, u1, u2, u2)) - increment64<SCH>(at, x0, v1, v2, v2);
}

// d x0 - M_r - M_theta of one label (Eqs. 19, 28): x0 the node, u1 and v1 its
// upwind neighbours in r and theta, u2 and v2 the next ones (Lax-Wendroff: the
// downwind neighbours).  In fixed point on the exponent of the largest of
// them, or in FP64 outside its range and where x0 is more than 2^5 smaller, so
// that a unit would be coarse for it (c: the pair's FP64 Courant entry at the row).
template <int SCH>
__device__ __forceinline__ double fx_carried(double x0, double u1, double u2, double v1, double v2,
                                             const FxCoef<SCH>& cr, const FxCoef<SCH>& ct, uint64_t dfx, int64_t dsign,
                                             double decay, const double* c, double inv_r) {
  const int e = fx_exponent(__double2hiint(x0), __double2hiint(u1), __double2hiint(u2), __double2hiint(v1),
                            __double2hiint(v2));
  if (!fx_range(e) || fx_exponent(__double2hiint(x0)) < e - 5) {
    return carried64<SCH>(x0, u1, u2, v1, v2, decay, c[0], c[2] * inv_r);
  }
  const int64_t i0 = fx_from_double(x0, e);
  auto M = [&](double n1, double n2, const FxCoef<SCH>& k) {
    const int64_t f = fx_from_double(n2, e);
    return fx_increment<SCH>(i0, fx_from_double(n1, e), f, f, k);
  };
  const int64_t keep = fx_signed(fx_mul(fx_abs(i0), dfx), (i0 >> 63) ^ dsign);
  return fx_to_double(keep - M(u1, u2, cr) - M(v1, v2, ct), e);
}

// The sums S, X = sum c_x f, Y = sum c_y f of a shell at one node: f its first
// label, planes `plane` apart.
__device__ __forceinline__ void shell_sums64(const double* f, size_t plane, const DvmConst<double>& d, double o[3]) {
  double a[kHalfDirs], b[kHalfDirs];
#pragma unroll
  for (int i = 0; i < kHalfDirs; ++i) {
    a[i] = f[i * plane];
    b[i] = f[(i + kHalfDirs) * plane];
  }
  auto hi = [](double x) { return __double2hiint(x); };
  const int e = fx_exponent(hi(a[0]), hi(a[1]), hi(a[2]), hi(a[3]), hi(b[0]), hi(b[1]), hi(b[2]), hi(b[3]));
  if (!fx_range(e)) {
    double S = 0.0, D[kHalfDirs];
#pragma unroll
    for (int i = 0; i < kHalfDirs; ++i) {
      S += a[i] + b[i];
      D[i] = a[i] - b[i];
    }
    o[0] = S;
    o[1] = fma(d.cx[2], D[1] - D[3], D[0]);
    o[2] = fma(d.cx[2], D[1] + D[3], D[2]);
    return;
  }
  int64_t S = 0, D[kHalfDirs];
#pragma unroll
  for (int i = 0; i < kHalfDirs; ++i) {
    const int64_t x = fx_from_double(a[i], e), y = fx_from_double(b[i], e);
    S += x + y;
    D[i] = x - y;
  }
  o[0] = fx_to_double(S, e);
  o[1] = fx_to_double(D[0] + fx_diagonal(D[1] - D[3]), e);
  o[2] = fx_to_double(D[2] + fx_diagonal(D[1] + D[3]), e);
}

// Node state from the rest value and the four shells' sums.
__device__ __forceinline__ NodeState<double> state_of_sums(double f0, const double* s, const DvmConst<double>& d) {
  double s0 = f0, sx = 0.0, sy = 0.0, se = 0.0;
#pragma unroll
  for (int k = 1; k <= 4; ++k) {
    s0 += s[3 * (k - 1)];
    sx = fma(d.speed[k], s[3 * (k - 1) + 1], sx);
    sy = fma(d.speed[k], s[3 * (k - 1) + 2], sy);
    se = fma(d.half_v2[k], s[3 * (k - 1)], se);
  }
  return node_state64(s0, sx, sy, se);
}

// Partial derivatives of M of Eq. (28) (mwb_partials in adjoint_common.cuh) with
// respect to D and Dp, from a2 = alpha^2 and k2 = 2 alpha (1 - alpha) in units of
// 2^-(63 + s).  With v = |D| / (|D| + |Dp|): D and Dp of one sign, M_D = a2 + 2 k2 v -
// k2 v^2 and M_Dp = -k2 v^2; of opposite signs, a2 + k2 and 0; D = 0, a2 + k2 / 2
// and 0; Dp = 0, a2 + k2 and -k2 / 2.  v is formed on integer mantissas
// (fx_switch), so the only FP64 operations are the caller's two differences.  Not
// finite: NaN.
__device__ __forceinline__ void fx_mwb_partials(double D, double Dp, uint64_t a2, uint64_t k2, int s, double& MD, double& MDp) {
  int e;
  const FxScaled v = fx_switch(D, Dp, e);
  const uint64_t w = fx_mul_frac(k2, v.a), wv = fx_mul_frac(w, v.a);   // times 2^-v.s and 2^-2v.s
  const int hD = __double2hiint(D), hP = __double2hiint(Dp);
  const bool zD = (((uint32_t)hD << 1) | (uint32_t)__double2loint(D)) == 0;
  const bool zP = (((uint32_t)hP << 1) | (uint32_t)__double2loint(Dp)) == 0;
  const bool opposite = (hD ^ hP) < 0;
  uint64_t md = a2 + 2 * (w >> min(v.s, 63)) - (wv >> min(2 * v.s, 63)), mp = wv;
  int sp = s + 2 * v.s;
  if (opposite || zP) { md = a2 + k2; mp = zP ? k2 >> 1 : 0; sp = s; }
  if (zD || e == 0) { md = a2 + (k2 >> 1); mp = 0; }
  const bool finite = e < 0x7ff;
  MD = finite ? fx_fraction_to_double(md, s) : __hiloint2double(0x7ff80000, 0);
  MDp = finite ? -fx_fraction_to_double(mp, sp) : MD;
}

}  // namespace pclb
