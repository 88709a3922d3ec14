// FP32 storage, N_i = 16 and 24: the moments of one node (Eqs. 3-5) and its
// state, in two forms.
//
// gen_state32: float-float sums, every value entering error-free (two-sum, two-
// product), good to ~2^-44, for float results of nodes whose magnitudes leave room
// for the low parts (gen_in_range).  The ~23 float operations per label take
// about a cycle each; sums in double took four FP64 operations and a conversion
// per label, and a quarter SM starts one warp-wide FP64 operation per 76 cycles
// (N_i = 16, 1024^2: moments 713 us, now 92).
//
// gen_state_int: sums of 64-bit integers, good to the last places of double at
// every magnitude, for double results and for the nodes outside that range.  A
// float is an integer of 24 bits times a power of two: as multiples of 2^-55 of the
// node's largest power of two the values are exact down to 2^-31 of it, their
// sums and differences are exact, and products with the velocities round to a
// unit; ~13 FP64 operations per node.  (With the float-float sums everywhere the
// least temperature of the integrals had 44 bits, and 30 where the state was
// scaled by 1e-36.)  Integrals of 1024^2, N_i = 16: 306 us a call (916 in
// double, 193 in float-float).
#pragma once

#include "device_common.cuh"
#include "dvm_generic.h"
#include "f32_state.cuh"
#include "fixed64.cuh"

namespace pclb {

// (h, l) += a + b with the rounding errors kept in l.
__device__ __forceinline__ void ff_accumulate(ff& s, float a, float b) {
  float t, e;
  two_sum(s.hi, a, t, e);
  s.hi = t;
  s.lo += e + b;
}

__device__ __forceinline__ ff ff_renorm(ff a) {
  const float h = __fadd_rn(a.hi, a.lo);
  return ff{h, __fsub_rn(a.lo, __fsub_rn(h, a.hi))};
}

// m = rho, j_x, j_y, e = rho (E + u^2/2) of the node at f, labels `plane` apart.
template <int ND>
__device__ __forceinline__ void gen_raw_moments(const float* f, size_t plane, const DvmG32& c, ff m[4]) {
  constexpr int H = ND / 2;
  m[0] = ff_of(f[0]);
  m[1] = m[2] = m[3] = ff_of(0.f);
  // a shell's values are loaded while the shell before it is summed
  float v[ND], next[ND];
  auto load = [&](int k, float* o) {
#pragma unroll
    for (int i = 0; i < ND; ++i) o[i] = __ldg(f + (size_t)(1 + (k - 1) * ND + i) * plane);
  };
  load(1, next);
#pragma unroll 1
  for (int k = 1; k <= 4; ++k) {
#pragma unroll
    for (int i = 0; i < ND; ++i) v[i] = next[i];
    if (k < 4) load(k + 1, next);
    ff S = ff_of(0.f), X = S, Y = S;
#pragma unroll
    for (int i = 0; i < H; ++i) {
      const float a = v[i], b = v[i + H];
      float sh, sl, dh, dl;
      two_sum(a, b, sh, sl);
      two_sum(a, -b, dh, dl);   // opposite unit vectors
      ff_accumulate(S, sh, sl);
      float p, pe;
      two_prod(c.cxh[i], dh, p, pe);
      ff_accumulate(X, p, pe + fmaf(c.cxl[i], dh, c.cxh[i] * dl));
      two_prod(c.cyh[i], dh, p, pe);
      ff_accumulate(Y, p, pe + fmaf(c.cyl[i], dh, c.cyh[i] * dl));
    }
    S = ff_renorm(S);
    m[0] = ff_add(m[0], S);
    m[1] = ff_add(m[1], ff_mul(ff{c.sph[k], c.spl[k]}, ff_renorm(X)));
    m[2] = ff_add(m[2], ff_mul(ff{c.sph[k], c.spl[k]}, ff_renorm(Y)));
    m[3] = ff_add(m[3], ff_mul(ff{c.hvh[k], c.hvl[k]}, S));
  }
}

template <int ND>
__device__ __forceinline__ State32 gen_state32(const float* f, size_t plane, const DvmG32& c) {
  ff m[4];
  gen_raw_moments<ND>(f, plane, c, m);
  State32 s;
  const ff inv = ff_recip(m[0]);
  s.rho = m[0];
  s.ux = ff_mul(m[1], inv);
  s.uy = ff_mul(m[2], inv);
  const ff ke = ff_add(ff_mul(m[1], s.ux), ff_mul(m[2], s.uy));   // |j|^2 / rho
  s.E = ff_mul(ff_add(m[3], ff_scale(ke, -0.5f)), inv);
  s.ok = m[0].hi > 0.f && s.E.hi > 0.f && isfinite(s.E.hi) && isfinite(s.ux.hi) && isfinite(s.uy.hi);
  return s;
}

// The low parts of the float-float sums, down to 2^-48 of their terms, are normal
// numbers or nearly so, nothing overflows, and the temperature is not left over from
// terms 2^8 its size.
__device__ __forceinline__ bool gen_in_range(const State32& m) {
  const float u2 = m.ux.hi * m.ux.hi + m.uy.hi * m.uy.hi;
  return m.rho.hi >= 0x1p-70f && m.rho.hi <= 0x1p+90f && m.E.hi >= 0x1p-30f && m.E.hi <= 0x1p+30f &&
         u2 <= 256.f * m.E.hi;
}

struct GenState {
  double rho, ux, uy, E;
  bool ok;
};

// Velocity and temperature from the sums rho, rho u, rho (E + u^2/2).
__device__ __forceinline__ GenState gen_state_of(double s0, double sx, double sy, double se) {
  GenState m;
  m.rho = s0;
  m.ux = sx / s0;
  m.uy = sy / s0;
  m.E = (se - 0.5 * (sx * m.ux + sy * m.uy)) / s0;
  m.ok = s0 > 0.0 && m.E > 0.0 && isfinite(m.E) && isfinite(m.ux) && isfinite(m.uy);
  return m;
}

// By plain double sums: nodes with NaN or infinity, speeds far from 1.
static __device__ __noinline__ GenState gen_state_plain(const float* f, size_t plane, const DvmG& d) {
  double s0 = 0.0, sx = 0.0, sy = 0.0, se = 0.0;
#pragma unroll 1
  for (int q = 0; q < d.q; ++q) {
    const double v = f[(size_t)q * plane];
    s0 += v;
    sx = fma(d.vx[q], v, sx);
    sy = fma(d.vy[q], v, sy);
    se = fma(d.half_v2[d.shell[q]], v, se);
  }
  return gen_state_of(s0, sx, sy, se);
}

// The node at f, labels `plane` apart.
template <int ND>
__device__ __forceinline__ GenState gen_state_int(const float* f, size_t plane, const DvmG& d, const DvmG32& c) {
  constexpr int H = ND / 2;
  auto bits = [&](int q) { return __float_as_uint(__ldg(f + (size_t)q * plane)); };
  uint32_t top = 0;
#pragma unroll 16
  for (int q = 0; q < 1 + 4 * ND; ++q) top = max(top, bits(q) & 0x7fffffffu);
  const int ek = max((int)(top >> 23), 1);   // f = x 2^(ek - 181)
  if (ek == 255 || !c.fx_ok) return gen_state_plain(f, plane, d);
  auto fixed = [&](uint32_t b) -> int64_t {
    const uint32_t e = (b >> 23) & 0xffu;
    const uint64_t m = (uint64_t)((b & 0x7fffffu) | (e ? 0x800000u : 0u)) << 32;
    const uint64_t x = ((m >> min(ek - (int)max(e, 1u), 63)) + 1) >> 1;   // < 2^55, rounded
    return fx_signed(x, (int32_t)b >> 31);
  };
  auto times = [](int64_t x, uint64_t k) { return fx_signed(fx_mul(fx_abs(x), k), x >> 63); };
  int64_t rho = fixed(bits(0)), S[4] = {0, 0, 0, 0}, X = 0, Y = 0;
#pragma unroll 2
  for (int i = 0; i < H; ++i) {
    int64_t Z = 0;   // sum over the shells of v_k (f_i - f_i+H)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t a = fixed(bits(1 + k * ND + i)), b = fixed(bits(1 + k * ND + i + H));
      S[k] += a + b;
      Z += times(a - b, c.fx_speed[k]);
    }
    X += times(c.fx_neg_x >> i & 1 ? -Z : Z, c.fx_cx[i]);   // opposite unit vectors
    Y += times(Z, c.fx_cy[i]);
  }
  int64_t e = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    rho += S[k];
    e += times(S[k], c.fx_half_v2[k]);
  }
  const int x = ek + 900;
  const double s0 = fx_to_double(rho, x), sx = fx_to_double(X, x + c.fx_exp_v), sy = fx_to_double(Y, x + c.fx_exp_v),
               se = fx_to_double(e, x + c.fx_exp_hv), inv = recip_newton(s0);
  GenState m;
  m.rho = s0;
  m.ux = sx * inv;
  m.uy = sy * inv;
  m.E = (se - 0.5 * (sx * m.ux + sy * m.uy)) * inv;
  m.ok = s0 > 0.0 && m.E > 0.0 && isfinite(m.E) && isfinite(m.ux) && isfinite(m.uy);
  return m;
}

// The same as a call, for the nodes out of range.
template <int ND>
__device__ __noinline__ GenState gen_state_f32(const float* f, size_t plane, const DvmG& d, const DvmG32& c) {
  return gen_state_int<ND>(f, plane, d, c);
}

}  // namespace pclb
