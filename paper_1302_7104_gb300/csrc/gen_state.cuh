// FP32 storage, N_i = 16 and 24: the moments of one node (Eqs. 3-5) and its
// state in float-float arithmetic, every value entering error-free (two-sum,
// two-product), so that the result is good to ~2^-44 and rounds to float as
// the double-precision sums do.
//
// The field kernels of these sets took four FP64 operations and a conversion
// per label before; the chip starts one warp-wide FP64 operation per 76
// cycles and quarter SM, and the ~23 float operations per label that replace
// them take about a cycle each (N_i = 16, 1024^2: set state 1140 us, moments
// 713 us before).
#pragma once

#include "device_common.cuh"
#include "dvm_generic.h"
#include "f32_state.cuh"

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

}  // namespace pclb
