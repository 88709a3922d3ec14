// FP32 path: the node state and equilibrium factors of two radially adjacent
// nodes in packed FP32x2 float-float arithmetic (Eqs. 10-11), shared by the
// step and the set-state kernel.
#pragma once

#include "device_common.cuh"
#include "f32_state.cuh"
#include "f32x2.cuh"

namespace pclb {

// Unit vectors of the first direction of each opposite pair, i = 0..3 of the
// octagon (Eq. 2), as float-float pairs: (1,0), (s,s), (0,1), (-s,s), s = 1/sqrt 2.
constexpr float kS = 0.7071067690849304f;
constexpr float kSl = 1.2101617152815436e-08f;

struct State2 {
  ff2 rho, ux, uy, E;
};

__device__ __forceinline__ ff2 ffc(float hi, float lo) { return ff2{bc2(hi), bc2(lo)}; }

struct Eq2 {
  f2 w[5];                  // rho F_k(E)
  f2 a0, a1, a1h;           // Eq. (10) polynomial coefficients
  f2 yh[kHalf], yl[kHalf];  // c_i . u / E, float-float
};

// F_k(E) of Eq. (11a).
__device__ __forceinline__ ff2 shell_weight2(const ff2& E, const DvmConst<float>& d, int k) {
  ff2 a = ffc(d.Fc[k][3], d.Fc_lo[k][3]);
#pragma unroll
  for (int n = 2; n >= 0; --n) a = ff2_mul_add(a, E, ffc(d.Fc[k][n], d.Fc_lo[k][n]));
  return ff2_mul(a, E);
}

// rho F_0 from the sum of F_1 .. F_4.
__device__ __forceinline__ f2 rest_weight2(const ff2& rho, const ff2& sum, const DvmConst<float>& d) {
  const ff2 f0 = ff2_add(ff2_of(bc2(1.f)), ff2_mul(ff2_of(bc2(-d.B0)), sum));   // F_0
  return ff2_round(ff2_mul(rho, f0));
}

// Everything but the weights.
__device__ __forceinline__ void eq2_polynomial(const State2& s, Eq2& q) {
  const ff2 invE = ff2_recip(s.E);
  const ff2 uxE = ff2_mul(s.ux, invE), uyE = ff2_mul(s.uy, invE);
  const ff2 u2E = ff2_add(ff2_mul(s.ux, uxE), ff2_mul(s.uy, uyE));   // u^2 / E
  const ff2 a1 = ff2_add(ff2_of(bc2(1.f)), ff2_scale(u2E, -0.5f));
  const ff2 a0 = ff2_add(a1, ff2_scale(ff2_mul(u2E, u2E), 0.125f));
  q.a1 = ff2_round(a1);
  q.a0 = ff2_round(a0);
  q.a1h = mul2(bc2(0.5f), q.a1);
  const ff2 sq = ffc(kS, kSl);
  const ff2 y1 = ff2_mul(sq, ff2_add(uxE, uyE));
  const ff2 y3 = ff2_mul(sq, ff2_add(uyE, ff2{neg2(uxE.hi), neg2(uxE.lo)}));
  q.yh[0] = uxE.hi; q.yl[0] = uxE.lo;
  q.yh[1] = y1.hi;  q.yl[1] = y1.lo;
  q.yh[2] = uyE.hi; q.yl[2] = uyE.lo;
  q.yh[3] = y3.hi;  q.yl[3] = y3.lo;
}

__device__ __forceinline__ Eq2 eq2(const State2& s, const DvmConst<float>& d) {
  Eq2 q;
  ff2 sum = ff2_of(bc2(0.f));
#pragma unroll
  for (int k = 1; k <= 4; ++k) {
    const ff2 a = shell_weight2(s.E, d, k);
    sum = ff2_add(sum, a);
    q.w[k] = ff2_round(ff2_mul(s.rho, a));
  }
  q.w[0] = rest_weight2(s.rho, sum, d);
  eq2_polynomial(s, q);
  return q;
}

// Equilibrium (Eq. 10) of direction i of a shell (speed sh + sl, weight wk =
// rho F_k) and of its opposite direction: with x = v.u/E, P(+x) = ev + od and
// P(-x) = ev - od share the even and odd parts of the polynomial; the pair
// is formed as w ev +- w od with fused multiply-adds.
__device__ __forceinline__ void feq_pair2(const Eq2& eq, f2 sh, f2 sl, int i, f2 wk, f2& fp, f2& fm) {
  const f2 x = fma2(sh, eq.yh[i], fma2(sh, eq.yl[i], mul2(sl, eq.yh[i])));
  const f2 x2 = mul2(x, x);
  const f2 ev = fma2(x2, fma2(x2, bc2(1.0f / 24.0f), eq.a1h), eq.a0);
  const f2 od = mul2(x, fma2(x2, bc2(1.0f / 6.0f), eq.a1));
  const f2 wev = mul2(wk, ev);                     // w (ev +- od) with one rounding after w ev
  fp = fma2(wk, od, wev);
  fm = fma2(neg2(wk), od, wev);
}

// Sums over one shell (plus, optionally, a second shell added direction by
// direction) of f, c_x f and c_y f for both nodes, with the octagon's exact
// unit vectors as float-float constants.  ld(q): the two nodes' f_q.
template <int K, int KADD, class LD>
__device__ __forceinline__ void shell_sums2(LD ld, f2& S, f2& X, f2& Xl, f2& Y, f2& Yl) {
  S = bc2(0.f); X = bc2(0.f); Xl = bc2(0.f); Y = bc2(0.f); Yl = bc2(0.f);
#pragma unroll
  for (int i = 0; i < kHalf; ++i) {
    const int q = 1 + (K - 1) * kNDirs + i;
    f2 fa = ld(q), fb = ld(q + kHalf);
    if (KADD > 0) {
      const int qa = 1 + (KADD - 1) * kNDirs + i;
      fa = add2(fa, ld(qa));
      fb = add2(fb, ld(qa + kHalf));
    }
    S = add2(S, add2(fa, fb));
    const f2 dd = sub2(fa, fb);
    if (i == 0) {
      X = add2(X, dd);
    } else if (i == 2) {
      Y = add2(Y, dd);
    } else {
      const float sx = i == 1 ? 1.f : -1.f;
      X = fma2(bc2(sx * kS), dd, X);
      Xl = fma2(bc2(sx * kSl), dd, Xl);
      Y = fma2(bc2(kS), dd, Y);
      Yl = fma2(bc2(kSl), dd, Yl);
    }
  }
}

// What one group of shells adds to the moments (Eqs. 3-5) of the two nodes.
// Groups: 0 shell 1; 1 shells 2 + 3 direction by direction, with the speed and
// v^2/2 of shell 2; 2 shell 3 again with the differences v_3 - v_2, (v_3^2 -
// v_2^2)/2 (S then does not enter rho); 3 shell 4.
struct Terms2 {
  f2 S;
  ff2 jx, jy, e;
};
template <int G, class LD>
__device__ __forceinline__ Terms2 group_terms2(LD ld, const DvmConst<float>& d) {
  f2 S, X, Xl, Y, Yl;
  shell_sums2<G == 0 ? 1 : (G == 1 ? 2 : (G == 2 ? 3 : 4)), G == 1 ? 3 : 0>(ld, S, X, Xl, Y, Yl);
  constexpr int k = G == 0 ? 1 : (G == 1 ? 2 : 4);
  const ff2 v = G == 2 ? ffc(d.dv23, d.dv23_lo) : ffc(d.speed[k], d.speed_lo[k]);
  const ff2 h = G == 2 ? ffc(d.dh23, d.dh23_lo) : ffc(d.half_v2[k], d.half_v2_lo[k]);
  return Terms2{S, ff2_mul(v, ff2{X, Xl}), ff2_mul(v, ff2{Y, Yl}), ff2_mul(h, ff2_of(S))};
}

// Adds the groups up in order and recovers velocity and temperature.
struct Moments2 {
  ff2 rho, jx, jy, e;
  __device__ __forceinline__ explicit Moments2(f2 f0) : rho(ff2_of(f0)), jx(ff2_of(bc2(0.f))), jy(jx), e(jx) {}
  template <int G>
  __device__ __forceinline__ void add(const Terms2& t) {
    if (G != 2) rho = ff2_add(rho, ff2_of(t.S));
    jx = ff2_add(jx, t.jx);
    jy = ff2_add(jy, t.jy);
    e = ff2_add(e, t.e);
  }
  __device__ __forceinline__ State2 state() const {
    State2 s;
    const ff2 inv = ff2_recip(rho);
    s.rho = rho;
    s.ux = ff2_mul(jx, inv);
    s.uy = ff2_mul(jy, inv);
    const ff2 ke = ff2_add(ff2_mul(jx, s.ux), ff2_mul(jy, s.uy));    // |j|^2 / rho
    s.E = ff2_mul(ff2_add(e, ff2_scale(ke, -0.5f)), inv);
    return s;
  }
};

}  // namespace pclb
