// Non-equilibrium manifestations of Sec. IV.
//
// For the weights w_q = f_q (moments) or w_q = f_q - f^eq_q (departures) and
// the velocities c_q = v_q (plain) or c_q = v_q - u (central), in polar
// components at the node, the groups are
//   M_2 = sum w c c (rr, r theta, theta theta),
//   M_3 = sum w c c c (rrr, rr theta, r theta theta, theta theta theta),
//   M_{3,1} = sum w (c.c/2) c (r, theta),
//   M_{4,2} = sum w (c.c/2) c c (rr, r theta, theta theta),
// for each requested group: M_m(f), Delta_m = M_m(f - f^eq), M*_m(f) and
// Delta*_m = M*_m(f - f^eq).
//
// One pass accumulates the 12 central moments M*_m(f) of the node.  The
// others follow per node:
//   * Delta*_m = M*_m(f) - M*_m(f^eq), and the central moments of the model's
//     equilibrium are those of the Maxwellian, (rho E I, 0, 0, 2 rho E^2 I)
//     (the relations the velocity set is built to satisfy, Eqs. 6-9);
//   * the plain moments from the central ones with v = u + c: with
//     S = M*_2, T = M*_3, V = M*_{3,1}, Q = M*_{4,2} and sum w c = 0,
//       M_2 = S + rho u u,
//       M_3 = T + (u S + S u + ...: the three placements of u) + rho u u u,
//       M_{3,1} = V + S u + u tr(S)/2 + rho u |u|^2/2,
//       M_{4,2} = Q + u V + V u + u.T + u u tr(S)/2 + u (S u) + (S u) u
//                 + |u|^2/2 S + rho |u|^2/2 u u;
//     the departures the same way from Delta*_m with rho replaced by
//     sum (f - f^eq) = 0 (f and f^eq share mass, momentum and energy).
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "dvm_generic.h"
#include "f32_eq2.cuh"
#include "f32_state.cuh"
#include "gen_state.cuh"
#include "pclb_internal.h"

namespace pclb {

namespace {

constexpr int kNeqThreads = 128;

// Plain moments (12 components, order as above) from central ones C with
// density R (0 for departures) and velocity (ur, ut), polar components.
template <class T>
__device__ __forceinline__ void plain_from_central(T R, T ur, T ut, const T* C, T* M) {
  const T Srr = C[0], Srt = C[1], Stt = C[2];
  const T Trrr = C[3], Trrt = C[4], Trtt = C[5], Tttt = C[6];
  const T Vr = C[7], Vt = C[8];
  const T trS2 = T(0.5) * (Srr + Stt);
  const T u2 = T(0.5) * (ur * ur + ut * ut);
  const T Sur = Srr * ur + Srt * ut, Sut = Srt * ur + Stt * ut;   // S u
  M[0] = Srr + R * ur * ur;
  M[1] = Srt + R * ur * ut;
  M[2] = Stt + R * ut * ut;
  M[3] = Trrr + T(3) * ur * Srr + R * ur * ur * ur;
  M[4] = Trrt + T(2) * ur * Srt + ut * Srr + R * ur * ur * ut;
  M[5] = Trtt + ur * Stt + T(2) * ut * Srt + R * ur * ut * ut;
  M[6] = Tttt + T(3) * ut * Stt + R * ut * ut * ut;
  M[7] = Vr + Sur + ur * trS2 + R * ur * u2;
  M[8] = Vt + Sut + ut * trS2 + R * ut * u2;
  // u.T for the pairs (rr, rt, tt): u_r T_r.. + u_t T_t..
  const T uTrr = ur * Trrr + ut * Trrt, uTrt = ur * Trrt + ut * Trtt, uTtt = ur * Trtt + ut * Tttt;
  M[9] = C[9] + T(2) * ur * Vr + uTrr + ur * ur * trS2 + T(2) * ur * Sur + u2 * Srr + R * u2 * ur * ur;
  M[10] = C[10] + ur * Vt + ut * Vr + uTrt + ur * ut * trS2 + ur * Sut + ut * Sur + u2 * Srt + R * u2 * ur * ut;
  M[11] = C[11] + T(2) * ut * Vt + uTtt + ut * ut * trS2 + T(2) * ut * Sut + u2 * Stt + R * u2 * ut * ut;
}

}  // namespace

// FP64: one node per thread.
__global__ void __launch_bounds__(kNeqThreads)
    noneq_kernel(const double* __restrict__ f, double* __restrict__ out, int groups,
                 const __grid_constant__ StepParams p, const __grid_constant__ DvmConst<double> d) {
  using T = double;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int t = blockIdx.y;
  if (r >= p.n_r || t >= p.n_theta) return;
  const size_t plane = (size_t)p.rows * p.pitch;
  const T* fn = f + (size_t)(t + kGhostRows) * p.pitch + r;
  const NodeState<T> m = node_moments(fn, plane, d);
  const T rho = m.rho, ux = m.ux, uy = m.uy;
  const T rE = m.rho * m.E, rE2 = 2.0 * m.rho * m.E * m.E;
  if (!m.ok) atomicOr(p.status, PCLB_FLAG_NONPHYS);
  const T cs = (T)p.cos_t[t], sn = (T)p.sin_t[t];
  const T u_r = ux * cs + uy * sn, u_t = uy * cs - ux * sn;

  // central moments of f
  T A[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) A[c] = T(0);
#pragma unroll
  for (int q = 0; q < kQ; ++q) {
    const T w = fn[(size_t)q * plane];
    const T cr = d.vx[q] * cs + d.vy[q] * sn - u_r, ct = d.vy[q] * cs - d.vx[q] * sn - u_t;
    const T h = T(0.5) * (cr * cr + ct * ct);
    const T wr = w * cr, wt = w * ct;
    const T wrr = wr * cr, wrt = wr * ct, wtt = wt * ct;
    A[0] += wrr;
    A[1] += wrt;
    A[2] += wtt;
    A[3] += wrr * cr;
    A[4] += wrr * ct;
    A[5] += wrt * ct;
    A[6] += wtt * ct;
    A[7] += h * wr;
    A[8] += h * wt;
    A[9] += h * wrr;
    A[10] += h * wrt;
    A[11] += h * wtt;
  }
  // central departures: minus the equilibrium's (rho E I, 0, 0, 2 rho E^2 I)
  T D[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) D[c] = A[c];
  D[0] = A[0] - rE;
  D[2] = A[2] - rE;
  D[9] = A[9] - rE2;
  D[11] = A[11] - rE2;

  const size_t nodes = (size_t)p.n_theta * p.n_r, n = (size_t)t * p.n_r + r;
  int slot = 0;
  T out_g[12];
#pragma unroll 1
  for (int g = 0; g < 4; ++g) {
    if (!(groups & (1 << g))) continue;
    if (g == 0) plain_from_central<T>(rho, u_r, u_t, A, out_g);
    else if (g == 1) plain_from_central<T>(T(0), u_r, u_t, D, out_g);
    else if (g == 2)
      for (int c = 0; c < 12; ++c) out_g[c] = A[c];
    else
      for (int c = 0; c < 12; ++c) out_g[c] = D[c];
#pragma unroll
    for (int c = 0; c < 12; ++c) out[(size_t)(slot * 12 + c) * nodes + n] = out_g[c];
    ++slot;
  }
}

// FP32: two radially adjacent nodes per thread in packed FP32x2 arithmetic, the
// node state and rho E, 2 rho E^2 in float-float.  Bound: HBM, with issue close
// behind (one node per thread and FP64 for the departures: 156 us on 1024 x
// 2048, all four groups, at 83% issue and half the FP64 pipe).
__global__ void __launch_bounds__(kNeqThreads)
    noneq_f32_kernel(const float* __restrict__ f, float* __restrict__ out, int groups,
                     const __grid_constant__ StepParams p, const __grid_constant__ DvmConst<float> d) {
  const int r = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  const int t = blockIdx.y;
  if (r >= p.n_r || t >= p.n_theta) return;
  const bool v1 = r + 1 < p.n_r;   // the second node exists (else its values, from the row's padding, are not stored)
  const size_t plane = (size_t)p.rows * p.pitch;
  const float* fn = f + (size_t)(t + kGhostRows) * p.pitch + r;
  auto ld = [&](int q) { return __ldg(reinterpret_cast<const float2*>(fn + (size_t)q * plane)); };
  Moments2 m(ld(0));
  m.add<0>(group_terms2<0>(ld, d));
  m.add<1>(group_terms2<1>(ld, d));
  m.add<2>(group_terms2<2>(ld, d));
  m.add<3>(group_terms2<3>(ld, d));
  const State2 st = m.state();
  auto physical = [](float rho, float E, float e, float jx, float jy) {
    return rho > 0.f && E > 0.f && isfinite(e) && isfinite(jx) && isfinite(jy);
  };
  if (!physical(m.rho.hi.x, st.E.hi.x, m.e.hi.x, m.jx.hi.x, m.jy.hi.x) ||
      (v1 && !physical(m.rho.hi.y, st.E.hi.y, m.e.hi.y, m.jx.hi.y, m.jy.hi.y)))
    atomicOr(p.status, PCLB_FLAG_NONPHYS);
  const f2 ux = ff2_round(st.ux), uy = ff2_round(st.uy), rho = ff2_round(st.rho);
  const float cs = (float)p.cos_t[t], sn = (float)p.sin_t[t];
  const f2 u_r = fma2(ux, bc2(cs), mul2(uy, bc2(sn))), u_t = fma2(uy, bc2(cs), neg2(mul2(ux, bc2(sn))));

  // central moments of f
  f2 A[12];
#pragma unroll
  for (int c = 0; c < 12; ++c) A[c] = bc2(0.f);
#pragma unroll
  for (int q = 0; q < kQ; ++q) {
    const f2 w = ld(q);
    const f2 cr = sub2(bc2(fmaf(d.vx[q], cs, d.vy[q] * sn)), u_r), ct = sub2(bc2(fmaf(d.vy[q], cs, -(d.vx[q] * sn))), u_t);
    const f2 h = mul2(bc2(0.5f), fma2(cr, cr, mul2(ct, ct)));
    const f2 wr = mul2(w, cr), wt = mul2(w, ct);
    const f2 wrr = mul2(wr, cr), wrt = mul2(wr, ct), wtt = mul2(wt, ct);
    A[0] = add2(A[0], wrr);
    A[1] = add2(A[1], wrt);
    A[2] = add2(A[2], wtt);
    A[3] = fma2(wrr, cr, A[3]);
    A[4] = fma2(wrr, ct, A[4]);
    A[5] = fma2(wrt, ct, A[5]);
    A[6] = fma2(wtt, ct, A[6]);
    A[7] = fma2(h, wr, A[7]);
    A[8] = fma2(h, wt, A[8]);
    A[9] = fma2(h, wrr, A[9]);
    A[10] = fma2(h, wrt, A[10]);
    A[11] = fma2(h, wtt, A[11]);
  }
  // central departures: minus the equilibrium's (rho E I, 0, 0, 2 rho E^2 I), in
  // double where the float-float products have no room
  const ff2 rE = ff2_mul(st.rho, st.E), rE2 = ff2_scale(ff2_mul(rE, st.E), 2.f);
  auto less = [](f2 a, ff2 b) { return sub2(sub2(a, b.hi), b.lo); };
  f2 D0 = less(A[0], rE), D2 = less(A[2], rE), D9 = less(A[9], rE2), D11 = less(A[11], rE2);
  auto room = [](float x, float y) { return x >= 0x1p-96f && y >= 0x1p-96f && x <= 0x1p+120f && y <= 0x1p+120f; };
  if (!(room(rE.hi.x, rE2.hi.x) && room(rE.hi.y, rE2.hi.y))) {
    auto exact = [](ff rho, ff E, float a0, float a2, float a9, float a11, float& d0, float& d2, float& d9, float& d11) {
      const double R = (double)rho.hi + rho.lo, e = (double)E.hi + E.lo, x = R * e, y = 2.0 * R * e * e;
      d0 = (float)(a0 - x);
      d2 = (float)(a2 - x);
      d9 = (float)(a9 - y);
      d11 = (float)(a11 - y);
    };
    exact(ff{st.rho.hi.x, st.rho.lo.x}, ff{st.E.hi.x, st.E.lo.x}, A[0].x, A[2].x, A[9].x, A[11].x, D0.x, D2.x, D9.x, D11.x);
    exact(ff{st.rho.hi.y, st.rho.lo.y}, ff{st.E.hi.y, st.E.lo.y}, A[0].y, A[2].y, A[9].y, A[11].y, D0.y, D2.y, D9.y, D11.y);
  }

  const size_t nodes = (size_t)p.n_theta * p.n_r;
  float* o = out + (size_t)t * p.n_r + r;
  const bool wide = v1 && (reinterpret_cast<uintptr_t>(o) & 7) == 0 && (nodes & 1) == 0;
  auto put = [&](int c, float x, float y) {
    float* oc = o + (size_t)c * nodes;
    if (wide) {
      *reinterpret_cast<float2*>(oc) = make_float2(x, y);
    } else {
      oc[0] = x;
      if (v1) oc[1] = y;
    }
  };
  int slot = 0;
#pragma unroll 1
  for (int g = 0; g < 4; ++g) {
    if (!(groups & (1 << g))) continue;
    const bool dep = (g & 1) != 0;
    float X[12], Y[12];
#pragma unroll
    for (int c = 0; c < 12; ++c) { X[c] = A[c].x; Y[c] = A[c].y; }
    if (dep) {
      X[0] = D0.x; X[2] = D2.x; X[9] = D9.x; X[11] = D11.x;
      Y[0] = D0.y; Y[2] = D2.y; Y[9] = D9.y; Y[11] = D11.y;
    }
    if (g < 2) {
      float PX[12], PY[12];
      plain_from_central<float>(dep ? 0.f : rho.x, u_r.x, u_t.x, X, PX);
      plain_from_central<float>(dep ? 0.f : rho.y, u_r.y, u_t.y, Y, PY);
#pragma unroll
      for (int c = 0; c < 12; ++c) put(slot * 12 + c, PX[c], PY[c]);
    } else {
#pragma unroll
      for (int c = 0; c < 12; ++c) put(slot * 12 + c, X[c], Y[c]);
    }
    ++slot;
  }
}

// The same for the N_i = 16 and 24 sets of Table I (Q = 65, 97, built to
// reproduce the same equilibrium moments, Eqs. 6-9): the node's moments in
// double (FP32 storage: gen_state.cuh), the central moments in the storage type
// with the velocities of the set (float tables for FP32).
template <class T, int ND>
__global__ void __launch_bounds__(kNeqThreads)
    noneq_gen_kernel(const T* __restrict__ f, T* __restrict__ out, int groups, const __grid_constant__ StepParams p,
                     const __grid_constant__ DvmG d, const __grid_constant__ DvmG32 c) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int t = blockIdx.y;
  if (r >= p.n_r || t >= p.n_theta) return;
  const size_t plane = (size_t)p.rows * p.pitch;
  const T* fn = f + (size_t)(t + kGhostRows) * p.pitch + r;
  // rho, rho u, rho (E + u^2/2) (Eqs. 3-5), then u and E
  double s0, uxd, uyd, E;
  if constexpr (sizeof(T) == 4) {
    const State32 m = gen_state32<ND>(fn, plane, c);
    if (gen_in_range(m)) {
      s0 = (double)m.rho.hi + m.rho.lo;
      uxd = (double)m.ux.hi + m.ux.lo;
      uyd = (double)m.uy.hi + m.uy.lo;
      E = (double)m.E.hi + m.E.lo;
    } else {
      const GenState x = gen_state_f32<ND>(fn, plane, d, c);
      s0 = x.rho;
      uxd = x.ux;
      uyd = x.uy;
      E = x.E;
    }
  } else {
    double sx = 0.0, sy = 0.0, se = 0.0;
    s0 = 0.0;
    for (int q = 0; q < d.q; ++q) {
      const double v = fn[(size_t)q * plane];
      s0 += v;
      sx = fma(d.vx[q], v, sx);
      sy = fma(d.vy[q], v, sy);
      se = fma(d.half_v2[d.shell[q]], v, se);
    }
    uxd = sx / s0;
    uyd = sy / s0;
    E = (se - 0.5 * (sx * uxd + sy * uyd)) / s0;
  }
  if (!(s0 > 0.0 && E > 0.0 && isfinite(E) && isfinite(uxd) && isfinite(uyd))) atomicOr(p.status, PCLB_FLAG_NONPHYS);
  const double rE = s0 * E, rE2 = 2.0 * s0 * E * E;
  const T rho = (T)s0, ux = (T)uxd, uy = (T)uyd;
  const T cs = (T)p.cos_t[t], sn = (T)p.sin_t[t];
  const T u_r = ux * cs + uy * sn, u_t = uy * cs - ux * sn;

  // central moments of f
  T A[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) A[k] = T(0);
  for (int q = 0; q < d.q; ++q) {
    const T w = fn[(size_t)q * plane];
    T vx, vy;
    if constexpr (sizeof(T) == 4) {
      vx = c.vx[q];
      vy = c.vy[q];
    } else {
      vx = d.vx[q];
      vy = d.vy[q];
    }
    const T cr = vx * cs + vy * sn - u_r, ct = vy * cs - vx * sn - u_t;
    const T h = T(0.5) * (cr * cr + ct * ct);
    const T wr = w * cr, wt = w * ct;
    const T wrr = wr * cr, wrt = wr * ct, wtt = wt * ct;
    A[0] += wrr;
    A[1] += wrt;
    A[2] += wtt;
    A[3] += wrr * cr;
    A[4] += wrr * ct;
    A[5] += wrt * ct;
    A[6] += wtt * ct;
    A[7] += h * wr;
    A[8] += h * wt;
    A[9] += h * wrr;
    A[10] += h * wrt;
    A[11] += h * wtt;
  }
  // central departures: minus the equilibrium's (rho E I, 0, 0, 2 rho E^2 I)
  T D[12];
#pragma unroll
  for (int k = 0; k < 12; ++k) D[k] = A[k];
  D[0] = (T)((double)A[0] - rE);
  D[2] = (T)((double)A[2] - rE);
  D[9] = (T)((double)A[9] - rE2);
  D[11] = (T)((double)A[11] - rE2);

  const size_t nodes = (size_t)p.n_theta * p.n_r, n = (size_t)t * p.n_r + r;
  int slot = 0;
  T out_g[12];
#pragma unroll 1
  for (int g = 0; g < 4; ++g) {
    if (!(groups & (1 << g))) continue;
    if (g == 0) plain_from_central<T>(rho, u_r, u_t, A, out_g);
    else if (g == 1) plain_from_central<T>(T(0), u_r, u_t, D, out_g);
    else if (g == 2)
      for (int k = 0; k < 12; ++k) out_g[k] = A[k];
    else
      for (int k = 0; k < 12; ++k) out_g[k] = D[k];
#pragma unroll
    for (int k = 0; k < 12; ++k) out[(size_t)(slot * 12 + k) * nodes + n] = out_g[k];
    ++slot;
  }
}

template <class T>
cudaError_t launch_noneq_gen(const T* f, T* out, int groups, const StepParams& p, const DvmG& d, const DvmG32& c,
                             cudaStream_t s) {
  dim3 grid((p.n_r + kNeqThreads - 1) / kNeqThreads, p.n_theta);
  if (d.n_dirs == 16)
    noneq_gen_kernel<T, 16><<<grid, kNeqThreads, 0, s>>>(f, out, groups, p, d, c);
  else
    noneq_gen_kernel<T, 24><<<grid, kNeqThreads, 0, s>>>(f, out, groups, p, d, c);
  return cudaGetLastError();
}

template cudaError_t launch_noneq_gen<float>(const float*, float*, int, const StepParams&, const DvmG&, const DvmG32&,
                                             cudaStream_t);
template cudaError_t launch_noneq_gen<double>(const double*, double*, int, const StepParams&, const DvmG&,
                                              const DvmG32&, cudaStream_t);

template <class T>
cudaError_t launch_noneq(const T* f, T* out, int groups, const StepParams& p, const DvmConst<T>& d,
                         cudaStream_t s) {
  constexpr int per = sizeof(T) == 4 ? 2 : 1;   // nodes per thread
  const dim3 grid((p.n_r + per * kNeqThreads - 1) / (per * kNeqThreads), p.n_theta);
  if constexpr (sizeof(T) == 4)
    noneq_f32_kernel<<<grid, kNeqThreads, 0, s>>>(f, out, groups, p, d);
  else
    noneq_kernel<<<grid, kNeqThreads, 0, s>>>(f, out, groups, p, d);
  return cudaGetLastError();
}

template cudaError_t launch_noneq<float>(const float*, float*, int, const StepParams&, const DvmConst<float>&,
                                         cudaStream_t);
template cudaError_t launch_noneq<double>(const double*, double*, int, const StepParams&, const DvmConst<double>&,
                                          cudaStream_t);

}  // namespace pclb
