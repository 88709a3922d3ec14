// The field kernels (both precisions) for the larger velocity sets of Table I,
// N_i = 16 and 24 directions per shell (Q = 65, 97): the same model (Eqs. 2-5,
// 10-11), one thread per node, the moments, the temperature and the equilibrium
// factors in double (FP32: gen_state.cuh, the equilibrium in float-float).  These sets serve the
// paper's velocity-set comparison; their steps are dvm_step_f64.cu and the tiled
// FP32 kernel of dvm_tiled32.cu.  The azimuthal ghost rows (Eq. 40) are stored
// rows, written by the producer of the seam rows with the label rotation, as in
// the rest of the library.
#include <algorithm>
#include <cfloat>
#include <cmath>
#include <cstddef>
#include <cuda_runtime.h>

#include "copy_rows.cuh"
#include "dvm_generic.h"
#include "f32_state.cuh"
#include "gen_state.cuh"
#include "pclb_internal.h"

namespace pclb {

namespace {

constexpr int kGenThreads = 128;

// Moments (Eqs. 3-5): rho = sum f, rho u = sum f v, rho (E + u^2/2) = sum f
// v^2/2, over the pairs of opposite velocities (2.5 FP64 operations per label
// instead of 4; FP64 issue bounds every caller).
__device__ GenState gen_moments_node(const double* f, size_t plane, const DvmG& d) {
  const int half = d.n_dirs / 2;
  double s0 = f[0], sx = 0.0, sy = 0.0, se = 0.0;
  for (int k = 1; k <= 4; ++k) {
    double S = 0.0;
#pragma unroll 4
    for (int i = 0; i < half; ++i) {
      const int q = 1 + (k - 1) * d.n_dirs + i;
      const double a = f[(size_t)q * plane], b = f[(size_t)(q + half) * plane];
      S += a + b;
      sx = fma(d.vx[q], a - b, sx);
      sy = fma(d.vy[q], a - b, sy);
    }
    s0 += S;
    se = fma(d.half_v2[k], S, se);
  }
  return gen_state_of(s0, sx, sy, se);
}

// Store of label q at interior node (t, r), and of the azimuthal ghost rows
// of the receiving labels when t is a seam row (Eq. 40).
template <class T>
__device__ __forceinline__ void gen_store(T* f, const StepParams& p, const DvmG& d, int q, int t, int r, T v) {
  const size_t plane = (size_t)p.rows * p.pitch;
  f[(size_t)q * plane + (size_t)(t + kGhostRows) * p.pitch + r] = v;
  if (t >= p.n_theta - 2)
    f[(size_t)d.recv_lo[q] * plane + (size_t)(t - (p.n_theta - 2)) * p.pitch + r] = v;
  if (t < 2) f[(size_t)d.recv_hi[q] * plane + (size_t)(p.n_theta + kGhostRows + t) * p.pitch + r] = v;
}

// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(kGenThreads)
    gen_moments_kernel(const double* __restrict__ f, double* rho, double* u_r, double* u_t, double* temp,
                       const __grid_constant__ StepParams p, const __grid_constant__ DvmG d) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int t = blockIdx.y;
  if (r >= p.n_r) return;
  const size_t plane = (size_t)p.rows * p.pitch;
  const GenState m = gen_moments_node(f + (size_t)(t + kGhostRows) * p.pitch + r, plane, d);
  const size_t n = (size_t)t * p.n_r + r;
  const double c = p.cos_t[t], s = p.sin_t[t];
  if (rho) rho[n] = m.rho;
  if (u_r) u_r[n] = m.ux * c + m.uy * s;
  if (u_t) u_t[n] = m.uy * c - m.ux * s;
  if (temp) temp[n] = m.E;
}

// f^eq of one node in double, rounded once per label: fields outside the range of
// the float-float form below.
static __device__ __noinline__ void gen_set_node(float* f, const StepParams& p, const DvmG& d, int t, int r, double R,
                                                 double ur, double ut, double E) {
  const double c = p.cos_t[t], s = p.sin_t[t], ux = ur * c - ut * s, uy = ur * s + ut * c;
  const double uxE = ux / E, uyE = uy / E, u2E = (ux * ux + uy * uy) / E;
  const double a1 = 1.0 - 0.5 * u2E, a0 = a1 + 0.125 * u2E * u2E;
  double Fs = 0.0;
#pragma unroll 1
  for (int q = 4 * d.n_dirs; q >= 0; --q) {   // the rest velocity last: F_0 = 1 - B0 (F_1 + .. + F_4)
    const int k = d.shell[q];
    const double F = k == 0 ? 1.0 - d.B0 * Fs
                            : E * (d.Fc[k][0] + E * (d.Fc[k][1] + E * (d.Fc[k][2] + E * d.Fc[k][3])));
    if (k > 0 && q == 1 + (k - 1) * d.n_dirs) Fs += F;
    const double x = d.vx[q] * uxE + d.vy[q] * uyE;
    gen_store<float>(f, p, d, q, t, r, (float)(R * F * (a0 + x * (a1 + x * (0.5 * a1 + x * (1.0 / 6.0 + x * (1.0 / 24.0)))))));
  }
}

// FP32 storage: f = f^eq of the fields, evaluated in float-float and rounded
// once per label.  Per node and shell the polynomial of Eq. (10) in x = v_k
// y_i, y_i = c_i.u/E, is folded into w ev = A + y^2 (B + y^2 C) and w od = y
// (O1 + y^2 O3), so that a pair of opposite velocities takes three multiply-adds,
// a product and two rounded sums.
template <int ND>
__global__ void __launch_bounds__(kGenThreads)
    gen_set_state_f32_kernel(float* __restrict__ f, const float* __restrict__ rho, const float* __restrict__ u_r,
                             const float* __restrict__ u_t, const float* __restrict__ temp,
                             const __grid_constant__ StepParams p, const __grid_constant__ DvmG d,
                             const __grid_constant__ DvmG32 c) {
  constexpr int H = ND / 2;
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int t = blockIdx.y;
  if (r >= p.n_r) return;
  const size_t n = (size_t)t * p.n_r + r;
  const ff R = ff_of(rho[n]), E = ff_of(temp[n]), ur = ff_of(u_r[n]), ut = ff_of(u_t[n]);   // E = T
  if (!(R.hi > 0.f && E.hi > 0.f)) atomicOr(p.status, PCLB_FLAG_NONPHYS);
  // the low parts stay normal numbers or nearly so, and nothing overflows
  if (!(R.hi >= 0x1p-60f && R.hi <= 0x1p+60f && E.hi >= 0x1p-20f && E.hi <= 0x1p+10f &&
        ur.hi * ur.hi + ut.hi * ut.hi <= 256.f * E.hi)) {
    gen_set_node(f, p, d, t, r, R.hi, ur.hi, ut.hi, E.hi);
    return;
  }
  const float4 cs = p.cs_ff[t];
  const ff co{cs.x, cs.y}, si{cs.z, cs.w};
  const ff ux = ff_add(ff_mul(ur, co), ff_neg(ff_mul(ut, si))), uy = ff_add(ff_mul(ur, si), ff_mul(ut, co));
  const ff invE = ff_recip(E);
  const ff uxE = ff_mul(ux, invE), uyE = ff_mul(uy, invE);
  const ff u2E = ff_add(ff_mul(ux, uxE), ff_mul(uy, uyE));   // u^2 / E
  const ff a1 = ff_add(ff_of(1.f), ff_scale(u2E, -0.5f));
  const ff a0 = ff_add(a1, ff_scale(ff_mul(u2E, u2E), 0.125f));
  ff sum = ff_of(0.f);
  ff A[4], B[4], C[4], O1[4], O3[4];
  const ff sixth{1.0f / 6.0f, (float)(1.0 / 6.0 - (double)(1.0f / 6.0f))};
#pragma unroll
  for (int k = 1; k <= 4; ++k) {
    ff F{c.Fch[k][3], c.Fcl[k][3]};
#pragma unroll
    for (int j = 2; j >= 0; --j) F = ff_mul_add(F, E, ff{c.Fch[k][j], c.Fcl[k][j]});
    F = ff_mul(F, E);
    sum = ff_add(sum, F);
    const ff w = ff_mul(R, F), v{c.sph[k], c.spl[k]}, wv = ff_mul(w, v), hv{c.hvh[k], c.hvl[k]};   // hv = v^2/2
    A[k - 1] = ff_mul(w, a0);
    B[k - 1] = ff_mul(ff_mul(w, hv), a1);
    O1[k - 1] = ff_mul(wv, a1);
    O3[k - 1] = ff_scale(ff_mul(ff_mul(wv, hv), sixth), 2.f);            // w v^3 / 6
    C[k - 1] = ff_mul(ff_mul(ff_mul(w, hv), hv), sixth);                  // w v^4 / 24
  }
  const ff w0 = ff_mul(R, ff_add(ff_of(1.f), ff_mul(ff{-c.B0h, -c.B0l}, sum)));
  const ff f0 = ff_mul(w0, a0);
  const size_t plane = (size_t)p.rows * p.pitch;
  float* row = f + (size_t)(t + kGhostRows) * p.pitch + r;
  const bool seam = t < 2 || t >= p.n_theta - 2;   // the row also feeds azimuthal ghost rows
  auto put = [&](int q, float v) {
    if (seam) gen_store<float>(f, p, d, q, t, r, v);
    else row[(size_t)q * plane] = v;
  };
  put(0, f0.hi + f0.lo);
#pragma unroll 1
  for (int i = 0; i < H; ++i) {
    const ff y = ff_add(ff_mul(ff{c.cxh[i], c.cxl[i]}, uxE), ff_mul(ff{c.cyh[i], c.cyl[i]}, uyE));
    const ff y2 = ff_mul(y, y);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const ff ev = ff_mul_add(y2, ff_mul_add(y2, C[k], B[k]), A[k]);
      const ff od = ff_mul(y, ff_mul_add(y2, O3[k], O1[k]));
      float h, e;
      two_sum(ev.hi, od.hi, h, e);
      put(1 + k * ND + i, h + (e + (ev.lo + od.lo)));
      two_sum(ev.hi, -od.hi, h, e);
      put(1 + k * ND + i + H, h + (e + (ev.lo - od.lo)));
    }
  }
}

template <int ND>
__global__ void __launch_bounds__(kGenThreads)
    gen_moments_f32_kernel(const float* __restrict__ f, float* rho, float* u_r, float* u_t, float* temp,
                           const __grid_constant__ StepParams p, const __grid_constant__ DvmG d,
                           const __grid_constant__ DvmG32 c) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int t = blockIdx.y;
  if (r >= p.n_r) return;
  const size_t plane = (size_t)p.rows * p.pitch;
  const float* fn = f + (size_t)(t + kGhostRows) * p.pitch + r;
  const size_t n = (size_t)t * p.n_r + r;
  const State32 s = gen_state32<ND>(fn, plane, c);
  if (gen_in_range(s)) {
    const float4 cs = p.cs_ff[t];
    const ff co{cs.x, cs.y}, si{cs.z, cs.w};
    auto put = [&](float* o, ff x) {
      if (o) o[n] = x.hi + x.lo;
    };
    put(rho, s.rho);
    put(u_r, ff_add(ff_mul(s.ux, co), ff_mul(s.uy, si)));
    put(u_t, ff_add(ff_mul(s.uy, co), ff_neg(ff_mul(s.ux, si))));
    put(temp, s.E);
    return;
  }
  const GenState m = gen_state_f32<ND>(fn, plane, d, c);
  const double co = p.cos_t[t], si = p.sin_t[t];
  if (rho) rho[n] = (float)m.rho;
  if (u_r) u_r[n] = (float)(m.ux * co + m.uy * si);
  if (u_t) u_t[n] = (float)(m.uy * co - m.ux * si);
  if (temp) temp[n] = (float)m.E;
}

// Global integrals with weight r dr dtheta (as pclb_diagnostics): per block a
// fixed grid-stride subset in a fixed order, the blocks' partials by six warps
// (diag_final_kernel).  The node state in double.
template <int ND>
__device__ __forceinline__ GenState gen_diag_state(const double* f, size_t plane, const DvmG& d, const DvmG32&) {
  return gen_moments_node(f, plane, d);
}
template <int ND>
__device__ __forceinline__ GenState gen_diag_state(const float* f, size_t plane, const DvmG& d, const DvmG32& c) {
  return gen_state_int<ND>(f, plane, d, c);
}

template <class T, int ND>
__global__ void __launch_bounds__(kGenThreads)
    gen_diag_partial_kernel(const T* __restrict__ f, double* partials, const __grid_constant__ StepParams p,
                            const __grid_constant__ DvmG d, const __grid_constant__ DvmG32 c, double dr, double dth,
                            double r_in) {
  const size_t plane = (size_t)p.rows * p.pitch;
  const size_t n_nodes = (size_t)p.n_r * p.n_theta;
  double v[6] = {0, 0, 0, 0, DBL_MAX, DBL_MAX};
  for (size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x; n < n_nodes; n += (size_t)gridDim.x * blockDim.x) {
    const int t = (int)(n / p.n_r), r = (int)(n % p.n_r);
    const GenState m = gen_diag_state<ND>(f + (size_t)(t + kGhostRows) * p.pitch + r, plane, d, c);
    const double w = (r_in + r * dr) * dr * dth * m.rho;
    v[0] += w;
    v[1] = fma(w, m.ux, v[1]);
    v[2] = fma(w, m.uy, v[2]);
    v[3] = fma(w, fma(0.5, m.ux * m.ux + m.uy * m.uy, m.E), v[3]);
    v[4] = fmin(v[4], m.rho);
    v[5] = fmin(v[5], m.E);
  }
  __shared__ double red[6][kGenThreads / 32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = 0; i < 6; ++i) {
    for (int off = 16; off > 0; off >>= 1) {
      const double o = __shfl_down_sync(0xffffffffu, v[i], off);
      v[i] = i < 4 ? v[i] + o : fmin(v[i], o);
    }
    if (lane == 0) red[i][warp] = v[i];
  }
  __syncthreads();
  if (threadIdx.x == 0)
    for (int i = 0; i < 6; ++i) {
      double s = red[i][0];
      for (int w = 1; w < kGenThreads / 32; ++w) s = i < 4 ? s + red[i][w] : fmin(s, red[i][w]);
      partials[(size_t)blockIdx.x * 8 + i] = s;
    }
}

}  // namespace

template <class T>
cudaError_t gen_launch_set_state(T* f, const T* rho, const T* ur, const T* ut, const T* temp, const StepParams& p,
                                 const DvmG& d, const DvmG32& c, cudaStream_t s) {
  const dim3 grid((p.n_r + kGenThreads - 1) / kGenThreads, p.n_theta);
  if constexpr (sizeof(T) == 8)
    return gen_launch_set_state_f64(f, rho, ur, ut, temp, p, d, s);
  else if (d.n_dirs == 16)
    gen_set_state_f32_kernel<16><<<grid, kGenThreads, 0, s>>>(f, rho, ur, ut, temp, p, d, c);
  else
    gen_set_state_f32_kernel<24><<<grid, kGenThreads, 0, s>>>(f, rho, ur, ut, temp, p, d, c);
  return cudaGetLastError();
}

template <class T>
cudaError_t gen_launch_moments(const T* f, T* rho, T* ur, T* ut, T* temp, const StepParams& p, const DvmG& d,
                               const DvmG32& c, cudaStream_t s) {
  const dim3 grid((p.n_r + kGenThreads - 1) / kGenThreads, p.n_theta);
  if constexpr (sizeof(T) == 8)
    gen_moments_kernel<<<grid, kGenThreads, 0, s>>>(f, rho, ur, ut, temp, p, d);
  else if (d.n_dirs == 16)
    gen_moments_f32_kernel<16><<<grid, kGenThreads, 0, s>>>(f, rho, ur, ut, temp, p, d, c);
  else
    gen_moments_f32_kernel<24><<<grid, kGenThreads, 0, s>>>(f, rho, ur, ut, temp, p, d, c);
  return cudaGetLastError();
}

template <class T>
cudaError_t gen_launch_pack(const T* f, T* out, const StepParams& p, const DvmG& d, cudaStream_t s) {
  return launch_copy_rows<T, false>(f, out, d.q, p, RecvLabels{}, s);
}

template <class T>
cudaError_t gen_launch_unpack(const T* in, T* f, const StepParams& p, const DvmG& d, cudaStream_t s) {
  return launch_copy_rows<T, true>(in, f, d.q, p, recv_labels(d, d.q), s);
}

void fill_dvm_generic32(DvmG32& c, const pclb_dvm& d, const DvmG& g) {
  const int nd = d.n_dirs;
  c = DvmG32{};
  auto split = [](double x, float& hi, float& lo) {
    hi = (float)x;
    lo = (float)(x - (double)hi);
  };
  for (int k = 0; k < 5; ++k) {
    split(d.speeds[k], c.sph[k], c.spl[k]);
    split(g.half_v2[k], c.hvh[k], c.hvl[k]);
    for (int n = 0; n < 4; ++n) split(g.Fc[k][n], c.Fch[k][n], c.Fcl[k][n]);
  }
  split(d.speeds[3] - d.speeds[2], c.dv23h, c.dv23l);
  split(g.half_v2[3] - g.half_v2[2], c.dh23h, c.dh23l);
  split(g.B0, c.B0h, c.B0l);
  for (int i = 0; i < nd / 2; ++i) {
    const double phi = 2.0 * M_PI * i / nd;
    const double u[2] = {std::cos(phi), std::sin(phi)};
    float* hi[2] = {c.cxh, c.cyh};
    float* lo[2] = {c.cxl, c.cyl};
    for (int j = 0; j < 2; ++j) {
      hi[j][i] = (float)u[j];
      lo[j][i] = (float)(u[j] - (double)hi[j][i]);
    }
  }
  {
    // fractions of the power of two above the largest speed; cos and sin as they are
    double v = 0.0, hv = 0.0;
    for (int k = 1; k < 5; ++k) {
      v = std::max(v, d.speeds[k]);
      hv = std::max(hv, g.half_v2[k]);
    }
    std::frexp(v, &c.fx_exp_v);
    std::frexp(hv, &c.fx_exp_hv);
    c.fx_ok = std::isfinite(hv) && std::abs(c.fx_exp_v) < 200 && std::abs(c.fx_exp_hv) < 400;
    auto fraction = [](double x) { return (uint64_t)std::nearbyint(std::ldexp(std::fabs(x), 63)); };   // |x| <= 1
    for (int k = 1; k < 5 && c.fx_ok; ++k) {
      c.fx_speed[k - 1] = fraction(std::ldexp(d.speeds[k], -c.fx_exp_v));
      c.fx_half_v2[k - 1] = fraction(std::ldexp(g.half_v2[k], -c.fx_exp_hv));
    }
    for (int i = 0; i < nd / 2; ++i) {
      const double phi = 2.0 * M_PI * i / nd;
      c.fx_cx[i] = fraction(std::cos(phi));
      c.fx_cy[i] = fraction(std::sin(phi));   // >= 0 in the first half
      c.fx_neg_x |= (std::cos(phi) < 0.0 ? 1 : 0) << i;
    }
  }
  // the same velocities as DvmG (opposite directions exactly antisymmetric)
  for (int k = 1; k <= 4; ++k)
    for (int i = 0; i < nd; ++i) {
      const int q = 1 + (k - 1) * nd + i;
      const int ib = i % (nd / 2);
      const double phi = 2.0 * M_PI * ib / nd, sgn = i < nd / 2 ? 1.0 : -1.0;
      c.vx[q] = (float)(d.speeds[k] * sgn * std::cos(phi));
      c.vy[q] = (float)(d.speeds[k] * sgn * std::sin(phi));
    }
}

template <class T>
cudaError_t gen_launch_diagnostics(const T* f, double* partials, double* out, const StepParams& p, const DvmG& d,
                                   const DvmG32& c, double dr, double dth, double r_in, cudaStream_t s) {
  if (d.n_dirs == 16)
    gen_diag_partial_kernel<T, 16><<<kDiagBlocks, kGenThreads, 0, s>>>(f, partials, p, d, c, dr, dth, r_in);
  else
    gen_diag_partial_kernel<T, 24><<<kDiagBlocks, kGenThreads, 0, s>>>(f, partials, p, d, c, dr, dth, r_in);
  const cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : launch_diag_final(partials, kDiagBlocks, out, (double)p.n_r * p.n_theta, s);
}

#define PCLB_GEN_INSTANTIATE(T)                                                                               \
  template cudaError_t gen_launch_set_state<T>(T*, const T*, const T*, const T*, const T*, const StepParams&, \
                                               const DvmG&, const DvmG32&, cudaStream_t);                     \
  template cudaError_t gen_launch_moments<T>(const T*, T*, T*, T*, T*, const StepParams&, const DvmG&,        \
                                             const DvmG32&, cudaStream_t);                                    \
  template cudaError_t gen_launch_pack<T>(const T*, T*, const StepParams&, const DvmG&, cudaStream_t);        \
  template cudaError_t gen_launch_unpack<T>(const T*, T*, const StepParams&, const DvmG&, cudaStream_t);      \
  template cudaError_t gen_launch_diagnostics<T>(const T*, double*, double*, const StepParams&, const DvmG&,  \
                                                 const DvmG32&, double, double, double, cudaStream_t);
PCLB_GEN_INSTANTIATE(float)
PCLB_GEN_INSTANTIATE(double)

}  // namespace pclb
