// Per-node kernels around the step: equilibrium initialisation (f = f^eq of
// given fields, Eq. 10), macroscopic fields out (Eqs. 3-5), copies between
// the packed [Q][n_theta][n_r] layout and the stored layout (with azimuthal
// ghost rows and padded rows), and the global diagnostics reduction.
#include <cuda_runtime.h>
#include <float.h>

#include <algorithm>

#include "copy_rows.cuh"
#include "device_common.cuh"
#include "f32_eq2.cuh"
#include "f32_state.cuh"
#include "pclb_internal.h"

namespace pclb {

constexpr int kDiagThreads32 = 512;   // two blocks per SM, 32 warps

// Write value v of label q at interior row t, column r of the stored layout,
// together with its copies in the azimuthal ghost rows (Eq. 40).
template <class T>
__device__ __forceinline__ void store_with_ghosts(T* f, const StepParams& p, const DvmConst<T>& d,
                                                  int q, int t, int r, T v) {
  const size_t plane = (size_t)p.rows * p.pitch;
  f[(size_t)q * plane + (size_t)(t + kGhostRows) * p.pitch + r] = v;
  if (t >= p.n_theta - 2)
    f[(size_t)d.recv_lo[q] * plane + (size_t)(t - (p.n_theta - 2)) * p.pitch + r] = v;
  if (t < 2) f[(size_t)d.recv_hi[q] * plane + (size_t)(p.n_theta + kGhostRows + t) * p.pitch + r] = v;
}

// FP64 path.  Bound: FP64 issue (see node_moments).  Per shell the polynomial
// of Eq. (10) in x = v_k y_i, y_i = c_i.u/E, is folded into w ev = A + y^2 (B +
// y^2 C) and w od = y (O1 + y^2 O3): six operations per pair of opposite
// velocities, where Horner's rule in x takes seven per label.
__global__ void set_state_kernel(double* __restrict__ f, const double* __restrict__ rho, const double* __restrict__ u_r,
                                 const double* __restrict__ u_t, const double* __restrict__ temp,
                                 const __grid_constant__ StepParams p, const __grid_constant__ DvmConst<double> d,
                                 int t_begin) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int t = blockIdx.y + t_begin;
  if (r >= p.n_r || t >= p.n_theta) return;
  const size_t n = (size_t)t * p.n_r + r;
  const double c = p.cos_t[t], s = p.sin_t[t];
  const double R = rho[n], ur = u_r[n], ut = u_t[n], E = temp[n];  // E = T for gamma = 2
  if (!(R > 0.0 && E > 0.0)) atomicOr(p.status, PCLB_FLAG_NONPHYS);
  const EqParams<double> e = eq_params<double>(R, ur * c - ut * s, ur * s + ut * c, E, d);
  const EqShells64 g = eq_shells(e, d);
  store_with_ghosts<double>(f, p, d, 0, t, r, e.w[0] * e.a0);
#pragma unroll
  for (int i = 0; i < kNDirs / 2; ++i) {
    const double y = g.y[i], y2 = y * y;
#pragma unroll
    for (int k = 1; k <= 4; ++k) {
      const int q = 1 + (k - 1) * kNDirs + i;
      const double ev = fma(y2, fma(y2, g.C[k - 1], g.B[k - 1]), g.A[k - 1]), z = fma(y2, g.O3[k - 1], g.O1[k - 1]);
      store_with_ghosts<double>(f, p, d, q, t, r, fma(y, z, ev));
      store_with_ghosts<double>(f, p, d, q + kNDirs / 2, t, r, fma(-y, z, ev));
    }
  }
}


// FP32 path: two radially adjacent nodes per thread in packed FP32x2
// arithmetic, with the step's float-float equilibrium (eq2, feq_pair2) of the
// given fields; the velocity is rotated to Cartesian components in
// float-float (no FP64 arithmetic), values are stored in pairs.
constexpr int kSetThreads32 = 128;   // 256 nodes of a row per block

__global__ void __launch_bounds__(kSetThreads32)
    set_state_f32_kernel(float* __restrict__ f, const float* __restrict__ rho, const float* __restrict__ u_r,
                         const float* __restrict__ u_t, const float* __restrict__ temp,
                         const __grid_constant__ StepParams p, const __grid_constant__ DvmConst<float> d,
                         int t_begin) {
  const int r = 2 * (blockIdx.x * blockDim.x + threadIdx.x);
  const int t = blockIdx.y + t_begin;
  if (r >= p.n_r || t >= p.n_theta) return;
  const bool v1 = r + 1 < p.n_r;             // the second node exists
  const size_t n = (size_t)t * p.n_r + r;
  auto field = [&](const float* a) { return mk2(a[n], v1 ? a[n + 1] : a[n]); };
  const f2 R = field(rho), E = field(temp);   // E = T for gamma = 2
  if (!(R.x > 0.f && E.x > 0.f && R.y > 0.f && E.y > 0.f)) atomicOr(p.status, PCLB_FLAG_NONPHYS);
  const float4 cs = p.cs_ff[t];
  const ff2 c = ffc(cs.x, cs.y), s = ffc(cs.z, cs.w);
  const ff2 ur = ff2_of(field(u_r)), ut = ff2_of(field(u_t));
  State2 st;
  st.rho = ff2_of(R);
  st.E = ff2_of(E);
  const ff2 uts = ff2_mul(ut, s);
  st.ux = ff2_add(ff2_mul(ur, c), ff2{neg2(uts.hi), neg2(uts.lo)});
  st.uy = ff2_add(ff2_mul(ur, s), ff2_mul(ut, c));
  const Eq2 eq = eq2(st, d);

  const size_t plane = (size_t)p.rows * p.pitch;
  float* row = f + (size_t)(t + kGhostRows) * p.pitch + r;
  float* lo = t >= p.n_theta - 2 ? f + (size_t)(t - (p.n_theta - 2)) * p.pitch + r : nullptr;
  float* hi = t < 2 ? f + (size_t)(p.n_theta + kGhostRows + t) * p.pitch + r : nullptr;
  // label q at this row, and at the azimuthal ghost rows it feeds (Eq. 40)
  auto put = [&](int q, f2 v) {
    auto one = [&](float* base) {
      if (v1)
        *reinterpret_cast<float2*>(base) = v;   // r even, pitch even: 8-byte aligned
      else
        base[0] = v.x;
    };
    one(row + (size_t)q * plane);
    if (lo) one(lo + (size_t)d.recv_lo[q] * plane);
    if (hi) one(hi + (size_t)d.recv_hi[q] * plane);
  };
  put(0, mul2(eq.w[0], eq.a0));
#pragma unroll
  for (int k = 1; k <= 4; ++k) {
    const f2 sh = bc2(d.speed[k]), sl = bc2(d.speed_lo[k]);
#pragma unroll
    for (int i = 0; i < kHalf; ++i) {
      const int q = 1 + (k - 1) * kNDirs + i;
      f2 fp, fm;
      feq_pair2(eq, sh, sl, i, eq.w[k], fp, fm);
      put(q, fp);
      put(q + kHalf, fm);
    }
  }
}

__global__ void moments_f32_kernel(const float* __restrict__ f, float* rho, float* u_r, float* u_t,
                                   float* temp, const __grid_constant__ StepParams p,
                                   const __grid_constant__ DvmConst<float> d, int t_begin) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int t = blockIdx.y + t_begin;
  if (r >= p.n_r || t >= p.n_theta) return;
  const size_t plane = (size_t)p.rows * p.pitch;
  const State32 m = state32(f + (size_t)(t + kGhostRows) * p.pitch + r, plane, d);
  const size_t n = (size_t)t * p.n_r + r;
  // polar components in float-float, rounded once (no FP64 arithmetic)
  const float4 cs = p.cs_ff[t];
  const ff c{cs.x, cs.y}, s{cs.z, cs.w};
  if (rho) rho[n] = m.rho.hi + m.rho.lo;
  if (u_r) u_r[n] = ff_add(ff_mul(m.ux, c), ff_mul(m.uy, s)).hi;
  if (u_t) u_t[n] = ff_add(ff_mul(m.uy, c), ff_neg(ff_mul(m.ux, s))).hi;
  if (temp) temp[n] = m.E.hi + m.E.lo;
}

template <class T>
__global__ void moments_kernel(const T* __restrict__ f, T* rho, T* u_r, T* u_t, T* temp,
                               const __grid_constant__ StepParams p, const __grid_constant__ DvmConst<T> d,
                               int t_begin) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  const int t = blockIdx.y + t_begin;
  if (r >= p.n_r || t >= p.n_theta) return;
  const size_t plane = (size_t)p.rows * p.pitch;
  const NodeState<T> m = node_moments(f + (size_t)(t + kGhostRows) * p.pitch + r, plane, d);
  const size_t n = (size_t)t * p.n_r + r;
  const T c = (T)p.cos_t[t], s = (T)p.sin_t[t];
  if (rho) rho[n] = m.rho;
  if (u_r) u_r[n] = m.ux * c + m.uy * s;
  if (u_t) u_t[n] = m.uy * c - m.ux * s;
  if (temp) temp[n] = m.E;
}

// Block reduction of the six integrals of a block (four sums, two minima) in a
// fixed order, written to the block's partial slot.
__device__ __forceinline__ void diag_block_reduce(const double (&acc)[4], const double (&mn)[2], double* partials) {
  __shared__ double red[6][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double v[6] = {acc[0], acc[1], acc[2], acc[3], mn[0], mn[1]};
#pragma unroll
  for (int i = 0; i < 6; ++i) {
    for (int off = 16; off > 0; off >>= 1) {
      const double o = __shfl_down_sync(0xffffffffu, v[i], off);
      v[i] = i < 4 ? v[i] + o : fmin(v[i], o);
    }
    if (lane == 0) red[i][warp] = v[i];
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    const int nw = blockDim.x / 32, i = threadIdx.x;
    double s = red[i][0];
    for (int w = 1; w < nw; ++w) s = i < 4 ? s + red[i][w] : fmin(s, red[i][w]);
    partials[(size_t)blockIdx.x * 8 + i] = s;
  }
}

// Global integrals with weight r dr dtheta, in double.  Each block reduces a
// fixed grid-stride subset in a fixed order, so results are reproducible.
__global__ void diag_partial_kernel(const double* __restrict__ f, double* partials, const __grid_constant__ StepParams p,
                                    const __grid_constant__ DvmConst<double> d, double dr, double dth, double r_in) {
  const size_t plane = (size_t)p.rows * p.pitch;
  const size_t n_nodes = (size_t)p.n_r * p.n_theta;
  double acc[4] = {0, 0, 0, 0};
  double mn[2] = {DBL_MAX, DBL_MAX};
  for (size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x; n < n_nodes;
       n += (size_t)gridDim.x * blockDim.x) {
    const int t = (int)(n / p.n_r), r = (int)(n % p.n_r);
    const NodeState<double> m = node_moments(f + (size_t)(t + kGhostRows) * p.pitch + r, plane, d);
    const double w = (r_in + r * dr) * dr * dth;
    acc[0] += w * m.rho;
    acc[1] += w * m.rho * m.ux;
    acc[2] += w * m.rho * m.uy;
    acc[3] += w * m.rho * (m.E + 0.5 * (m.ux * m.ux + m.uy * m.uy));
    mn[0] = fmin(mn[0], m.rho);
    mn[1] = fmin(mn[1], m.E);
  }
  diag_block_reduce(acc, mn, partials);
}

// The moments rho, j, e of `rows` nodes of a column added up in double.
__device__ __noinline__ void column_sums_double(const float* f, size_t plane, int pitch, int rows,
                                                const DvmConst<float>& d, double v[4]) {
  v[0] = v[1] = v[2] = v[3] = 0.0;
  for (int t = 0; t < rows; ++t) {
    ff m[4];
    const State32 st = state32(f + (size_t)t * pitch, plane, d, m);
    const float bad[4] = {0.f, st.ux.hi - st.ux.hi, st.uy.hi - st.uy.hi, st.E.hi - st.E.hi};   // NaN as in the kernel
    for (int i = 0; i < 4; ++i) v[i] += (double)m[i].hi + m[i].lo + bad[i];
  }
}

// FP32: the same integrals from the raw float-float moments (rho, j, e =
// rho (E + u^2/2)), without FP64 work per node: a thread adds up to `rows`
// nodes of one column in float-float and enters the double sums once, weighted
// by the column's r dr dtheta.  The form above spent ~30 FP64 operations per
// node (conversions, weights and sums; 121 us on 1024 x 2048, FP64-bound),
// this one is bound by the read of f.
__global__ void __launch_bounds__(kDiagThreads32, 2)
    diag_partial_f32_kernel(const float* __restrict__ f, double* partials, const __grid_constant__ StepParams p,
                            const __grid_constant__ DvmConst<float> d, double dr, double dth, double r_in, int rows) {
  const size_t plane = (size_t)p.rows * p.pitch;
  const size_t items = (size_t)((p.n_theta + rows - 1) / rows) * p.n_r;
  double acc[4] = {0, 0, 0, 0};
  float mh[2] = {FLT_MAX, FLT_MAX}, ml[2] = {0.f, 0.f};   // least rho and E so far, float-float
  bool any = false;
  for (size_t n = (size_t)blockIdx.x * blockDim.x + threadIdx.x; n < items; n += (size_t)gridDim.x * blockDim.x) {
    const int r = (int)(n % p.n_r), t0 = (int)(n / p.n_r) * rows, t1 = min(t0 + rows, p.n_theta);
    ff s[4] = {ff_of(0.f), ff_of(0.f), ff_of(0.f), ff_of(0.f)};
#pragma unroll 1
    for (int t = t0; t < t1; ++t) {
      ff m[4];
      const State32 st = state32(f + (size_t)(t + kGhostRows) * p.pitch + r, plane, d, m);
      // a node whose velocity or temperature is not finite makes its sums NaN
      m[1].hi += st.ux.hi - st.ux.hi;
      m[2].hi += st.uy.hi - st.uy.hi;
      m[3].hi += st.E.hi - st.E.hi;
#pragma unroll
      for (int i = 0; i < 4; ++i) s[i] = ff_add(s[i], m[i]);
      auto least = [&](int i, ff x) {
        if (x.hi < mh[i] || (x.hi == mh[i] && x.lo < ml[i])) { mh[i] = x.hi; ml[i] = x.lo; }
      };
      least(0, st.rho);
      least(1, st.E);
    }
    any = true;
    const double w = (r_in + r * dr) * dr * dth;
    double v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = (double)s[i].hi + s[i].lo;
    // the rows' moments may be floats and their sums not
    if (!(isfinite(s[0].hi) && isfinite(s[1].hi) && isfinite(s[2].hi) && isfinite(s[3].hi)))
      column_sums_double(f + (size_t)(t0 + kGhostRows) * p.pitch + r, plane, p.pitch, t1 - t0, d, v);
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i] += w * v[i];
  }
  const double mn[2] = {any && mh[0] < FLT_MAX ? (double)mh[0] + ml[0] : DBL_MAX,
                        any && mh[1] < FLT_MAX ? (double)mh[1] + ml[1] : DBL_MAX};
  diag_block_reduce(acc, mn, partials);
}

// The blocks' partials to the result: warp i adds (or takes the least of) the
// i-th integral, lanes over blocks (one thread over all of them took 112 us).
__global__ void __launch_bounds__(192) diag_final_kernel(const double* partials, int n_blocks, double* out, double n_nodes) {
  const int i = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double s = i < 4 ? 0.0 : DBL_MAX;
  for (int b = lane; b < n_blocks; b += 32) {
    const double v = partials[(size_t)b * 8 + i];
    s = i < 4 ? s + v : fmin(s, v);
  }
  for (int off = 16; off > 0; off >>= 1) {
    const double o = __shfl_down_sync(0xffffffffu, s, off);
    s = i < 4 ? s + o : fmin(s, o);
  }
  if (lane == 0) out[i] = s;
  if (threadIdx.x == 0) {
    out[6] = n_nodes;
    out[7] = 0.0;
  }
}

cudaError_t launch_diag_final(const double* partials, int n_blocks, double* out, double n_nodes, cudaStream_t s) {
  diag_final_kernel<<<1, 192, 0, s>>>(partials, n_blocks, out, n_nodes);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Launchers.
// ---------------------------------------------------------------------------
constexpr int kRowThreads = 128;

// Rows [t_begin, t_end) of the grid (t_end < 0: to the last row); the field
// arrays are always indexed with the full [n_theta][n_r] layout.
template <class T>
cudaError_t launch_set_state(T* f, const T* rho, const T* ur, const T* ut, const T* temp,
                             const StepParams& p, const DvmConst<T>& d, cudaStream_t s, int t_begin, int t_end) {
  if (t_end < 0) t_end = p.n_theta;
  if (t_begin < 0 || t_end <= t_begin) return cudaSuccess;
  if constexpr (sizeof(T) == 4) {
    const dim3 grid((p.n_r + 2 * kSetThreads32 - 1) / (2 * kSetThreads32), t_end - t_begin);
    set_state_f32_kernel<<<grid, kSetThreads32, 0, s>>>(f, rho, ur, ut, temp, p, d, t_begin);
  } else {
    const dim3 grid((p.n_r + kRowThreads - 1) / kRowThreads, t_end - t_begin);
    set_state_kernel<<<grid, kRowThreads, 0, s>>>(f, rho, ur, ut, temp, p, d, t_begin);
  }
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_moments(const T* f, T* rho, T* ur, T* ut, T* temp, const StepParams& p,
                           const DvmConst<T>& d, cudaStream_t s, int t_begin, int t_end) {
  if (t_end < 0) t_end = p.n_theta;
  if (t_begin < 0 || t_end <= t_begin) return cudaSuccess;
  dim3 grid((p.n_r + kRowThreads - 1) / kRowThreads, t_end - t_begin);
  if constexpr (sizeof(T) == 4)
    moments_f32_kernel<<<grid, kRowThreads, 0, s>>>(f, rho, ur, ut, temp, p, d, t_begin);
  else
    moments_kernel<T><<<grid, kRowThreads, 0, s>>>(f, rho, ur, ut, temp, p, d, t_begin);
  return cudaGetLastError();
}

template <class T>
cudaError_t launch_pack(const T* f, T* out, const StepParams& p, cudaStream_t s) {
  return launch_copy_rows<T, false>(f, out, kQ, p, RecvLabels{}, s);
}

template <class T>
cudaError_t launch_unpack(const T* in, T* f, const StepParams& p, const DvmConst<T>& d, cudaStream_t s) {
  return launch_copy_rows<T, true>(in, f, kQ, p, recv_labels(d, kQ), s);
}

template <class T>
cudaError_t launch_diagnostics(const T* f, double* partials, double* out, const StepParams& p,
                               const DvmConst<T>& d, double dr, double dth, double r_in,
                               cudaStream_t s) {
  if constexpr (sizeof(T) == 4) {
    // rows per thread: as many as keep every thread of the grid at work, at most 8
    const size_t per = (size_t)p.n_r * p.n_theta / ((size_t)kDiagBlocks * kDiagThreads32);
    diag_partial_f32_kernel<<<kDiagBlocks, kDiagThreads32, 0, s>>>(f, partials, p, d, dr, dth, r_in,
                                                                   (int)std::min<size_t>(8, std::max<size_t>(1, per)));
  } else {
    diag_partial_kernel<<<kDiagBlocks, 256, 0, s>>>(f, partials, p, d, dr, dth, r_in);
  }
  cudaError_t e = cudaGetLastError();
  return e != cudaSuccess ? e : launch_diag_final(partials, kDiagBlocks, out, (double)p.n_r * p.n_theta, s);
}

#define PCLB_INSTANTIATE(T)                                                                         \
  template cudaError_t launch_set_state<T>(T*, const T*, const T*, const T*, const T*,             \
                                           const StepParams&, const DvmConst<T>&, cudaStream_t,    \
                                           int, int);                                              \
  template cudaError_t launch_moments<T>(const T*, T*, T*, T*, T*, const StepParams&,              \
                                         const DvmConst<T>&, cudaStream_t, int, int);              \
  template cudaError_t launch_pack<T>(const T*, T*, const StepParams&, cudaStream_t);              \
  template cudaError_t launch_unpack<T>(const T*, T*, const StepParams&, const DvmConst<T>&,       \
                                        cudaStream_t);                                             \
  template cudaError_t launch_diagnostics<T>(const T*, double*, double*, const StepParams&,        \
                                             const DvmConst<T>&, double, double, double,           \
                                             cudaStream_t);
PCLB_INSTANTIATE(float)
PCLB_INSTANTIATE(double)

}  // namespace pclb
