// The FP64 initial state and step (Eq. 38) of the N_i = 16 and 24 velocity sets;
// a step is two launches, the radial ghost layers and the nodes.
//
// What bounds it: FP64 issue (a quarter SM starts one warp-wide FP64 operation
// per 64-76 cycles).  The convection increments, ~36 FP64 operations per update
// with their divisions, are therefore formed in 64-bit fixed point on each
// stencil's exponent (fixed64.cuh); FP64 keeps the sums, the states, the
// equilibrium and the final sums.  A block is 32 nodes of one row: four warps
// share the directions (H / 4 of the H pairs each, over the four shells), a fifth
// forms the states from their sums while they convect.  On small grids this
// also gives every node four threads.
// N_i = 16, 512 x 512: 379 us per step (1639 before, one thread per node and all
// of it in FP64); 64 x 64: 33 us (236, of which 150 the ghosts, one thread per wall
// row; now a warp per row).
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "dvm_generic.h"
#include "fixed64.cuh"
#include "pclb_internal.h"

namespace pclb {

namespace {

constexpr int kGhostWarps = 4;   // wall rows per block of the ghost kernel
constexpr int kParts = 4;        // warps that share a row's directions

// Equilibrium factors of rho, u, E: w_k = rho F_k (Eq. 11) and the coefficients
// of the polynomial of Eq. (10) in x = v.u / E.
struct GenFactors {
  double w[5], a0, a1, uxE, uyE;
};
__device__ __forceinline__ GenFactors gen_factors(double rho, double ux, double uy, double E, const DvmG& d) {
  GenFactors g;
  double Fs = 0.0;
#pragma unroll
  for (int k = 1; k <= 4; ++k) {
    const double F = E * fma(E, fma(E, fma(E, d.Fc[k][3], d.Fc[k][2]), d.Fc[k][1]), d.Fc[k][0]);
    g.w[k] = rho * F;
    Fs += F;
  }
  g.w[0] = rho * fma(-d.B0, Fs, 1.0);
  const double invE = recip_newton(E);
  g.uxE = ux * invE;
  g.uyE = uy * invE;
  const double s = fma(ux, g.uxE, uy * g.uyE);   // u^2 / E
  g.a1 = fma(-0.5, s, 1.0);
  g.a0 = fma(0.125 * s, s, g.a1);
  return g;
}

// What the nodes of a block share with the warps that own the directions: per
// shell A, B, C, O1, O3 of scale f^eq = A + y^2 (B + y^2 C) +- y (O1 + y^2 O3), y
// = c_i.u / E, and u / (E v_1) (DvmG holds c_i v_1), for 32 nodes.
struct GenPoly {
  double c[4][5][32], uxv[32], uyv[32];
};
__device__ __forceinline__ void put_poly(GenPoly& o, int lane, const GenFactors& g, int nd, const DvmG& d) {
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double w = g.w[k + 1], v = d.vx[1 + k * nd], hv = d.half_v2[k + 1], wa = w * g.a1, wh = w * hv;
    o.c[k][0][lane] = w * g.a0;
    o.c[k][1][lane] = wa * hv;
    o.c[k][2][lane] = wh * hv * (1.0 / 6.0);
    o.c[k][3][lane] = wa * v;
    o.c[k][4][lane] = wh * v * (1.0 / 3.0);
  }
  const double iv = recip_newton(d.vx[1]);
  o.uxv[lane] = g.uxE * iv;
  o.uyv[lane] = g.uyE * iv;
}

// f^eq of a block's 32 nodes from their fields, the directions over four warps.
// Bound: FP64 issue (90%), 3.4 operations per label with the direction's y shared
// by the shells (5.5 with x = v_q.u / E of each pair, and a thread per node):
// 512 x 512, N_i = 16, 130 us (197).
template <int ND>
__global__ void __launch_bounds__(32 * kParts)
    gen_set_state64(double* __restrict__ f, const double* __restrict__ rho, const double* __restrict__ u_r,
                    const double* __restrict__ u_t, const double* __restrict__ temp,
                    const __grid_constant__ StepParams p, const __grid_constant__ DvmG d) {
  constexpr int H = ND / 2, DIRS = H / kParts;
  __shared__ GenPoly poly;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = blockIdx.x * 32 + lane, t = blockIdx.y;
  const size_t plane = (size_t)p.rows * p.pitch;
  auto put = [&](int q, double v) {
    f[(size_t)q * plane + (size_t)(t + kGhostRows) * p.pitch + r] = v;
    if (t >= p.n_theta - 2) f[(size_t)d.recv_lo[q] * plane + (size_t)(t - (p.n_theta - 2)) * p.pitch + r] = v;
    if (t < 2) f[(size_t)d.recv_hi[q] * plane + (size_t)(p.n_theta + kGhostRows + t) * p.pitch + r] = v;
  };
  if (warp == 0) {
    const size_t n = (size_t)t * p.n_r + min(r, p.n_r - 1);
    const double c = p.cos_t[t], s = p.sin_t[t];
    const double R = rho[n], ur = u_r[n], ut = u_t[n], E = temp[n];   // E = T
    if (!(R > 0.0 && E > 0.0)) atomicOr(p.status, PCLB_FLAG_NONPHYS);
    const GenFactors g = gen_factors(R, ur * c - ut * s, ur * s + ut * c, E, d);
    put_poly(poly, lane, g, ND, d);
    if (r < p.n_r) put(0, g.w[0] * g.a0);
  }
  __syncthreads();
  if (r >= p.n_r) return;
#pragma unroll 1
  for (int j = 0; j < DIRS; ++j) {
    const int i = warp + kParts * j;
    const double y = fma(d.vx[1 + i], poly.uxv[lane], d.vy[1 + i] * poly.uyv[lane]), y2 = y * y;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double(&c)[5][32] = poly.c[k];
      const double ev = fma(y2, fma(y2, c[2][lane], c[1][lane]), c[0][lane]), z = fma(y2, c[4][lane], c[3][lane]);
      put(1 + k * ND + i, fma(y, z, ev));
      put(1 + k * ND + i + H, fma(-y, z, ev));
    }
  }
}

// Radial ghost layers of wall blockIdx.y, a warp per row: layer l sits at r = -1
// - l (inner) or n_r + l (outer).  Eq. (39) applied twice to the wall node a
// and the next node b: g0 = 2a - b, g1 = 2 g0 - a, for the components the
// boundary kind extrapolates; the others prescribed.  Lanes: pairs of opposite
// velocities for the sums and the values; (node) and (layer 0, 1, wall node) for
// the states and the factors.  Bound by the latency of ~150 dependent operations.
template <int ND>
__global__ void __launch_bounds__(32 * kGhostWarps)
    gen_ghost_kernel(const double* f, double* __restrict__ ghost, const __grid_constant__ StepParams p,
                     const __grid_constant__ DvmG d) {
  constexpr int H = ND / 2, NP = 4 * H, N = (NP + 31) / 32;
  __shared__ GenFactors fac[kGhostWarps][3];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int t = blockIdx.x * kGhostWarps + warp, side = blockIdx.y;
  pdl_wait();      // the step before this one has written f and read the ghosts
  pdl_launch();
  if (t >= p.n_theta) return;
  const size_t plane = (size_t)p.rows * p.pitch;
  const int ra = side == 0 ? 0 : p.n_r - 1, step = side == 0 ? 1 : -1;
  const double* fa = f + (size_t)(t + kGhostRows) * p.pitch + ra;
  auto first = [&](int pair) { return 1 + pair / H * ND + pair % H; };
  double wp[N], wm[N];   // the wall node's values
  double s[2][4];        // sums of nodes a and b
#pragma unroll
  for (int n = 0; n < 2; ++n) {
    s[n][0] = lane == 0 ? fa[n * step] : 0.0;
    s[n][1] = s[n][2] = s[n][3] = 0.0;
  }
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int pair = lane + 32 * j;
    wp[j] = wm[j] = 0.0;
    if (pair >= NP) continue;
    const int q = first(pair);
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const double a = fa[(size_t)q * plane + n * step], b = fa[(size_t)(q + H) * plane + n * step];
      if (n == 0) { wp[j] = a; wm[j] = b; }
      const double S = a + b, D = a - b;
      s[n][0] += S;
      s[n][1] = fma(d.vx[q], D, s[n][1]);
      s[n][2] = fma(d.vy[q], D, s[n][2]);
      s[n][3] = fma(d.half_v2[1 + pair / H], S, s[n][3]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int n = 0; n < 2; ++n)
#pragma unroll
      for (int i = 0; i < 4; ++i) s[n][i] += __shfl_xor_sync(0xffffffffu, s[n][i], o);
  const int node = lane >> 4, slot = min(lane >> 3, 2);
  const NodeState<double> m = node == 0 ? node_state64(s[0][0], s[0][1], s[0][2], s[0][3])
                                        : node_state64(s[1][0], s[1][1], s[1][2], s[1][3]);
  const int kind = p.bc_kind[side] & ~PCLB_BC_NEQ;
  const bool neq = (p.bc_kind[side] & PCLB_BC_NEQ) != 0;
  const double v[4] = {m.rho, m.ux, m.uy, m.E};
  double g[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const double a = __shfl_sync(0xffffffffu, v[i], 0), b = __shfl_sync(0xffffffffu, v[i], 16), g0 = 2.0 * a - b;
    g[i] = slot == 0 ? g0 : (slot == 1 ? 2.0 * g0 - a : a);
  }
  bool ok = m.ok;
  if (slot < 2) {
    if (kind != PCLB_BC_EXTRAP) {
      const double c = p.cos_t[t], sn = p.sin_t[t];
      const double* b = p.bc_vals + (size_t)((side * 2 + slot) * 4) * p.n_theta + t;
      const double ur = b[1 * p.n_theta], ut = b[2 * p.n_theta];
      g[1] = ur * c - ut * sn;
      g[2] = ur * sn + ut * c;
      if (kind == PCLB_BC_DIRICHLET) {
        g[0] = b[0];
        g[3] = b[3 * p.n_theta];
      }
    }
    ok = ok && positive64(g[0]) && positive64(g[3]);
  }
  if (!ok) atomicOr(p.status, PCLB_FLAG_NONPHYS);
  const GenFactors e = gen_factors(g[0], g[1], g[2], g[3], d);
  if ((lane & 7) == 0 && lane < 24) fac[warp][slot] = e;
  __syncwarp();
  double* out = ghost + ((size_t)(side * 2) * p.n_theta + t) * d.q;   // layer 1 at + n_theta Q
  const size_t layer = (size_t)p.n_theta * d.q;
  auto pair_values = [&](const GenFactors& x, int q, int k, double& fp, double& fm) {
    const double y = fma(d.vx[q], x.uxE, d.vy[q] * x.uyE), y2 = y * y;
    const double ev = fma(y2, fma(y2, 1.0 / 24.0, 0.5 * x.a1), x.a0), od = y * fma(y2, 1.0 / 6.0, x.a1);
    fp = x.w[k] * (ev + od);
    fm = x.w[k] * (ev - od);
  };
#pragma unroll
  for (int j = 0; j < N; ++j) {
    const int pair = lane + 32 * j;
    if (pair >= NP) continue;
    const int q = first(pair), k = 1 + pair / H;
    double ap = 0.0, am = 0.0;
    if (neq) {   // the wall node's departure
      pair_values(fac[warp][2], q, k, ap, am);
      ap = wp[j] - ap;
      am = wm[j] - am;
    }
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      double fp, fm;
      pair_values(fac[warp][l], q, k, fp, fm);
      out[l * layer + q] = fp + ap;
      out[l * layer + q + H] = fm + am;
    }
  }
}

template <int SCH>
struct GenTab {
  FxCoef<SCH> r;    // radial
  uint64_t at;      // |C_theta| at the block's first column, units of 2^-63
  int64_t fl;       // bit 0: v_r < 0, bit 1: v_theta < 0 for the first label of the pair
};

template <int SCH, int ND>
__global__ void __launch_bounds__(32 * (kParts + 1), 5)
    gen_step_kernel(const double* f, double* __restrict__ f_out, const double* ghost,
                    const __grid_constant__ StepParams p, const __grid_constant__ DvmG d) {
  constexpr int H = ND / 2, NP = 4 * H, DIRS = H / kParts;
  __shared__ GenTab<SCH> tab[NP];
  __shared__ double part[kParts][4][32];
  __shared__ double carried[2 * DIRS * 4][32 * kParts];   // d f - M_r - M_theta of each thread's labels
  __shared__ GenPoly poly;   // of (1 - d) f^eq
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r0 = blockIdx.x * 32, r = r0 + lane, t = blockIdx.y;
  const bool valid = r < p.n_r;
  const int rc = min(r, p.n_r - 1);   // threads without a node repeat the last one
  const int srow = t + kGhostRows;
  const size_t plane = (size_t)p.rows * p.pitch;
  const double inv_r0 = p.inv_r[r0], inv_r = p.inv_r[rc];
  const double* c64 = p.courant64 + (size_t)srow * NP * 4;
  for (int i = threadIdx.x; i < NP; i += blockDim.x) {
    const double* e = c64 + 4 * i;
    GenTab<SCH> x;
    x.r = fx_coef<SCH>(fx_fraction(e[0]));
    x.at = fx_fraction(e[2] * inv_r0);
    x.fl = (int64_t)e[3];
    tab[i] = x;
  }
  const double decay = p.decay, omd = 1.0 - decay;
  // label q at this node and at the azimuthal ghost rows it feeds (Eq. 40)
  auto put = [&](int q, double v) {
    f_out[(size_t)q * plane + (size_t)srow * p.pitch + r] = v;
    if (t >= p.n_theta - 2)
      f_out[(size_t)d.recv_lo[q] * plane + (size_t)(t - (p.n_theta - 2)) * p.pitch + r] = v;
    if (t < 2) f_out[(size_t)d.recv_hi[q] * plane + (size_t)(p.n_theta + kGhostRows + t) * p.pitch + r] = v;
  };
  pdl_wait();      // the ghost layers are written, f_out is free
  pdl_launch();
  const double* fn = f + (size_t)srow * p.pitch + rc;
  if (warp == kParts) {   // the states, from the other warps' sums
    const double f0 = fn[0];
    __syncthreads();
    double s[4] = {f0, 0.0, 0.0, 0.0};
#pragma unroll
    for (int w = 0; w < kParts; ++w)
#pragma unroll
      for (int i = 0; i < 4; ++i) s[i] += part[w][i][lane];
    const NodeState<double> m = node_state64(s[0], s[1], s[2], s[3]);
    if (valid && !m.ok) atomicOr(p.status, PCLB_FLAG_NONPHYS);
    const GenFactors g = gen_factors(omd * m.rho, m.ux, m.uy, m.E, d);
    put_poly(poly, lane, g, ND, d);
    __syncthreads();
    if (valid) put(0, fma(decay, f0, g.w[0] * g.a0));   // rest velocity: no convection
    return;
  }
  // sums over this warp's directions i = warp + 4 j
  double s0 = 0.0, sx = 0.0, sy = 0.0, se = 0.0;
#pragma unroll
  for (int k = 1; k <= 4; ++k) {
    double S = 0.0;
#pragma unroll
    for (int j = 0; j < DIRS; ++j) {
      const int q = 1 + (k - 1) * ND + warp + kParts * j;
      const double a = fn[(size_t)q * plane], b = fn[(size_t)(q + H) * plane], D = a - b;
      S += a + b;
      sx = fma(d.vx[q], D, sx);
      sy = fma(d.vy[q], D, sy);
    }
    s0 += S;
    se = fma(d.half_v2[k], S, se);
  }
  part[warp][0][lane] = s0;
  part[warp][1][lane] = sx;
  part[warp][2][lane] = sy;
  part[warp][3][lane] = se;
  __syncthreads();
  // d f - M_r - M_theta of this warp's labels
  const uint64_t dfx = fx_fraction(fabs(decay));
  const int64_t dsign = decay < 0.0 ? -1 : 0;
  const uint64_t ratio = fx_fraction(inv_r * recip_newton(inv_r0));   // 1/r relative to the block's first column
  // label q at radial index rr of row t (a ghost layer outside the grid)
  auto radial = [&](const double* fq, int q, int rr) -> const double& {
    if (rr < 0) return ghost[((size_t)(-1 - rr) * p.n_theta + t) * d.q + q];
    if (rr >= p.n_r) return ghost[((size_t)(2 + rr - p.n_r) * p.n_theta + t) * d.q + q];
    return fq[rr - rc];
  };
  // (rolled: unrolled, the loop was 64 KB of code and instruction fetch held it up, 703 us a step against 376)
#pragma unroll 1
  for (int n = 0; n < 4 * DIRS; ++n) {
    const int k = n & 3, i = warp + kParts * (n >> 2), pair = k * H + i, q1 = 1 + k * ND + i;
    const GenTab<SCH>& e = tab[pair];
    const FxCoef<SCH> cr = e.r, ct = fx_coef<SCH>(fx_mul_frac(e.at, ratio));
    const int fl = (int)e.fl;
#pragma unroll
    for (int L = 0; L < 2; ++L) {
      const int sr = ((fl & 1) != 0) != (L != 0) ? 1 : -1;               // upwind at larger r
      const ptrdiff_t st = ((fl & 2) != 0) != (L != 0) ? p.pitch : -(ptrdiff_t)p.pitch;   // upwind at larger theta
      constexpr int far = SCH == PCLB_SCHEME_LW ? -1 : 2;
      const int q = q1 + L * H;
      const double* x = fn + (size_t)q * plane;
      carried[2 * n + L][threadIdx.x] =
          fx_carried<SCH>(x[0], radial(x, q, rc + sr), radial(x, q, rc + far * sr), x[st], x[far * st], cr, ct, dfx,
                          dsign, decay, c64 + 4 * pair, inv_r);
    }
  }
  __syncthreads();
  if (!valid) return;
#pragma unroll 1
  for (int j = 0; j < DIRS; ++j) {
    const int i = warp + kParts * j;
    const double y = fma(d.vx[1 + i], poly.uxv[lane], d.vy[1 + i] * poly.uyv[lane]), y2 = y * y;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const double(&c)[5][32] = poly.c[k];
      const double ev = fma(y2, fma(y2, c[2][lane], c[1][lane]), c[0][lane]), z = fma(y2, c[4][lane], c[3][lane]);
      const int q = 1 + k * ND + i, n = 4 * j + k;
      put(q, fma(y, z, ev + carried[2 * n][threadIdx.x]));
      put(q + H, fma(-y, z, ev + carried[2 * n + 1][threadIdx.x]));
    }
  }
}

template <int SCH, int ND>
cudaError_t gen_step(const double* f, double* f_out, double* ghost, const StepParams& p, const DvmG& d,
                     cudaStream_t s) {
  const cudaError_t e = launch_overlapped(gen_ghost_kernel<ND>, dim3((p.n_theta + kGhostWarps - 1) / kGhostWarps, 2),
                                          32 * kGhostWarps, 0, s, f, ghost, p, d);
  if (e != cudaSuccess) return e;
  return launch_overlapped(gen_step_kernel<SCH, ND>, dim3((p.n_r + 31) / 32, p.n_theta), 32 * (kParts + 1), 0, s, f,
                           f_out, (const double*)ghost, p, d);
}

template <int ND>
cudaError_t gen_step_scheme(const double* f, double* f_out, double* ghost, const StepParams& p, const DvmG& d,
                            cudaStream_t s) {
  switch (p.scheme) {
    case PCLB_SCHEME_WB: return gen_step<PCLB_SCHEME_WB, ND>(f, f_out, ghost, p, d, s);
    case PCLB_SCHEME_LW: return gen_step<PCLB_SCHEME_LW, ND>(f, f_out, ghost, p, d, s);
    case PCLB_SCHEME_UPWIND2: return gen_step<PCLB_SCHEME_UPWIND2, ND>(f, f_out, ghost, p, d, s);
    default: return gen_step<PCLB_SCHEME_MWB, ND>(f, f_out, ghost, p, d, s);
  }
}

}  // namespace

cudaError_t gen_launch_set_state_f64(double* f, const double* rho, const double* ur, const double* ut,
                                     const double* temp, const StepParams& p, const DvmG& d, cudaStream_t s) {
  const dim3 grid((p.n_r + 31) / 32, p.n_theta);
  if (d.n_dirs == 16)
    gen_set_state64<16><<<grid, 32 * kParts, 0, s>>>(f, rho, ur, ut, temp, p, d);
  else
    gen_set_state64<24><<<grid, 32 * kParts, 0, s>>>(f, rho, ur, ut, temp, p, d);
  return cudaGetLastError();
}

cudaError_t gen_launch_step_f64(const double* f, double* f_out, double* ghost, const StepParams& p, const DvmG& d,
                                cudaStream_t s) {
  return d.n_dirs == 16 ? gen_step_scheme<16>(f, f_out, ghost, p, d, s) : gen_step_scheme<24>(f, f_out, ghost, p, d, s);
}

}  // namespace pclb
