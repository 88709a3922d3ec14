// The walls' part of the adjoint step (both precisions): the ghost states of a
// tile's rows and the cotangent that flows back from the ghosts through f^eq of
// the extrapolated state (Eq. 39).
#pragma once

#include "adjoint_common.cuh"
#include "device_common.cuh"
#include "f32_state.cuh"
#include "pclb_internal.h"

namespace pclb {

template <class T>
struct Cour {
  T a_r, k_r, a_w;
  int up_r, up_t;   // upwind offsets in r (columns) and theta (rows): -1 or +1
};

__device__ __forceinline__ void courant_entry(const StepParams& p, int row, int pair, float& ar, float& kr,
                                              float& aw, int& fl) {
  const float4 e = p.courant[(size_t)row * (4 * kNDirs / 2) + pair];
  ar = e.x; kr = e.y; aw = e.z; fl = __float_as_int(e.w);
}
__device__ __forceinline__ void courant_entry(const StepParams& p, int row, int pair, double& ar, double& kr,
                                              double& aw, int& fl) {
  const double* e = p.courant64 + ((size_t)row * (4 * kNDirs / 2) + pair) * 4;
  ar = e[0]; kr = e[1]; aw = e[2]; fl = (int)e[3];
}

// Courant data of label q at stored row `row` (ghost rows included), from
// the table of opposite-velocity pairs.
template <class T>
__device__ __forceinline__ Cour<T> courant(const StepParams& p, const DvmConst<T>& d, int q, int row) {
  Cour<T> c;
  if (q == 0) {
    c.a_r = T(0); c.k_r = T(0); c.a_w = T(0); c.up_r = -1; c.up_t = -1;
    return c;
  }
  const int k = d.shell[q];
  const int i = (q - 1) % kNDirs;
  const bool second = i >= kNDirs / 2;
  const int pair = (k - 1) * (kNDirs / 2) + (second ? i - kNDirs / 2 : i);
  int fl;
  courant_entry(p, row, pair, c.a_r, c.k_r, c.a_w, fl);
  const bool vr_neg = ((fl & 1) != 0) != second;   // the partner has the opposite velocity
  const bool vt_neg = ((fl & 2) != 0) != second;
  c.up_r = vr_neg ? 1 : -1;
  c.up_t = vt_neg ? 1 : -1;
  return c;
}

// f^eq_q of a node state (rho and E in double as the step evaluates them).
template <class T>
__device__ __forceinline__ T adj_feq(const EqParams<T>& e, const DvmConst<T>& d, int q) {
  return feq_q<T>(e, d.vx[q], d.vy[q], d.shell[q]);
}

// What a wall's tiles keep per row, in the workspace: equilibrium parameters
// of the two ghost layers and of the wall node (non-equilibrium ghosts carry
// its departure), the cotangent g_wall for the wall node (node 0) and the next
// node inward (node 1), and the per-label cotangent non-equilibrium ghosts hand
// straight to the wall node.  Slots: 0 the inner wall, 1 the outer wall for
// the last radial tile, 2 the outer wall for the tile before it (whose
// stencils reach the ghosts when the last tile is one node wide); a block
// writes and reads its own rows of its own slots only.
template <class T>
struct WallScratch {
  EqParams<T>* ghost;   // [slot][layer 0, 1, wall node][n_theta]
  T* gwall;             // [slot][node][n_theta][4]
  T* gdir;              // [slot][n_theta][Q]
  __device__ __forceinline__ static int slot(int side, bool last_tile) { return side == 0 ? 0 : (last_tile ? 1 : 2); }
};

// Shared-memory scratch of adjoint_walls for TT rows.
template <class T, int TT>
struct WallShared {
  double rho_d[2][TT], E_d[2][TT];               // nodes a (the wall node) and b
  T rho[2][TT], ux[2][TT], uy[2][TT], E[2][TT];
  double grho[2][TT], gE[2][TT];                 // ghost layers
  T gux[2][TT], guy[2][TT];
  EqParams<T> eq[3][TT];                         // ghost layers, wall node
};

// Rows t0 .. t0 + TT - 1 of wall `side` into `slot` of ws, by all threads of the
// block (256); ends with a block barrier.  f, lam: the stored planes.
// values: if given, the ghost values themselves, [layer][TT][Q] (the FP64
// kernel copies them into its windows; forming them pair by pair took 36
// FP64 operations per pair between two block barriers).
//
// Bound: latency.  The node states use FP64 (a warp-wide operation per ~76
// cycles and quarter SM): they are formed once per row, a lane each, instead of
// in every lane of a warp per row.
template <class T, int TT>
__device__ __noinline__ void adjoint_walls(const T* f, const T* lam, int side, int slot,
                                           int t0, const WallScratch<T>& ws, WallShared<T, TT>& sh, T* values,
                                           const StepParams& p, const DvmConst<T>& d) {
  const int tid = threadIdx.x;
  const size_t plane = (size_t)p.rows * p.pitch;
  const int step = side == 0 ? 1 : -1;                // towards the interior
  const int out = -step;                              // the upwind offset that reads the ghosts
  const int ra = side == 0 ? 0 : p.n_r - 1;
  const int kind = p.bc_kind[side] & ~PCLB_BC_NEQ;
  const bool neq = (p.bc_kind[side] & PCLB_BC_NEQ) != 0;
  EqParams<T>* ghost = ws.ghost + (size_t)slot * 3 * p.n_theta;
  T* gwall = ws.gwall + (size_t)slot * 2 * p.n_theta * 4;
  T* gdir = ws.gdir + (size_t)slot * p.n_theta * kQ;
  if (tid < 2 * TT) {
    const int row = tid % TT, node = tid / TT, t = min(t0 + row, p.n_theta - 1);
    const NodeState<T> m = node_moments(f + (size_t)(t + kGhostRows) * p.pitch + ra + node * step, plane, d);
    sh.rho_d[node][row] = m.rho_d; sh.E_d[node][row] = m.E_d;
    sh.rho[node][row] = m.rho; sh.ux[node][row] = m.ux; sh.uy[node][row] = m.uy; sh.E[node][row] = m.E;
  }
  __syncthreads();
  if (tid < 3 * TT) {
    const int row = tid % TT, l = tid / TT, t = min(t0 + row, p.n_theta - 1);
    EqParams<T> e{};
    if (l < 2) {
      // Eq. (39), applied twice: g0 = 2a - b, g1 = 2 g0 - a
      double r0 = 2.0 * sh.rho_d[0][row] - sh.rho_d[1][row], E0 = 2.0 * sh.E_d[0][row] - sh.E_d[1][row];
      T x0 = T(2) * sh.ux[0][row] - sh.ux[1][row], y0 = T(2) * sh.uy[0][row] - sh.uy[1][row];
      if (l == 1) {
        r0 = 2.0 * r0 - sh.rho_d[0][row];
        E0 = 2.0 * E0 - sh.E_d[0][row];
        x0 = T(2) * x0 - sh.ux[0][row];
        y0 = T(2) * y0 - sh.uy[0][row];
      }
      if (kind != PCLB_BC_EXTRAP) {
        const double c = p.cos_t[t], s = p.sin_t[t];
        const double* v = p.bc_vals + (size_t)((side * 2 + l) * 4) * p.n_theta + t;
        x0 = (T)(v[1 * p.n_theta] * c - v[2 * p.n_theta] * s);
        y0 = (T)(v[1 * p.n_theta] * s + v[2 * p.n_theta] * c);
        if (kind == PCLB_BC_DIRICHLET) {
          r0 = v[0];
          E0 = v[3 * p.n_theta];
        }
      }
      if (!(r0 > 0.0 && E0 > 0.0)) atomicOr(p.status, PCLB_FLAG_NONPHYS);
      sh.grho[l][row] = r0; sh.gE[l][row] = E0; sh.gux[l][row] = x0; sh.guy[l][row] = y0;
      e = eq_params<T>(r0, x0, y0, E0, d);
    } else if (neq) {
      e = eq_params<T>(sh.rho_d[0][row], sh.ux[0][row], sh.uy[0][row], sh.E_d[0][row], d);
    }
    sh.eq[l][row] = e;
    if (t0 + row < p.n_theta) ghost[(size_t)l * p.n_theta + t] = e;
  }
  __syncthreads();
  constexpr int half = kNDirs / 2;
  if (values) {
    for (int it = tid; it < 2 * 4 * half * TT; it += blockDim.x) {   // layer, row, pair
      const int pair = it % (4 * half), row = it / (4 * half) % TT, l = it / (4 * half * TT);
      const int q1 = 1 + pair / half * kNDirs + pair % half, t = min(t0 + row, p.n_theta - 1);
      const T* fa = f + (size_t)(t + kGhostRows) * p.pitch + ra;
#pragma unroll
      for (int L = 0; L < 2; ++L) {
        const int q = q1 + L * half;
        T v = adj_feq<T>(sh.eq[l][row], d, q);
        if (neq) v += fa[(size_t)q * plane] - adj_feq<T>(sh.eq[2][row], d, q);
        values[(l * TT + row) * kQ + q] = v;
      }
    }
    __syncthreads();
  }
  // a pair of opposite velocities of one row per thread, 16 lanes a row
  for (int it = tid; it < 4 * half * TT; it += blockDim.x) {
    const int row = it / (4 * half), pair = it % (4 * half), t = min(t0 + row, p.n_theta - 1);
    const bool live = t0 + row < p.n_theta;
    const int srow = t + kGhostRows;
    const T* fa = f + (size_t)srow * p.pitch + ra;
    const T* fb = fa + step;
    const T* la = lam + (size_t)srow * p.pitch + ra;
    const T* lb = la + step;
    const EqParams<T> e0 = sh.eq[0][row], e1 = sh.eq[1][row], ea = sh.eq[2][row];
    // per layer: the sums A, Bx, By, Cs, Dx, Fq of eq_cotangent over this
    // thread's pair; layer 2: those at the wall node's own state for the
    // departure of non-equilibrium ghosts
    T c[3][6];
#pragma unroll
    for (int l = 0; l < 3; ++l)
#pragma unroll
      for (int j = 0; j < 6; ++j) c[l][j] = T(0);
    const int k = 1 + pair / half;
    const int q1 = 1 + (k - 1) * kNDirs + pair % half;
    // cotangent of the ghost values f_q(layer l) = -sum_n lam_q(n) dM_q(n)/df_q(ghost l):
    // the wall node a reads (a, g0, g1), the next node b reads (b, a, g0)
    T lg[2][2];                                        // [label][layer]
#pragma unroll
    for (int L = 0; L < 2; ++L) {
      const int q = q1 + L * half;
      const Cour<T> cr = courant<T>(p, d, q, srow);
      lg[L][0] = lg[L][1] = T(0);
      if (cr.up_r == out) {
        const T f_a = fa[(size_t)q * plane], f_b = fb[(size_t)q * plane];
        // the ghost values as the step forms them (plus the departure f_q(a)
        // - f^eq_q(a) for non-equilibrium ghosts)
        T g0, g1;
        if (values) {
          g0 = values[row * kQ + q];
          g1 = values[(TT + row) * kQ + q];
        } else {
          const T dep = neq ? f_a - adj_feq<T>(ea, d, q) : T(0);
          g0 = adj_feq<T>(e0, d, q) + dep;
          g1 = adj_feq<T>(e1, d, q) + dep;
        }
        T MDa, MPa, MDb, MPb;
        mwb_partials<T>(cr.a_r, cr.k_r, f_a - g0, g0 - g1, MDa, MPa);
        mwb_partials<T>(cr.a_r, cr.k_r, f_b - f_a, f_a - g0, MDb, MPb);
        const T lam_a = la[(size_t)q * plane], lam_b = lb[(size_t)q * plane];
        lg[L][0] = lam_a * (MDa - MPa) + lam_b * MPb;
        lg[L][1] = lam_a * MPa;
      }
    }
    // the ghost values' cotangents flow, for non-equilibrium ghosts, straight
    // to f_q(a) (coefficient 1) and, with the opposite sign, through f^eq_q(a)
    if (live) {
      T* gd = gdir + (size_t)t * kQ;
      if (pair == 0) gd[0] = T(0);   // the rest velocity reads no ghost
      gd[q1] = lg[0][0] + lg[0][1];
      gd[q1 + half] = lg[1][0] + lg[1][1];
    }
    const T lneq[2] = {neq ? -(lg[0][0] + lg[0][1]) : T(0), neq ? -(lg[1][0] + lg[1][1]) : T(0)};
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      if (l == 2 && !neq) break;                      // the departure's terms: non-equilibrium ghosts only
      const int m = l < 2 ? l : 0;
      const T E = l < 2 ? (T)sh.gE[m][row] : sh.E[0][row], ux = l < 2 ? sh.gux[m][row] : sh.ux[0][row],
              uy = l < 2 ? sh.guy[m][row] : sh.uy[0][row];
      const T lp = l < 2 ? lg[0][m] : lneq[0], lm = l < 2 ? lg[1][m] : lneq[1];
      const T* cf = d.Fc[k];
      const T F = E * (cf[0] + E * (cf[1] + E * (cf[2] + E * cf[3])));
      const T Fd = cf[0] + E * (T(2) * cf[1] + E * (T(3) * cf[2] + E * T(4) * cf[3]));
      const T invE = recip1(E);
      const T s = (ux * ux + uy * uy) * invE;
      const T a1 = T(1) - T(0.5) * s;
      const T a0 = a1 + T(0.125) * s * s;
      T Ak = 0, Bxk = 0, Byk = 0, Ck = 0, Dk = 0;
      pair_terms<T>(d.vx[q1], d.vy[q1], ux * invE, uy * invE, s, a0, a1, lp, lm, Ak, Bxk, Byk, Ck, Dk);
      c[l][0] = F * Ak; c[l][1] = F * Bxk; c[l][2] = F * Byk; c[l][3] = F * Ck; c[l][4] = F * Dk; c[l][5] = Fd * Ak;
    }
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      if (l == 2 && !neq) break;
#pragma unroll
      for (int j = 0; j < 6; ++j)
#pragma unroll
        for (int o = 2 * half; o > 0; o >>= 1) c[l][j] += __shfl_xor_sync(0xffffffffu, c[l][j], o);
    }
    if (pair != 0 || !live) continue;
    T Gl[3][4];
#pragma unroll
    for (int l = 0; l < 3; ++l) {
      // G of eq_cotangent at the ghost state, and at the wall node's state for
      // the departure (the rest velocity returns nothing)
      if (l == 2 && !neq) {
        Gl[2][0] = Gl[2][1] = Gl[2][2] = Gl[2][3] = T(0);
        break;
      }
      const int m = l < 2 ? l : 0;
      const T rho = l < 2 ? (T)sh.grho[m][row] : sh.rho[0][row], E = l < 2 ? (T)sh.gE[m][row] : sh.E[0][row];
      const T ux = l < 2 ? sh.gux[m][row] : sh.ux[0][row], uy = l < 2 ? sh.guy[m][row] : sh.uy[0][row];
      const T invE = recip1(E);
      const T s = (ux * ux + uy * uy) * invE;
      Gl[l][0] = c[l][0];
      Gl[l][1] = rho * (c[l][1] + T(2) * ux * c[l][3]) * invE;
      Gl[l][2] = rho * (c[l][2] + T(2) * uy * c[l][3]) * invE;
      Gl[l][3] = rho * (c[l][5] - (c[l][4] + s * c[l][3]) * invE);
    }
    // back through the extrapolation g0 = 2a - b, g1 = 3a - 2b (extrapolated components only)
    const bool ext_rho_E = kind != PCLB_BC_DIRICHLET;
    const bool ext_u = kind == PCLB_BC_EXTRAP;
    T Ga[4], Gb[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool ext = (j == 0 || j == 3) ? ext_rho_E : ext_u;
      Ga[j] = (ext ? T(2) * Gl[0][j] + T(3) * Gl[1][j] : T(0)) + (neq ? Gl[2][j] : T(0));
      Gb[j] = ext ? -Gl[0][j] - T(2) * Gl[1][j] : T(0);
    }
    T ga[4], gb[4];
    to_moment_cotangent<T>(sh.rho[0][row], sh.ux[0][row], sh.uy[0][row], sh.E[0][row], Ga, ga);
    to_moment_cotangent<T>(sh.rho[1][row], sh.ux[1][row], sh.uy[1][row], sh.E[1][row], Gb, gb);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      gwall[(size_t)t * 4 + j] = ga[j];
      gwall[((size_t)p.n_theta + t) * 4 + j] = gb[j];
    }
  }
  __syncthreads();
}

}  // namespace pclb
