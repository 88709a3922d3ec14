// Radial ghost columns of an FP64 shared-memory window, Sec. II C 1.
#pragma once

#include "device_common.cuh"
#include "pclb_internal.h"

namespace pclb {

// Values of scratch that ghost_columns_f64 needs for a tile of TT rows:
// per wall, node and row the four shells' sums (S, X, Y); in the same place
// afterwards the equilibrium factors of the two ghost layers and of the wall node.
template <int TT>
constexpr int kGhostScratch64 = 2 * 3 * TT * 12;

// Both walls' ghost columns of the tile at (r0, t0) from the window itself,
// by all threads of the block (at least 16 TT): inner wall node at
// window column kLeft with ghosts kLeft - 1 (layer 0) and kLeft - 2 (layer 1);
// outer wall node at n_r - 1 - r0 + kLeft, ghosts at the next two columns.
// Called for tiles that hold such columns; ends with a block barrier.
//
// Bound: FP64 issue (one warp-wide operation per ~76 cycles and quarter SM)
// and its latency.  One thread per wall row ran ~1400 dependent operations
// (180 us of a 206 us step on 100 x 20); here the sums are split by shell and
// node, the states of both nodes and the factors of both layers are formed in
// different lanes, and the ghost values by all threads, ~120 operations deep.
template <int TT, int PLANE>
__device__ __forceinline__ void ghost_columns_f64(double* sm, double* scratch, int r0, int t0, const StepParams& p,
                                                  const DvmConst<double>& d) {
  const int tid = threadIdx.x;
  const int cw_out = p.n_r - 1 - r0 + kLeft;
  auto active = [&](int side) { return side == 0 ? r0 == 0 : cw_out <= kLeft + kTileR; };
  auto wall = [&](int side) { return side == 0 ? kLeft : cw_out; };
  // one wall's part: the sums [node][row][shell][3], then the factors [ghost layer 0, 1, wall node][row][12]
  constexpr int kSide = 3 * TT * 12;

  // 1. sums of one shell at one node (the wall node or the next one inward)
  if (tid < 16 * TT) {
    const int row = tid % TT, node = (tid / TT) & 1, k = 1 + ((tid / (2 * TT)) & 3), side = tid / (8 * TT);
    if (active(side) && t0 + row < p.n_theta) {
      const int col = wall(side) + (side == 0 ? node : -node);
      const double* f = sm + (size_t)(1 + (k - 1) * kNDirs) * PLANE + (row + 2) * kWinR + col;
      double S = 0.0, D[kNDirs / 2];
#pragma unroll
      for (int i = 0; i < kNDirs / 2; ++i) {
        const double a = f[i * PLANE], b = f[(i + kNDirs / 2) * PLANE];
        S += a + b;
        D[i] = a - b;
      }
      double* o = scratch + side * kSide + (node * TT + row) * 12 + (k - 1) * 3;
      o[0] = S;
      o[1] = fma(d.cx[2], D[1] - D[3], D[0]);
      o[2] = fma(d.cx[2], D[1] + D[3], D[2]);
    }
  }
  __syncthreads();
  // 2. lanes (wall, node, row): the node's state; then lane (wall, layer, row)
  // the layer's state (Eq. 39 applied twice: g0 = 2a - b, g1 = 2 g0 - a, or
  // the prescribed values) and its factors
  EqParams<double> e, ea;
  const int row2 = tid % TT, layer = (tid / TT) & 1, side2 = tid / (2 * TT);
  const bool mine = tid < 4 * TT && active(side2) && t0 + row2 < p.n_theta;
  if (tid < (4 * TT < 32 ? 32 : 4 * TT)) {   // whole warps (shuffles)
    NodeState<double> m;
    m.rho = m.E = 1.0; m.ux = m.uy = 0.0; m.ok = true;
    if (mine) {
      const double* s = scratch + side2 * kSide + (layer * TT + row2) * 12;
      double s0 = sm[(row2 + 2) * kWinR + wall(side2) + (side2 == 0 ? layer : -layer)], sx = 0.0, sy = 0.0, se = 0.0;
#pragma unroll
      for (int k = 1; k <= 4; ++k) {
        s0 += s[(k - 1) * 3];
        sx = fma(d.speed[k], s[(k - 1) * 3 + 1], sx);
        sy = fma(d.speed[k], s[(k - 1) * 3 + 2], sy);
        se = fma(d.half_v2[k], s[(k - 1) * 3], se);
      }
      m = node_state64(s0, sx, sy, se);
    }
    const double v[4] = {m.rho, m.ux, m.uy, m.E};
    double a[4], g[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const double o = __shfl_xor_sync(0xffffffffu, v[j], TT);   // the other node's value
      a[j] = layer == 0 ? v[j] : o;
      const double b = layer == 0 ? o : v[j];
      const double g0 = 2.0 * a[j] - b;
      g[j] = layer == 0 ? g0 : 2.0 * g0 - a[j];
    }
    bool ok = m.ok;
    if (mine) {
      const int kind = p.bc_kind[side2] & ~PCLB_BC_NEQ, t = t0 + row2;
      if (kind != PCLB_BC_EXTRAP) {
        const double c = p.cos_t[t], s = p.sin_t[t];
        const double* b = p.bc_vals + (size_t)((side2 * 2 + layer) * 4) * p.n_theta + t;
        const double ur = b[1 * p.n_theta], ut = b[2 * p.n_theta];
        g[1] = ur * c - ut * s;
        g[2] = ur * s + ut * c;
        if (kind == PCLB_BC_DIRICHLET) {
          g[0] = b[0];
          g[3] = b[3 * p.n_theta];
        }
      }
      ok = ok && g[0] > 0.0 && g[3] > 0.0;
      if (!ok) atomicOr(p.status, PCLB_FLAG_NONPHYS);
      e = eq_params<double>(g[0], g[1], g[2], g[3], d);
      // the wall node's own factors, for the departure it hands to its ghosts
      if (p.bc_kind[side2] & PCLB_BC_NEQ) ea = eq_params<double>(a[0], a[1], a[2], a[3], d);
    }
  }
  __syncthreads();   // the partial sums have been read
  if (mine) {
    auto put = [&](int slot, const EqParams<double>& x) {
      double* o = scratch + side2 * kSide + (slot * TT + row2) * 12;
#pragma unroll
      for (int k = 0; k < 5; ++k) o[k] = x.w[k];
      o[5] = x.a0; o[6] = x.a1; o[7] = x.a1h; o[8] = x.uxE; o[9] = x.uyE;
    };
    put(layer, e);
    if (layer == 0 && (p.bc_kind[side2] & PCLB_BC_NEQ)) put(2, ea);
  }
  __syncthreads();
  // 3. the ghost values, a pair of opposite velocities of one layer and row
  // per item (the first pair's item also the rest velocity)
  for (int it = tid; it < 64 * TT; it += blockDim.x) {
    const int row = it % TT, lay = (it / TT) & 1, side = (it / (2 * TT)) & 1, pair = it / (4 * TT);
    const int col = wall(side) - (side == 0 ? 1 : -1) * (1 + lay);
    if (!active(side) || t0 + row >= p.n_theta || col < 0 || col >= kWinR) continue;
    const int k = 1 + pair / (kNDirs / 2), q1 = 1 + (k - 1) * kNDirs + pair % (kNDirs / 2), q2 = q1 + kNDirs / 2;
    double* w = sm + (row + 2) * kWinR;
    // f^eq of the pair, P(+-x) = ev +- od, and of the rest velocity
    auto feq = [&](int slot, double& fp, double& fm, double& f0) {
      const double* x = scratch + side * kSide + (slot * TT + row) * 12;
      const double y = d.vx[q1] * x[8] + d.vy[q1] * x[9], y2 = y * y;
      const double ev = x[5] + y2 * (x[7] + y2 * (1.0 / 24.0)), od = y * (x[6] + y2 * (1.0 / 6.0));
      fp = x[k] * (ev + od);
      fm = x[k] * (ev - od);
      if (pair == 0) f0 = x[0] * x[5];
    };
    double fp, fm, f0 = 0.0;
    feq(lay, fp, fm, f0);
    if (p.bc_kind[side] & PCLB_BC_NEQ) {
      double ap, am, a0 = 0.0;
      feq(2, ap, am, a0);
      const double* fa = w + wall(side);
      fp += fa[(size_t)q1 * PLANE] - ap;
      fm += fa[(size_t)q2 * PLANE] - am;
      f0 += fa[0] - a0;
    }
    w[(size_t)q1 * PLANE + col] = fp;
    w[(size_t)q2 * PLANE + col] = fm;
    if (pair == 0) w[col] = f0;
  }
  __syncthreads();
}

}  // namespace pclb
