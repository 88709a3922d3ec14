// Reverse-mode adjoint of one time step (Eq. 38 with the boundary nodes of
// Sec. II C): given the state f^n and the cotangent lam^{n+1} of f^{n+1},
// computes lam^n = J(f^n)^T lam^{n+1}.
//
// With m = (rho, j_x, j_y, e) the moments (linear in f, psi_q = (1, v_x, v_y,
// |v|^2/2)), the step is F_q(c) = (1-d) f^eq_q(m(c)) + d f_q(c) - M^r_q(c) -
// M^theta_q(c), d = exp(-dt/tau) (Eq. 19), M the MWB increments (Eq. 28)
// M = a D + K h(D, Dp), h = |D|(D - Dp)/(|D| + |Dp|), a = |C|, K = |C|(1-|C|),
// D, Dp the upwind differences of the node.  Hence, per node c and label q,
//   lam^n_q(c) = d lam_q(c) + (1-d) psi_q . g(c)
//              - sum over the nodes n whose stencil reads f_q(c) of
//                lam_q(n) dM_q(n)/df_q(c)                    (r and theta)
//              + psi_q . g_wall(c)  for the two nodes next to a wall,
// with g(c) = (dm/d(rho,u,E))^T sum_q' lam_q'(c) df^eq_q'/d(rho,u,E), and
// g_wall the cotangent that flows back from the radial ghost nodes through
// f^eq of the extrapolated state (Eq. 39).  |x| is differentiated as
// sign(x) with sign(0) = 0 (the switch function on its active branch); at
// D = Dp = 0 the derivative of h is 0.
//
// One launch per step, tiles of 32 (r) x TT (theta) nodes: the FP32 kernel is
// adjoint_f32x2.cu (two nodes per thread), the FP64 kernel adjoint_pair_kernel
// below (one node per thread).
//   * Tiles at a wall first form their rows' ghost states (Eq. 39 or
//     prescribed) and the cotangent g_wall they return (adjoint_walls.cuh).
//     They come first in the launch.  (As a kernel of its own on a side
//     stream, with the wall tiles after it, this took 19 us (FP32) and 31 us
//     (FP64) of each step with most of the chip idle, and four event calls.)
//   * Each thread forms g of its node from f^n and lam^{n+1} read from global
//     memory (a reduction over the 33 labels).  Then the velocities, in pairs
//     of opposite labels, stream their f and lam windows over [r0-4, r0+36) x
//     [t0-2, t0+TT+2) through a ring of shared-memory stages filled by TMA
//     while earlier pairs compute.  Each pair runs in two phases: (A) every
//     node whose upwind stencil can reach the tile forms lam(n) dM(n)/dD and
//     lam(n) dM(n)/dDp once, in r and in theta; (B) every tile node gathers
//     the products of the nodes that read it and adds d lam + psi . ((1-d) g +
//     g_wall).  One barrier per pair separates the phases; a stage is refilled
//     as soon as its pair's phase (A) is done.
// The FP64 kernel is bound by FP64 issue (a warp-wide operation per ~76 cycles
// and quarter SM); the partials are therefore formed in integers
// (fx_mwb_partials, 10 of 14 FP64 operations less per label and direction).
// TT = 8 rows; 4 on grids whose tiles would leave SMs idle.
#include <cuda.h>
#include <cuda_runtime.h>

#include <type_traits>

#include "device_common.cuh"
#include "adjoint_common.cuh"
#include "adjoint_walls.cuh"
#include "fixed64.cuh"
#include "f32_state.cuh"
#include "pclb_internal.h"

namespace pclb {

// Courant entry of one pair of opposite velocities at one theta row, in units
// of 2^-63: alpha^2 and 2 alpha (1 - alpha) of alpha = |C_r|, and |C_theta| at
// the tile's first column; flag bit 0 set when v_r < 0 and bit 1 when v_theta
// < 0 for the first label of the pair.
struct alignas(32) CourEntry {
  uint64_t a2, k2, at;
  int fl;
};

// bytes of one part of the wall scratch, aligned for the next
static size_t scratch_part(size_t bytes) { return (bytes + 255) & ~(size_t)255; }

constexpr int kAdjStages = 2;   // ring depth of the pair-streaming kernel (2 measured best of 1..4)
static_assert(sizeof(EqParams<float>) == 10 * sizeof(float) && sizeof(EqParams<double>) == 10 * sizeof(double),
              "ghost-state scratch holds 10 values per EqParams");

template <int TT>
struct AdjSize {
  static constexpr int threads = 32 * TT;
  static constexpr int min_blocks = 24 / TT;   // at most 85 registers
  static constexpr int plane = kWinR * (TT + 4);
  static constexpr int npairs = 4 * kNDirs / 2;
  // products of one label: radial A, B over TT rows x 36 columns (tile
  // columns -2 .. 33), azimuthal A, B over TT + 4 rows (-2 .. TT + 1) x 32
  static constexpr int rcols = kTileR + 4;
  static constexpr int prod = 2 * TT * rcols + 2 * (TT + 4) * kTileR;
  static constexpr int ring_bytes = kAdjStages * 4 * plane * 8;   // f, f', lam, lam' per stage
  static constexpr int prod_bytes = 2 * 2 * prod * 8;             // 2 buffers x 2 labels
  static constexpr int ratio_bytes = kTileR * 8;
  static constexpr int tab_bytes = (TT + 4) * npairs * (int)sizeof(CourEntry);
  static constexpr int smem = ring_bytes + prod_bytes + ratio_bytes + tab_bytes + 128;
  // the ring's planes are TMA destinations: 128-byte aligned
  static_assert((plane * 8) % 128 == 0, "TMA destinations must stay 128-byte aligned");
};

namespace {


// (rho, u_x, u_y, E) of one node for the cotangent of the equilibrium (FP64;
// the FP32 pair kernel forms the state of its two nodes in float-float).
__device__ __forceinline__ void adj_node_state(const double* f, int plane, const DvmConst<double>& d, double& rho,
                                               double& ux, double& uy, double& E, bool& ok) {
  const NodeState<double> m = node_moments(f, plane, d);
  rho = m.rho; ux = m.ux; uy = m.uy; E = m.E; ok = m.ok;
}


// ---- the pair-streaming kernel's stencil pieces ------------------------------
// Products of both labels of a pair at one node in one direction: q1 has its
// upwind side at offset U, q2 (the opposite velocity) at -U.  sf, sl: the
// pair's f and lam planes (q2 at +PLANE); o: the node in a plane; pr: its
// product slot (M_D products; the M_Dp ones at +DB, q2's at +PROD).
template <int U, int PLANE, int PROD, int DB>
__device__ __forceinline__ void radial_pair(const double* sf, const double* sl, double* pb, int o, int pr, uint64_t a2,
                                            uint64_t k2, double lam[2]) {
#pragma unroll
  for (int L = 0; L < 2; ++L) {
    constexpr int kU[2] = {U, -U};
    const double* f = sf + L * PLANE + o;
    double MD, MP;
    fx_mwb_partials(f[0] - f[kU[L]], f[kU[L]] - f[2 * kU[L]], a2, k2, MD, MP);
    lam[L] = sl[L * PLANE + o];
    pb[L * PROD + pr] = lam[L] * MD;
    pb[L * PROD + pr + DB] = lam[L] * MP;
  }
}

template <int U, int PLANE, int PROD, int DB>
__device__ __forceinline__ void azimuthal_pair(const double* sf, const double lam[2], double* pb, int o, int pa,
                                               uint64_t a2, uint64_t k2) {
#pragma unroll
  for (int L = 0; L < 2; ++L) {
    constexpr int kU[2] = {U, -U};
    const double* f = sf + L * PLANE + o;
    double MD, MP;
    fx_mwb_partials(f[0] - f[kU[L]], f[kU[L]] - f[2 * kU[L]], a2, k2, MD, MP);
    pb[L * PROD + pa] = lam[L] * MD;
    pb[L * PROD + pa + DB] = lam[L] * MP;
  }
}

// One label at one halo node, upwind side at offset U.
template <int U>
__device__ __forceinline__ void azimuthal_one(const double* fw, const double* lw, double* pa, int DB, uint64_t a2,
                                              uint64_t k2) {
  double MD, MP;
  fx_mwb_partials(fw[0] - fw[U], fw[U] - fw[2 * U], a2, k2, MD, MP);
  const double lam = lw[0];
  pa[0] = lam * MD;
  pa[DB] = lam * MP;
}

// Gather of the radial products at one node: the node n = c + j u reads f(n),
// f(n + u), f(n + 2 u), so dM(n)/df(c) collects M_D of n = c, M_Dp - M_D of
// n = c - u and -M_Dp of n = c - 2u (u = U for q1, -U for q2).
template <class T, int U, int PROD, int DB>
__device__ __forceinline__ void gather_radial(const T* pb, int pr, T acc[2]) {
  acc[0] = pb[pr] - pb[pr - U] + pb[pr + DB - U] - pb[pr + DB - 2 * U];
  const T* p2 = pb + PROD;
  acc[1] = p2[pr] - p2[pr + U] + p2[pr + DB + U] - p2[pr + DB + 2 * U];
}

// Azimuthal gather when the rows -2 .. +2 around the node all have q1's
// upwind side on the same side: the readers of the node sit at +V, +2V for
// q1 and at -V, -2V for q2 (V = +-row stride).
template <class T, int V, int PROD, int DB>
__device__ __forceinline__ void gather_azimuthal(const T* pb, int pa, T acc[2]) {
  acc[0] += pb[pa] + pb[pa + DB + V] - pb[pa + V] - pb[pa + DB + 2 * V];
  const T* p2 = pb + PROD;
  acc[1] += p2[pa] + p2[pa + DB - V] - p2[pa - V] - p2[pa + DB - 2 * V];
}

// The same where the upwind side changes within the five rows: bit o of neg
// set when row o - 2 has v_theta < 0 for q1 (its reader of row 0 is then the
// row below it).
template <class T, int PROD, int DB>
__device__ __forceinline__ void gather_azimuthal_mixed(const T* pb, int pa, int tneg, T acc[2]) {
#pragma unroll
  for (int L = 0; L < 2; ++L) {
    const T* P = pb + L * PROD;
    const int neg = L ? (tneg ^ 0x1f) : tneg;          // the partner has the opposite velocity
    T a = P[pa];
    if (neg & 2) a += P[pa + DB - kTileR] - P[pa - kTileR];
    if (!(neg & 8)) a += P[pa + DB + kTileR] - P[pa + kTileR];
    if (neg & 1) a -= P[pa + DB - 2 * kTileR];
    if (!(neg & 16)) a -= P[pa + DB + 2 * kTileR];
    acc[L] += a;
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// Pair-streaming part.
// ---------------------------------------------------------------------------
template <int TT>
__global__ void __launch_bounds__(AdjSize<TT>::threads, AdjSize<TT>::min_blocks)
    adjoint_pair_kernel(const __grid_constant__ CUtensorMap tmap_f, const __grid_constant__ CUtensorMap tmap_l,
                        const double* __restrict__ f, const double* __restrict__ lam_in, double* __restrict__ lam_out,
                        const __grid_constant__ WallScratch<double> ws, const __grid_constant__ AdjOrder order,
                        const __grid_constant__ StepParams p, const __grid_constant__ DvmConst<double> d) {
  using T = double;
  using SZ = AdjSize<TT>;
  constexpr int PLANE = SZ::plane;
  constexpr int NP = SZ::npairs, RC = SZ::rcols, PROD = SZ::prod;
  constexpr int S = kAdjStages;
  // offsets inside one label's products
  constexpr int AR = 0, BR = TT * RC, AT = 2 * TT * RC, BT = 2 * TT * RC + (TT + 4) * kTileR;
  constexpr uint32_t kStageBytes = (uint32_t)(4 * PLANE * sizeof(T));
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* ring = reinterpret_cast<T*>(smem_raw);                 // [stage][f q1, f q2, lam q1, lam q2][PLANE]
  T* prod = ring + S * 4 * PLANE;                             // [buffer][label][products]
  uint64_t* ratio = reinterpret_cast<uint64_t*>(prod + 2 * 2 * PROD);   // 1/r of the tile columns relative to the first
  CourEntry* ctab = reinterpret_cast<CourEntry*>(ratio + kTileR);        // [TT + 4][NP]
  uint64_t* bar = reinterpret_cast<uint64_t*>(ctab + (TT + 4) * NP);     // [S]

  int tx, ty;
  order.tile(blockIdx.x, tx, ty);
  const int r0 = tx * kTileR;
  const int t0 = ty * TT;
  const int tid = threadIdx.x;
  const int lane = tid & 31, rowl = tid >> 5;

  // the planes of pair pr (labels q1, q1 + N_i/2) into stage s (thread 0)
  auto issue_pair = [&](int pr, int s) {
    const int k = 1 + pr / (kNDirs / 2);
    const int q1 = 1 + (k - 1) * kNDirs + pr % (kNDirs / 2), q2 = q1 + kNDirs / 2;
    T* st = ring + s * 4 * PLANE;
    mbar_arrive_expect_tx(&bar[s], kStageBytes);
    tma_load_3d(st, &tmap_f, r0 - kLeft, t0, q1, &bar[s]);
    tma_load_3d(st + PLANE, &tmap_f, r0 - kLeft, t0, q2, &bar[s]);
    tma_load_3d(st + 2 * PLANE, &tmap_l, r0 - kLeft, t0, q1, &bar[s]);
    tma_load_3d(st + 3 * PLANE, &tmap_l, r0 - kLeft, t0, q2, &bar[s]);
  };
  if (tid == 0) {
    tma_prefetch_desc(&tmap_f);
    tma_prefetch_desc(&tmap_l);
    for (int s = 0; s < S; ++s) mbar_init(&bar[s], 1);
    mbar_fence_init();
  }
  pdl_wait();      // the step before this one has written lam and read lam_out
  pdl_launch();    // the next one may start its set-up
  // wall tiles: the ghost states of this tile's rows and their cotangent
  const int cw_out = p.n_r - 1 - r0 + kLeft;
  const bool inner = r0 == 0, outer = cw_out <= kLeft + kTileR;
  const int slots[2] = {0, WallScratch<T>::slot(1, tx == order.nt - 1)};
  static_assert(sizeof(WallShared<T, TT>) <= (TT + 4) * NP * sizeof(CourEntry), "wall scratch inside the Courant table");
  for (int side = 0; side < 2; ++side)
    if (side == 0 ? inner : outer)
      adjoint_walls<T, TT>(f, lam_in, side, slots[side], t0, ws, *reinterpret_cast<WallShared<T, TT>*>(ctab), p, d);
  const double inv_r0 = p.inv_r[r0];
  if (tid < kTileR) ratio[tid] = r0 + tid < p.n_r ? fx_fraction(p.inv_r[r0 + tid] * recip_newton(inv_r0)) : 0;
  // Courant entries of the stored rows t0 .. t0 + TT + 3 (theta rows t0 - 2 .. t0 + TT + 1)
  for (int i = tid; i < (TT + 4) * NP; i += blockDim.x) {
    const int srow = t0 + i / NP, pr = i % NP;
    CourEntry e{0, 0, 0, 0};
    if (srow < p.rows) {
      const double* c = p.courant64 + ((size_t)srow * NP + pr) * 4;
      const uint64_t alpha = fx_fraction(c[0]);
      e.a2 = fx_mul_frac(alpha, alpha);
      e.k2 = 2 * (alpha - e.a2);
      e.at = fx_fraction(c[2] * inv_r0);
      e.fl = (int)c[3];
    }
    ctab[i] = e;
  }
  __syncthreads();
  // bits 2..6 of the tile rows' flags: bit 1 (v_theta < 0 for q1) of the rows
  // -2 .. +2 around them, the rows whose azimuthal stencils reach the node
  for (int i = tid; i < TT * NP; i += blockDim.x) {
    const int w = 2 + i / NP, pr = i % NP;
    int m = 0;
#pragma unroll
    for (int o = 0; o < 5; ++o) m |= ((ctab[(w - 2 + o) * NP + pr].fl >> 1) & 1) << o;
    ctab[w * NP + pr].fl |= m << 2;
  }
  __syncthreads();
  if (tid == 0)
    for (int s = 0; s < S && s < NP; ++s) issue_pair(s, s);

  // ---- this thread's node -----------------------------------------------------
  const int row = 2 + rowl;
  const int col = kLeft + lane;
  const int t = t0 + rowl;
  const int r = r0 + lane;
  const bool valid = r < p.n_r && t < p.n_theta;
  const int srow = t + kGhostRows;
  const size_t plane_out = (size_t)p.rows * p.pitch;
  const T decay = (T)p.decay;
  T gs[4] = {T(0), T(0), T(0), T(0)};
  if (valid) {
    // (1 - d) g of this node, read from global memory while the first pairs'
    // windows land (the TMA copies then mostly hit L2)
    const int plane = p.rows * p.pitch;
    const size_t off = (size_t)srow * p.pitch + r;
    const T* ln = lam_in + off;
    T rho, ux, uy, E;
    bool nok;
    adj_node_state(f + off, plane, d, rho, ux, uy, E, nok);
    if (!nok) atomicOr(p.status, PCLB_FLAG_NONPHYS);
    T G[4], g[4];
    eq_cotangent<T>(rho, ux, uy, E, d, [&](int q) -> T { return ln[(size_t)q * plane]; }, G);
    to_moment_cotangent<T>(rho, ux, uy, E, G, g);
#pragma unroll
    for (int j = 0; j < 4; ++j) gs[j] = (T(1) - decay) * g[j];
    // the cotangent the ghost nodes return to the two nodes next to each wall
    auto add_wall = [&](int side, int node) {
#pragma unroll
      for (int j = 0; j < 4; ++j) gs[j] += ws.gwall[((size_t)(slots[side] * 2 + node) * p.n_theta + t) * 4 + j];
    };
    if (r == 0) add_wall(0, 0);
    if (r == 1) add_wall(0, 1);
    if (r == p.n_r - 1) add_wall(1, 0);
    if (r == p.n_r - 2) add_wall(1, 1);
  }
  const int o_node = row * kWinR + col;                 // this node in a window plane
  const int p_rad = AR + rowl * RC + lane + 2;          // its radial product slot
  const int p_az = AT + row * kTileR + lane;            // its azimuthal product slot
  const uint64_t my_ratio = ratio[lane];
  auto store = [&](int q, T v) {
    lam_out[(size_t)q * plane_out + (size_t)srow * p.pitch + r] = v;
    if (t >= p.n_theta - 2)
      lam_out[(size_t)d.recv_lo[q] * plane_out + (size_t)(t - (p.n_theta - 2)) * p.pitch + r] = v;
    if (t < 2) lam_out[(size_t)d.recv_hi[q] * plane_out + (size_t)(p.n_theta + kGhostRows + t) * p.pitch + r] = v;
  };
  // rest velocity: no convection
  if (valid) store(0, decay * lam_in[(size_t)srow * p.pitch + r] + gs[0] + gs[3] * d.half_v2[0]);

  // wall tiles: the ghost states of the rows this thread fills (warp 0: inner, warp 1: outer)
  const bool wall_tile = inner || outer;
  const int gside = rowl == 0 ? 0 : 1;
  const bool fills = wall_tile && rowl < 2 && lane < TT && t0 + lane < p.n_theta && (gside == 0 ? inner : outer);
  const EqParams<T>* eg = ws.ghost + (size_t)(slots[gside] * 3) * p.n_theta + t0 + lane;   // layer l at + l n_theta
  const bool gneq = (p.bc_kind[gside] & PCLB_BC_NEQ) != 0;   // its ghosts carry the wall node's departure

  bool ok = true;
  int brk = NP;                                         // the pair at which a wait timed out
#pragma unroll 1
  for (int pair = 0; pair < NP; ++pair) {
    const int k = 1 + pair / (kNDirs / 2);
    const int q1 = 1 + (k - 1) * kNDirs + pair % (kNDirs / 2);
    const int q2 = q1 + kNDirs / 2;                      // opposite velocity
    const int s = pair % S;
    const T* st = ring + s * 4 * PLANE;
    T* pb = prod + (pair & 1) * 2 * PROD;                // this pair's products: [label][...]
    if (ok) ok = p.wait_ns != 0 && mbar_wait_bounded(&bar[s], (uint32_t)((pair / S) & 1), p.wait_ns);
    if (wall_tile) {
      // radial ghost columns of this pair's f planes (f = f^eq of the ghost
      // states, plus the wall node's departure for non-equilibrium ghosts)
      if (fills && ok) {
        T* fw = const_cast<T*>(st) + (2 + lane) * kWinR;
        const int c0 = gside == 0 ? kLeft : cw_out, stp = gside == 0 ? 1 : -1;
        T dep1 = T(0), dep2 = T(0);
        if (gneq) {
          const EqParams<T> ea = eg[(size_t)2 * p.n_theta];
          dep1 = fw[c0] - adj_feq<T>(ea, d, q1);
          dep2 = fw[PLANE + c0] - adj_feq<T>(ea, d, q2);
        }
        for (int l = 0; l < 2; ++l) {
          const int c = c0 - stp * (1 + l);
          if (c < 0 || c >= kWinR) continue;
          const EqParams<T> e = eg[(size_t)l * p.n_theta];
          fw[c] = adj_feq<T>(e, d, q1) + dep1;
          fw[PLANE + c] = adj_feq<T>(e, d, q2) + dep2;
        }
      }
      __syncthreads();
    }

    // (A) products lam(n) M_D(n), lam(n) M_Dp(n) of every node that can reach the
    // tile.  Warp w forms those of tile row w at its 32 columns (both labels),
    // warps 0..3 the halo rows -2, -1, TT, TT + 1 for the label whose upwind
    // side points into the tile, and the next warps the halo columns.  The
    // upwind sides are uniform across a warp (one row), so each warp takes a
    // branch in which the stencil offsets are constants.
    const T* sfp = st;                                    // f q1, f q2 at +PLANE
    const T* slp = st + 2 * PLANE;                        // lam q1, lam q2 at +PLANE
    const CourEntry e = ctab[row * NP + pair];
    const int fl_c = e.fl;                                // flags of this node's row
    T lam_c[2];                                           // lam^{n+1} of both labels at this node
    if (fl_c & 1)
      radial_pair<1, PLANE, PROD, BR - AR>(sfp, slp, pb, o_node, p_rad, e.a2, e.k2, lam_c);
    else
      radial_pair<-1, PLANE, PROD, BR - AR>(sfp, slp, pb, o_node, p_rad, e.a2, e.k2, lam_c);
    // alpha^2 and 2 alpha (1 - alpha) of |C_theta| at this node
    auto azimuthal = [&](uint64_t at, uint64_t& a2, uint64_t& k2) {
      const uint64_t alpha = fx_mul_frac(at, my_ratio);
      a2 = fx_mul_frac(alpha, alpha);
      k2 = 2 * (alpha - a2);
    };
    {
      uint64_t a2, k2;
      azimuthal(e.at, a2, k2);
      if (fl_c & 2)
        azimuthal_pair<kWinR, PLANE, PROD, BT - AT>(sfp, lam_c, pb, o_node, p_az, a2, k2);
      else
        azimuthal_pair<-kWinR, PLANE, PROD, BT - AT>(sfp, lam_c, pb, o_node, p_az, a2, k2);
    }
    if (rowl < 4) {
      // halo rows: warps 0..3 take window rows 0, 1, TT + 2, TT + 3; rows
      // above the tile are read by labels whose upwind side is +theta
      const int rr = rowl < 2 ? rowl : TT + rowl;
      const CourEntry eh = ctab[rr * NP + pair];
      const bool q1_up_pos = (eh.fl & 2) != 0;
      uint64_t ath, kth;
      azimuthal(eh.at, ath, kth);
      const int o = rr * kWinR + col;
      if (rowl < 2)
        azimuthal_one<kWinR>(sfp + (q1_up_pos ? 0 : PLANE) + o, slp + (q1_up_pos ? 0 : PLANE) + o,
                                pb + (q1_up_pos ? 0 : PROD) + AT + rr * kTileR + lane, BT - AT, ath, kth);
      else
        azimuthal_one<-kWinR>(sfp + (q1_up_pos ? PLANE : 0) + o, slp + (q1_up_pos ? PLANE : 0) + o,
                                 pb + (q1_up_pos ? PROD : 0) + AT + rr * kTileR + lane, BT - AT, ath, kth);
    }
    {
      // halo columns: 4 per tile row (label, column); the warps after the first
      // four take them, or warp 0 as well when the tile has too few rows.
      // Upwind at larger r (+1) reads the tile from columns -2, -1, at
      // smaller r from 32, 33.
      constexpr int HW = (4 * TT + 31) / 32;
      constexpr bool kSep = TT >= 4 + HW;
      if (kSep ? (rowl >= 4 && rowl < 4 + HW) : rowl < HW) {
        const int h = (kSep ? rowl - 4 : rowl) * 32 + lane;
        if (h < 4 * TT) {
          const int hr = h >> 2, L = (h >> 1) & 1, j = h & 1;
          const CourEntry eh = ctab[(hr + 2) * NP + pair];
          const int uh = (eh.fl & 1) ? 1 : -1, uL = L ? -uh : uh;
          const int c = uL == 1 ? j - 2 : kTileR + j;
          const int o = (hr + 2) * kWinR + c + kLeft;
          const T* fw = sfp + L * PLANE + o;
          T MD, MP;
          fx_mwb_partials(fw[0] - fw[uL], fw[uL] - fw[2 * uL], eh.a2, eh.k2, MD, MP);
          const T lam = slp[L * PLANE + o];
          pb[L * PROD + AR + hr * RC + c + 2] = lam * MD;
          pb[L * PROD + BR + hr * RC + c + 2] = lam * MP;
        }
      }
    }
    if (__syncthreads_or(!ok)) {
      brk = pair;
      break;
    }
    // the stage of this pair is free: the planes of pair + S start now
    if (tid == 0 && pair + S < NP) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue_pair(pair + S, s);
    }

    // (B) gather at this node: node n = c + j u_n reads f(n), f(n + u_n),
    // f(n + 2 u_n), so dM(n)/df(n) = M_D, dM(n)/df(n + u_n) = M_Dp - M_D,
    // dM(n)/df(n + 2 u_n) = -M_Dp.
    if (valid) {
      T acc[2];
      if (fl_c & 1)
        gather_radial<T, 1, PROD, BR - AR>(pb, p_rad, acc);
      else
        gather_radial<T, -1, PROD, BR - AR>(pb, p_rad, acc);
      const int tneg = fl_c >> 2;                        // bit o: row o - 2 has v_theta < 0 for q1
      if (tneg == 0)
        gather_azimuthal<T, kTileR, PROD, BT - AT>(pb, p_az, acc);
      else if (tneg == 31)
        gather_azimuthal<T, -kTileR, PROD, BT - AT>(pb, p_az, acc);
      else
        gather_azimuthal_mixed<T, PROD, BT - AT>(pb, p_az, tneg, acc);
      const T A = gs[0] + gs[3] * d.half_v2[k];
      const T B = gs[1] * d.vx[q1] + gs[2] * d.vy[q1];
      T o1 = decay * lam_c[0] + (A + B) - acc[0], o2 = decay * lam_c[1] + (A - B) - acc[1];
      if (wall_tile) {
        // non-equilibrium ghosts hand their cotangent straight to f_q of the wall node
        for (int sd = 0; sd < 2; ++sd)
          if ((p.bc_kind[sd] & PCLB_BC_NEQ) && r == (sd == 0 ? 0 : p.n_r - 1)) {
            o1 += ws.gdir[((size_t)slots[sd] * p.n_theta + t) * kQ + q1];
            o2 += ws.gdir[((size_t)slots[sd] * p.n_theta + t) * kQ + q2];
          }
      }
      store(q1, o1);
      store(q2, o2);
    }
  }
  if (brk < NP && tid == 0) {
    // a copy did not land in time: report it, give the copies still in
    // flight (the last one issued into each stage) a bounded time to finish
    atomicOr(p.status, PCLB_FLAG_TIMEOUT);
    const int issued = brk + S < NP ? brk + S : NP;
    for (int s = 0; s < S && s < issued; ++s) {
      const int last = s + ((issued - 1 - s) / S) * S;
      mbar_wait_bounded(&bar[s], (uint32_t)((last / S) & 1), kDefaultWaitNs);
    }
  }
}

template <class T>
cudaError_t launch_adjoint(const CUtensorMap* tmap_f, const CUtensorMap* tmap_l, const CUtensorMap* tmap_fn,
                           const CUtensorMap* tmap_ln, const T* f, const T* lam_in, T* lam_out, unsigned char* scratch,
                           const StepParams& p, const DvmConst<T>& d, cudaStream_t stream) {
  WallScratch<T> ws;
  ws.ghost = reinterpret_cast<EqParams<T>*>(scratch);
  ws.gwall = reinterpret_cast<T*>(scratch + scratch_part((size_t)9 * p.n_theta * 10 * sizeof(T)));
  ws.gdir = reinterpret_cast<T*>(reinterpret_cast<unsigned char*>(ws.gwall) +
                                 scratch_part((size_t)24 * p.n_theta * sizeof(T)));
  const int rows = p.adj_rows;
  AdjOrder order;
  order.nt = (p.n_r + kTileR - 1) / kTileR;
  order.ny = (p.n_theta + rows - 1) / rows;
  // tile 0 and the tiles with r0 >= n_r - 33 are wall tiles
  order.first_outer = p.n_r - 33 > 0 ? (p.n_r - 33 + kTileR - 1) / kTileR : 0;
  if (order.first_outer < 1) order.first_outer = 1;
  if constexpr (sizeof(T) == 4) {
    // FP32: the packed two-nodes-per-thread pair kernel (adjoint_f32x2.cu)
    return launch_adjoint_pairs_f32(tmap_f, tmap_l, tmap_fn, tmap_ln, f, lam_in, lam_out, ws, order, p, d, stream);
  } else {
    auto go = [&](auto tt) {
      constexpr int TT = decltype(tt)::value;
      static std::atomic<unsigned long long> configured{0};
      const cudaError_t e = set_smem_once(adjoint_pair_kernel<TT>, AdjSize<TT>::smem, configured);
      if (e != cudaSuccess) return e;
      return launch_overlapped(adjoint_pair_kernel<TT>, dim3((unsigned)order.blocks()), AdjSize<TT>::threads,
                               AdjSize<TT>::smem, stream, *tmap_f, *tmap_l, f, lam_in, lam_out, ws, order, p, d);
    };
    return rows == kAdjRows64 ? go(std::integral_constant<int, kAdjRows64>{})
                              : go(std::integral_constant<int, kAdjRows64Small>{});
  }
}

size_t adjoint_scratch_bytes(int n_theta, int elem) {
  // the parts of WallScratch: three slots of 3 EqParams (10 values), of 2 x 4
  // values and of Q values per row
  return scratch_part((size_t)9 * n_theta * 10 * elem) + scratch_part((size_t)24 * n_theta * elem) +
         scratch_part((size_t)3 * n_theta * kQ * elem);
}

template cudaError_t launch_adjoint<float>(const CUtensorMap*, const CUtensorMap*, const CUtensorMap*,
                                           const CUtensorMap*, const float*, const float*, float*, unsigned char*,
                                           const StepParams&, const DvmConst<float>&, cudaStream_t);
template cudaError_t launch_adjoint<double>(const CUtensorMap*, const CUtensorMap*, const CUtensorMap*,
                                            const CUtensorMap*, const double*, const double*, double*, unsigned char*,
                                            const StepParams&, const DvmConst<double>&, cudaStream_t);

}  // namespace pclb
