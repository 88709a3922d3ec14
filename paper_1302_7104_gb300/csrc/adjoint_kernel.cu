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
// TT = 8 rows, one thread per node; on grids whose tiles would leave SMs idle
// 4 rows and two threads per node (LS = 2), one label of each pair each, or 2
// rows and four threads (LS = 4), which also work on two pairs at a time (half
// the barriers): 64 x 128, 73.3 us per adjoint step with LS = 4, 103 with LS = 2,
// 154 with 8 rows.
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

// Courant entry of one pair of opposite velocities at one theta row: alpha^2 and
// 2 alpha (1 - alpha) of alpha = |C_r| in units of 2^-(63 + sr), and |C_theta| at
// the tile's first column in units of 2^-(63 + st) (in plain units of 2^-63 the
// partials of an alpha of 1e-10 had 30 digits left); flag bit 0 set when v_r <
// 0 and bit 1 when v_theta < 0 for the first label of the pair.
struct alignas(32) CourEntry {
  uint64_t a2, k2, at;
  int fl;
  int16_t sr, st;
};

// bytes of one part of the wall scratch, aligned for the next
static size_t scratch_part(size_t bytes) { return (bytes + 255) & ~(size_t)255; }

constexpr int kAdjStages = 2;   // ring depth of the pair-streaming kernel (2 measured best of 1..4)
static_assert(sizeof(EqParams<float>) == 10 * sizeof(float) && sizeof(EqParams<double>) == 10 * sizeof(double),
              "ghost-state scratch holds 10 values per EqParams");

// TT rows; LS = 2: two threads per node, one label of each pair each; LS = 4:
// four, and two pairs at a time.
template <int TT, int LS>
struct AdjSize {
  static constexpr int threads = 32 * TT * LS;
  static constexpr int pp = LS == 4 ? 2 : 1;   // pairs at a time
  static constexpr int min_blocks = 2;   // what shared memory allows with 8 rows, and 124 registers with fewer
  static constexpr int plane = kWinR * (TT + 4);
  static constexpr int npairs = 4 * kNDirs / 2;
  // products of one label: radial A, B over TT rows x 36 columns (tile
  // columns -2 .. 33), azimuthal A, B over TT + 4 rows (-2 .. TT + 1) x 32
  static constexpr int rcols = kTileR + 4;
  static constexpr int prod = 2 * TT * rcols + 2 * (TT + 4) * kTileR;
  static constexpr int ring_bytes = kAdjStages * pp * 4 * plane * 8;   // f, f', lam, lam' per stage and pair
  static constexpr int prod_bytes = 2 * pp * 2 * prod * 8;             // 2 buffers x 2 labels of each pair
  static constexpr int ratio_bytes = kTileR * 8;
  static constexpr int tab_bytes = (TT + 4) * npairs * (int)sizeof(CourEntry);
  static constexpr int ghost_bytes = 2 * 2 * TT * kQ * 8;         // both walls' ghost values
  static constexpr int smem = ring_bytes + prod_bytes + ratio_bytes + tab_bytes + ghost_bytes + 128;
  static_assert(LS == 1 || LS * 12 * 32 * TT * 8 <= prod_bytes, "exchange of the node phase inside the product buffers");
  // the ring's planes are TMA destinations: 128-byte aligned
  static_assert((plane * 8) % 128 == 0, "TMA destinations must stay 128-byte aligned");
};

namespace {


// ---- the pair-streaming kernel's stencil pieces ------------------------------
// lam(n) M_D(n), lam(n) M_Dp(n) of one label at one node in one direction, its
// upwind neighbours at offsets u and 2u, to P and P + DB.
__device__ __forceinline__ void products(const double* f, int u, double lam, double* P, int DB, uint64_t a2, uint64_t k2,
                                         int s) {
  double MD, MP;
  const double f1 = f[u];
  fx_mwb_partials(f[0] - f1, f1 - f[2 * u], a2, k2, s, MD, MP);
  P[0] = lam * MD;
  P[DB] = lam * MP;
}

// Gather of one label's products at one node: the node n = c + j u reads f(n),
// f(n + u), f(n + 2 u), so dM(n)/df(c) collects M_D of n = c, M_Dp - M_D of
// n = c - u and -M_Dp of n = c - 2u.
__device__ __forceinline__ double gather(const double* P, int DB, int u) { return P[0] - P[-u] + P[DB - u] - P[DB - 2 * u]; }

// The azimuthal gather where the upwind side changes within the five rows: bit
// o of neg set when row o - 2 has v_theta < 0 for this label (its reader of row 0
// is then the row below it).
__device__ __forceinline__ double gather_mixed(const double* P, int DB, int neg) {
  double a = P[0];
  if (neg & 2) a += P[DB - kTileR] - P[-kTileR];
  if (!(neg & 8)) a += P[DB + kTileR] - P[kTileR];
  if (neg & 1) a -= P[DB - 2 * kTileR];
  if (!(neg & 16)) a -= P[DB + 2 * kTileR];
  return a;
}

// The sums of eq_cotangent (adjoint_common.cuh) over shells k0 .. k1, and the
// rest velocity's if l0 is given: A, Bx, By, Cs, Dx, Fq.
template <class LamFn>
__device__ __forceinline__ void cotangent_sums(double ux, double uy, double E, const DvmConst<double>& d, int k0, int k1,
                                               const double* l0, LamFn lam, double o[6]) {
  const double invE = recip_newton(E);
  const double s = (ux * ux + uy * uy) * invE;
  const double a1 = 1.0 - 0.5 * s, a0 = a1 + 0.125 * s * s;
  const double uxE = ux * invE, uyE = uy * invE;
  auto weight = [&](int k, double& F, double& Fd) {   // F_k(E) and its derivative
    const double* c = d.Fc[k];
    F = E * (c[0] + E * (c[1] + E * (c[2] + E * c[3])));
    Fd = c[0] + E * (2.0 * c[1] + E * (3.0 * c[2] + E * 4.0 * c[3]));
  };
#pragma unroll
  for (int j = 0; j < 6; ++j) o[j] = 0.0;
  if (l0) {   // x = 0
    double Fs = 0.0, Fds = 0.0;
#pragma unroll
    for (int k = 1; k <= 4; ++k) {
      double F, Fd;
      weight(k, F, Fd);
      Fs += F;
      Fds += Fd;
    }
    const double l0F = *l0 * (1.0 - d.B0 * Fs);
    o[0] = l0F * a0;
    o[3] = l0F * (-0.5 + 0.25 * s);
    o[5] = *l0 * (-d.B0 * Fds) * a0;
  }
  constexpr int half = kNDirs / 2;
#pragma unroll 1
  for (int k = k0; k <= k1; ++k) {
    double F, Fd, Ak = 0, Bxk = 0, Byk = 0, Ck = 0, Dk = 0;
    weight(k, F, Fd);
#pragma unroll
    for (int i = 0; i < half; ++i) {
      const int q = 1 + (k - 1) * kNDirs + i;
      pair_terms<double>(d.vx[q], d.vy[q], uxE, uyE, s, a0, a1, lam(q), lam(q + half), Ak, Bxk, Byk, Ck, Dk);
    }
    o[0] += F * Ak;
    o[1] += F * Bxk;
    o[2] += F * Byk;
    o[3] += F * Ck;
    o[4] += F * Dk;
    o[5] += Fd * Ak;
  }
}

}  // namespace

// ---------------------------------------------------------------------------
// Pair-streaming part.
// ---------------------------------------------------------------------------
template <int TT, int LS>
__global__ void __launch_bounds__(AdjSize<TT, LS>::threads, AdjSize<TT, LS>::min_blocks)
    adjoint_pair_kernel(const __grid_constant__ CUtensorMap tmap_f, const __grid_constant__ CUtensorMap tmap_l,
                        const double* f, const double* lam_in, double* __restrict__ lam_out,
                        const __grid_constant__ WallScratch<double> ws, const __grid_constant__ AdjOrder order,
                        const __grid_constant__ StepParams p, const __grid_constant__ DvmConst<double> d) {
  using T = double;
  using SZ = AdjSize<TT, LS>;
  constexpr int PLANE = SZ::plane;
  constexpr int NP = SZ::npairs, RC = SZ::rcols, PROD = SZ::prod;
  constexpr int S = kAdjStages, PP = SZ::pp, NIT = NP / PP;   // stages; pairs at a time, iterations
  // offsets inside one label's products
  constexpr int AR = 0, BR = TT * RC, AT = 2 * TT * RC, BT = 2 * TT * RC + (TT + 4) * kTileR;
  constexpr uint32_t kStageBytes = (uint32_t)(PP * 4 * PLANE * sizeof(T));
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* ring = reinterpret_cast<T*>(smem_raw);                 // [stage][pair][f q1, f q2, lam q1, lam q2][PLANE]
  T* prod = ring + S * PP * 4 * PLANE;                        // [buffer][pair][label][products]
  uint64_t* ratio = reinterpret_cast<uint64_t*>(prod + 2 * PP * 2 * PROD);   // 1/r of the tile columns relative to the first
  CourEntry* ctab = reinterpret_cast<CourEntry*>(ratio + kTileR);        // [TT + 4][NP]
  T* gval = reinterpret_cast<T*>(ctab + (TT + 4) * NP);                  // [side][layer][TT][Q] ghost values
  uint64_t* bar = reinterpret_cast<uint64_t*>(gval + 2 * 2 * TT * kQ);   // [S]

  int tx, ty;
  order.tile(blockIdx.x, tx, ty);
  const int r0 = tx * kTileR;
  const int t0 = ty * TT;
  const int tid = threadIdx.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int rowl = warp % TT;               // tile row
  const int part = warp / TT;               // of LS threads per node
  const int half_of = part & 1, pair_of = part >> 1;   // this thread's label of a pair, and pair of those at a time

  // the planes of iteration it's pairs (labels q1, q1 + N_i/2) into stage s (thread 0)
  auto issue_pairs = [&](int it, int s) {
    mbar_arrive_expect_tx(&bar[s], kStageBytes);
#pragma unroll
    for (int j = 0; j < PP; ++j) {
      const int pr = it * PP + j, k = 1 + pr / (kNDirs / 2);
      const int q1 = 1 + (k - 1) * kNDirs + pr % (kNDirs / 2), q2 = q1 + kNDirs / 2;
      T* st = ring + (s * PP + j) * 4 * PLANE;
      tma_load_3d(st, &tmap_f, r0 - kLeft, t0, q1, &bar[s]);
      tma_load_3d(st + PLANE, &tmap_f, r0 - kLeft, t0, q2, &bar[s]);
      tma_load_3d(st + 2 * PLANE, &tmap_l, r0 - kLeft, t0, q1, &bar[s]);
      tma_load_3d(st + 3 * PLANE, &tmap_l, r0 - kLeft, t0, q2, &bar[s]);
    }
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
      adjoint_walls<T, TT>(f, lam_in, side, slots[side], t0, ws, *reinterpret_cast<WallShared<T, TT>*>(ctab),
                           gval + side * 2 * TT * kQ, p, d);
  const double inv_r0 = p.inv_r[r0];
  if (tid < kTileR) ratio[tid] = r0 + tid < p.n_r ? fx_fraction(p.inv_r[r0 + tid] * recip_newton(inv_r0)) : 0;
  // Courant entries of the stored rows t0 .. t0 + TT + 3 (theta rows t0 - 2 .. t0 + TT + 1)
  for (int i = tid; i < (TT + 4) * NP; i += blockDim.x) {
    const int srow = t0 + i / NP, pr = i % NP;
    CourEntry e{0, 0, 0, 0, 0, 0};
    if (srow < p.rows) {
      const double* c = p.courant64 + ((size_t)srow * NP + pr) * 4;
      const FxScaled r = fx_scaled(c[0]), th = fx_scaled(c[2] * inv_r0);
      fx_partial_coefs(r, e.a2, e.k2);
      e.at = th.a;
      e.sr = (int16_t)r.s;
      e.st = (int16_t)th.s;
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
    for (int s = 0; s < S && s < NIT; ++s) issue_pairs(s, s);

  // ---- this thread's node -----------------------------------------------------
  const int row = 2 + rowl;
  const int col = kLeft + lane;
  const int t = t0 + rowl;
  const int r = r0 + lane;
  const bool valid = r < p.n_r && t < p.n_theta;
  const int srow = t + kGhostRows;
  const size_t plane_out = (size_t)p.rows * p.pitch;
  const T decay = (T)p.decay;
  T gs[4];
  {
    // (1 - d) g of this node, read from global memory while the first pairs'
    // windows land (the TMA copies then mostly hit L2); threads without a node
    // repeat the nearest one
    const size_t plane = plane_out;
    const size_t off = (size_t)(min(t, p.n_theta - 1) + kGhostRows) * p.pitch + min(r, p.n_r - 1);
    const T* fn = f + off;
    const T* ln = lam_in + off;
    T* all = prod + (rowl * 32 + lane) * LS * 12;                // exchange of the node's threads, which share the shells
    T* mine = all + part * 12;
    const int k0 = LS == 1 ? 1 : 4 / LS * part + 1, k1 = k0 + 4 / LS - 1;
    const T lam0 = ln[0];
    T m[4] = {part == 0 ? fn[0] : T(0), T(0), T(0), T(0)};    // rho, j_x, j_y, e
#pragma unroll 1
    for (int k = k0; k <= k1; ++k) {
      T S = T(0), D[kNDirs / 2];
#pragma unroll
      for (int i = 0; i < kNDirs / 2; ++i) {
        const int q = 1 + (k - 1) * kNDirs + i;
        const T a = fn[(size_t)q * plane], b = fn[(size_t)(q + kNDirs / 2) * plane];
        S += a + b;
        D[i] = a - b;
      }
      m[0] += S;
      m[1] = fma(d.speed[k], fma(d.cx[2], D[1] - D[3], D[0]), m[1]);
      m[2] = fma(d.speed[k], fma(d.cx[2], D[1] + D[3], D[2]), m[2]);
      m[3] = fma(d.half_v2[k], S, m[3]);
    }
    // the sums of the node's threads' values j0 .. j0 + n - 1
    auto exchange = [&](T* v, int j0, int n) {
#pragma unroll
      for (int j = 0; j < n; ++j) mine[j0 + j] = v[j];
      __syncthreads();
#pragma unroll
      for (int j = 0; j < n; ++j) {
        v[j] = all[j0 + j];
#pragma unroll
        for (int o = 1; o < LS; ++o) v[j] += all[o * 12 + j0 + j];
      }
    };
    if constexpr (LS > 1) exchange(m, 0, 4);
    const NodeState<T> st = node_state64(m[0], m[1], m[2], m[3]);
    if (valid && !st.ok) atomicOr(p.status, PCLB_FLAG_NONPHYS);
    T c[6];
    cotangent_sums(st.ux, st.uy, st.E, d, k0, k1, part == 0 ? &lam0 : nullptr,
                   [&](int q) -> T { return ln[(size_t)q * plane]; }, c);
    if constexpr (LS > 1) {
      exchange(c, 4, 6);
      __syncthreads();   // read before the pairs' products take the buffer
    }
    const T invE = recip_newton(st.E), s = (st.ux * st.ux + st.uy * st.uy) * invE, rE = st.rho * invE;
    const T G[4] = {c[0], rE * (c[1] + T(2) * st.ux * c[3]), rE * (c[2] + T(2) * st.uy * c[3]),
                    st.rho * (c[5] - (c[4] + s * c[3]) * invE)};
    T g[4];
    to_moment_cotangent<T>(st.rho, st.ux, st.uy, st.E, G, g);
#pragma unroll
    for (int j = 0; j < 4; ++j) gs[j] = (T(1) - decay) * g[j];
    // the cotangent the ghost nodes return to the two nodes next to each wall
    auto add_wall = [&](int side, int node) {
#pragma unroll
      for (int j = 0; j < 4; ++j) gs[j] += ws.gwall[((size_t)(slots[side] * 2 + node) * p.n_theta + t) * 4 + j];
    };
    if (valid && r == 0) add_wall(0, 0);
    if (valid && r == 1) add_wall(0, 1);
    if (valid && r == p.n_r - 1) add_wall(1, 0);
    if (valid && r == p.n_r - 2) add_wall(1, 1);
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
  if (valid && part == 0) store(0, decay * lam_in[(size_t)srow * p.pitch + r] + gs[0] + gs[3] * d.half_v2[0]);

  const bool wall_tile = inner || outer;

  bool ok = true;
  int brk = NIT;                                        // the iteration at which a wait timed out
#pragma unroll 1
  for (int it = 0; it < NIT; ++it) {
    const int pair = it * PP + pair_of;
    const int k = 1 + pair / (kNDirs / 2);
    const int q1 = 1 + (k - 1) * kNDirs + pair % (kNDirs / 2);
    const int q2 = q1 + kNDirs / 2;                      // opposite velocity
    const int s = it % S;
    T* stage = ring + s * PP * 4 * PLANE;
    T* buffer = prod + (it & 1) * PP * 2 * PROD;
    const T* st = stage + pair_of * 4 * PLANE;
    T* pb = buffer + pair_of * 2 * PROD;                 // this pair's products: [label][...]
    if (ok) ok = p.wait_ns != 0 && mbar_wait_bounded(&bar[s], (uint32_t)((it / S) & 1), p.wait_ns);
    if (wall_tile) {
      // radial ghost columns of the pairs' f planes: pair, wall, layer, label, row
      if (tid < 8 * TT * PP && ok) {
        const int rr = tid % TT, L = tid / TT & 1, l = tid / (2 * TT) & 1, side = tid / (4 * TT) & 1, j = tid / (8 * TT);
        const int c = (side == 0 ? kLeft : cw_out) - (side == 0 ? 1 : -1) * (1 + l), pr = it * PP + j;
        const int q = 1 + pr / (kNDirs / 2) * kNDirs + pr % (kNDirs / 2) + L * (kNDirs / 2);
        if ((side == 0 ? inner : outer) && t0 + rr < p.n_theta && c >= 0 && c < kWinR)
          stage[(j * 4 + L) * PLANE + (2 + rr) * kWinR + c] = gval[((side * 2 + l) * TT + rr) * kQ + q];
      }
      __syncthreads();
    }

    // (A) products lam(n) M_D(n), lam(n) M_Dp(n) of every node that can reach the
    // tile: each thread those of its node (both labels, or its own), warps
    // 0..3 the halo rows -2, -1, TT, TT + 1 for the label whose upwind side
    // points into the tile, and the next warp the halo columns.
    const T* sfp = st;                                    // f q1, f q2 at +PLANE
    const T* slp = st + 2 * PLANE;                        // lam q1, lam q2 at +PLANE
    const CourEntry e = ctab[row * NP + pair];
    const int fl_c = e.fl;                                // flags of this node's row
    // label L's upwind offsets at this node's row
    auto up_r = [&](int L) { return ((fl_c & 1) != 0) != (L != 0) ? 1 : -1; };
    auto up_t = [&](int L) { return ((fl_c & 2) != 0) != (L != 0) ? kWinR : -kWinR; };
    // alpha^2 and 2 alpha (1 - alpha) of |C_theta| at this thread's column
    auto azimuthal = [&](const CourEntry& x, uint64_t& a2, uint64_t& k2) {
      fx_partial_coefs(FxScaled{fx_mul_frac(x.at, my_ratio), x.st}, a2, k2);
    };
    T lam_c[LS == 1 ? 2 : 1];                             // lam^{n+1} of the label(s) at this node
    {
      uint64_t a2, k2;
      azimuthal(e, a2, k2);
#pragma unroll
      for (int j = 0; j < (LS == 1 ? 2 : 1); ++j) {
        const int L = LS == 1 ? j : half_of;
        const T* fw = sfp + L * PLANE + o_node;
        lam_c[j] = slp[L * PLANE + o_node];
        products(fw, up_r(L), lam_c[j], pb + L * PROD + p_rad, BR - AR, e.a2, e.k2, e.sr);
        products(fw, up_t(L), lam_c[j], pb + L * PROD + p_az, BT - AT, a2, k2, e.st);
      }
    }
    if (warp < 4 * PP) {
      // halo rows: window rows 0, 1, TT + 2, TT + 3; rows above the tile are
      // read by labels whose upwind side is +theta
      const int h = warp & 3, j = warp >> 2, rr = h < 2 ? h : TT + h;
      const CourEntry eh = ctab[rr * NP + it * PP + j];
      const bool q1_up_pos = (eh.fl & 2) != 0;
      uint64_t a2, k2;
      azimuthal(eh, a2, k2);
      const int L = (h < 2) == q1_up_pos ? 0 : 1, o = rr * kWinR + col;
      const T* w = stage + j * 4 * PLANE + L * PLANE + o;
      products(w, h < 2 ? kWinR : -kWinR, w[2 * PLANE], buffer + (j * 2 + L) * PROD + AT + rr * kTileR + lane, BT - AT, a2,
               k2, eh.st);
    }
    if (warp == (PP == 1 ? 4 : TT * LS - 1)) {
      // halo columns: 4 per pair and tile row (label, column).  Upwind at larger r
      // (+1) reads the tile from columns -2, -1, at smaller r from 32, 33.
      static_assert(4 * TT * PP <= 32 && TT * LS >= 5 && TT * LS >= 4 * PP, "halo rows and columns: a warp each");
      if (lane < 4 * TT * PP) {
        const int hr = (lane >> 2) % TT, j = lane / (4 * TT), L = (lane >> 1) & 1, i = lane & 1;
        const CourEntry eh = ctab[(hr + 2) * NP + it * PP + j];
        const int u = ((eh.fl & 1) != 0) != (L != 0) ? 1 : -1;
        const int c = u == 1 ? i - 2 : kTileR + i;
        const T* w = stage + (j * 4 + L) * PLANE + (hr + 2) * kWinR + c + kLeft;
        products(w, u, w[2 * PLANE], buffer + (j * 2 + L) * PROD + AR + hr * RC + c + 2, BR - AR, eh.a2, eh.k2, eh.sr);
      }
    }
    if (__syncthreads_or(!ok)) {
      brk = it;
      break;
    }
    // the stage is free: the planes of iteration it + S start now
    if (tid == 0 && it + S < NIT) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      issue_pairs(it + S, s);
    }

    // (B) gather at this node
    if (valid) {
      const T A = gs[0] + gs[3] * d.half_v2[k];
      const T B = gs[1] * d.vx[q1] + gs[2] * d.vy[q1];
      const int tneg = fl_c >> 2;                        // bit o: row o - 2 has v_theta < 0 for q1
#pragma unroll
      for (int j = 0; j < (LS == 1 ? 2 : 1); ++j) {
        const int L = LS == 1 ? j : half_of, q = L ? q2 : q1;
        const T* P = pb + L * PROD;
        T acc = gather(P + p_rad, BR - AR, up_r(L));
        // one side for all rows -2 .. +2 around the node: the readers sit
        // upwind's opposite way; else row by row
        if (tneg == 0 || tneg == 31)
          acc += gather(P + p_az, BT - AT, (tneg == 0) == (L == 0) ? -kTileR : kTileR);
        else
          acc += gather_mixed(P + p_az, BT - AT, L ? tneg ^ 0x1f : tneg);
        T o = decay * lam_c[j] + (L ? A - B : A + B) - acc;
        if (wall_tile) {
          // non-equilibrium ghosts hand their cotangent straight to f_q of the wall node
          for (int sd = 0; sd < 2; ++sd)
            if ((p.bc_kind[sd] & PCLB_BC_NEQ) && r == (sd == 0 ? 0 : p.n_r - 1))
              o += ws.gdir[((size_t)slots[sd] * p.n_theta + t) * kQ + q];
        }
        store(q, o);
      }
    }
  }
  if (brk < NIT && tid == 0) {
    // a copy did not land in time: report it, give the copies still in
    // flight (the last one issued into each stage) a bounded time to finish
    atomicOr(p.status, PCLB_FLAG_TIMEOUT);
    const int issued = brk + S < NIT ? brk + S : NIT;
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
    auto go = [&](auto tt, auto ls) {
      constexpr int TT = decltype(tt)::value, LS = decltype(ls)::value;
      static std::atomic<unsigned long long> configured{0};
      const cudaError_t e = set_smem_once(adjoint_pair_kernel<TT, LS>, std::max(AdjSize<TT, LS>::smem, kOwnSmBytes), configured);
      if (e != cudaSuccess) return e;
      return launch_overlapped(adjoint_pair_kernel<TT, LS>, dim3((unsigned)order.blocks()), AdjSize<TT, LS>::threads,
                               adjoint_smem(AdjSize<TT, LS>::smem, order.blocks()), stream, *tmap_f, *tmap_l, f, lam_in, lam_out, ws, order, p, d);
    };
    if (rows == kAdjRows64) return go(std::integral_constant<int, kAdjRows64>{}, std::integral_constant<int, 1>{});
    if (rows == kAdjRows64Small) return go(std::integral_constant<int, kAdjRows64Small>{}, std::integral_constant<int, 2>{});
    return go(std::integral_constant<int, kAdjRows64Tiny>{}, std::integral_constant<int, 4>{});
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
