// Fused FP32 time step of the polar-coordinate FDLB model (Eq. 38), the hot
// kernel of the library.
//
// Work per CTA: a tile of 32 (r) x TT (theta) nodes, 256 threads.  One thread
// issues 33 TMA box copies (one per velocity plane) of the window
// [r0-4, r0+36) x [t0-2, t0+TT+2) into shared memory, in four groups with a
// barrier each (rest + shell 1, shells 2, 3, 4), while the others copy the
// tile's rows of the host-computed Courant table.  Each thread then owns two
// radially adjacent nodes of one row and processes them together with packed
// FP32x2 arithmetic:
//   * moments (Eqs. 3-5), temperature recovery and the weights rho F_k(E)
//     (Eqs. 11a-b) in float-float arithmetic, so that the rounded equilibrium
//     keeps the collision invariants of the exact one;
//   * radial ghost columns for tiles at a wall (Eq. 39, f = f^eq), computed in
//     shared memory by one warp per wall;
//   * for every pair (q, q') of opposite velocities of a shell: v_q.u/E from
//     float-float constants, the even and odd parts of the equilibrium
//     polynomial (Eq. 10) shared by q and q'; then per velocity the relaxation
//     (Eq. 19) minus the MWB increments (Eq. 28) in r and theta, stored with
//     8-byte streaming stores, plus the azimuthal ghost rows of the seam
//     (Eq. 40).  The convection increments -M_r - M_theta are summed first
//     and added once to the relaxed value, so that they cost one rounding at
//     the magnitude of f instead of four (this halves the FP32 path's drift
//     from the FP64 one over long runs).
// TT = 16: one thread per node pair, for grids that fill the chip with such
// tiles.  TT = 4: four threads per node pair, a shell each (the node state
// formed by all four), and two warps of their own for the ghost columns; for
// small grids, where the latency of one tile is the time of the step.  The results
// do not depend on TT.
// Consecutive steps overlap their starts: a step's launch, barrier set-up and
// table rows run while the step before it drains (programmatic dependent
// launch); its window copies wait for that step.
#include <cuda.h>
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "f32_eq2.cuh"
#include "f32_state.cuh"
#include "f32x2.cuh"
#include "pclb_internal.h"

namespace pclb {

namespace {

constexpr int kPairs = 4 * kHalf;                    // 16
template <int TT>
struct F32Size {
  static constexpr int split = 16 / TT;                          // threads per node pair
  static constexpr int plane = kWinR * (TT + 4);                 // floats per plane window
  static constexpr int planes_bytes = kQ * plane * 4;            // 105600 for TT = 16
  static constexpr int tab_bytes = kPairs * TT * 16;             // one float4 per (pair, row)
  // split: the node pairs' exchange, [4 groups][7] terms, f_0, then [4 shells][2] weights
  static constexpr int pairs = 16 * TT;
  static constexpr int exchange_bytes = split > 1 ? (29 + 8) * pairs * 8 : 0;
  static constexpr int smem = planes_bytes + tab_bytes + exchange_bytes + 128;
  static constexpr int threads = kStepThreads32 + (split > 1 ? 64 : 0);   // two warps for the ghost columns
  // every plane window is a TMA destination: 128-byte aligned (a tile height
  // whose window breaks this faults with a misaligned address)
  static_assert((plane * 4) % 128 == 0 && planes_bytes % 16 == 0, "TMA destinations must stay 128-byte aligned");
};
constexpr int kGroups = 4;
__device__ __forceinline__ int group_first(int g) { return g == 0 ? 0 : 1 + g * kNDirs; }
__device__ __forceinline__ int group_planes(int g) { return g == 0 ? 1 + kNDirs : kNDirs; }

__device__ __forceinline__ f2 ld2(const float* p) { return *reinterpret_cast<const float2*>(p); }

// The state of the two nodes.  ready(g) is called before plane group g (the
// rest plane and shell 1, then shells 2, 3, 4) is first read, so the sums start
// while later groups still land.
template <int PL, class Ready>
__device__ __forceinline__ State2 state2(const float* f, const DvmConst<float>& d, Ready ready) {
  auto ld = [&](int q) { return ld2(f + q * PL); };
  ready(0);
  Moments2 m(ld(0));
  m.template add<0>(group_terms2<0>(ld, d));
  ready(1);
  ready(2);
  m.template add<1>(group_terms2<1>(ld, d));
  m.template add<2>(group_terms2<2>(ld, d));
  ready(3);
  m.template add<3>(group_terms2<3>(ld, d));
  return m.state();
}

// The same with the groups spread over the four threads of a node pair (thread
// `split` forms group `split`), which exchange them through x [group][7][pairs]
// (`pairs` node pairs, this one `ip`).  barrier() joins the threads and tells
// whether all of them have their planes.
template <int PL, class Ready, class Barrier>
__device__ __forceinline__ State2 state2_split(const float* f, const DvmConst<float>& d, int split, f2* x, int pairs,
                                               int ip, Ready ready, Barrier barrier) {
  auto ld = [&](int q) { return ld2(f + q * PL); };
  Terms2 t;
  switch (split) {
    case 0: ready(0); t = group_terms2<0>(ld, d); break;
    case 1: ready(1); ready(2); t = group_terms2<1>(ld, d); break;
    case 2: ready(2); t = group_terms2<2>(ld, d); break;
    default: ready(3); t = group_terms2<3>(ld, d); break;
  }
  f2* o = x + split * 7 * pairs + ip;
  o[0] = t.S;
  o[1 * pairs] = t.jx.hi; o[2 * pairs] = t.jx.lo;
  o[3 * pairs] = t.jy.hi; o[4 * pairs] = t.jy.lo;
  o[5 * pairs] = t.e.hi;  o[6 * pairs] = t.e.lo;
  if (split == 0) x[28 * pairs + ip] = ld2(f);
  barrier();
  auto get = [&](int g) {
    const f2* i = x + g * 7 * pairs + ip;
    return Terms2{i[0], ff2{i[1 * pairs], i[2 * pairs]}, ff2{i[3 * pairs], i[4 * pairs]}, ff2{i[5 * pairs], i[6 * pairs]}};
  };
  Moments2 m(x[28 * pairs + ip]);
  m.template add<0>(get(0));
  m.template add<1>(get(1));
  m.template add<2>(get(2));
  m.template add<3>(get(3));
  return m.state();
}

// Ghost columns of one wall (wall node at window column cw) for the tile's TT
// rows, by one warp, Sec. II C 1: lane (row, node) forms the state of the wall
// node a or of the next node b, then lane (row, layer) the layer's state and
// its equilibrium.  (One lane per row forming both states and both layers took
// about 8 of the 19 us of a small step.)  With TT = 4 the four groups of lanes
// share that work shell by shell, with shuffles: the sums of Eqs. 3-5, the
// weights of Eq. 11 and the values stored; what does not depend on f is formed
// before ready() waits for the planes.  Same operations, same results.
template <int TT, class Ready>
__device__ __noinline__ void ghost_columns_f32(float* sm, int lane, int side, int cw, int t0, const StepParams& p,
                                               const DvmConst<float>& d, Ready ready) {
  constexpr int PL = F32Size<TT>::plane;
  constexpr bool kShare = TT == 4;
  static_assert(TT == 16 || TT == 4, "32 lanes: row, node, and for 4 rows the shell");
  const int step = side == 0 ? 1 : -1;
  const int row = 2 + lane % TT, layer = (lane / TT) & 1, group = lane / (2 * TT);
  const int base = lane % (2 * TT);   // this lane's (row, node) in group 0
  const int t = min(t0 + lane % TT, p.n_theta - 1);
  const int kind = p.bc_kind[side] & ~PCLB_BC_NEQ;
  const bool neq = (p.bc_kind[side] & PCLB_BC_NEQ) != 0;

  State32 g;   // the layer's state: prescribed components first
  if (kind != PCLB_BC_EXTRAP) {
    const double c = p.cos_t[t], s = p.sin_t[t];
    const double* v = p.bc_vals + (size_t)((side * 2 + layer) * 4) * p.n_theta + t;
    const double ur = v[1 * p.n_theta], ut = v[2 * p.n_theta];
    g.ux = ff_from(ur * c - ut * s);
    g.uy = ff_from(ur * s + ut * c);
    if (kind == PCLB_BC_DIRICHLET) {
      g.rho = ff_from(v[0]);
      g.E = ff_from(v[3 * p.n_theta]);
    }
  }
  // equilibrium factors of a state; with kShare w[1] holds the weight of
  // shell group + 1
  auto factors = [&](const State32& s) {
    if constexpr (!kShare) {
      return eq32(s, d);
    } else {
      Eq32 q;
      const ff F = shell_weight32(s.E, d, group + 1);
      ff sum = ff_of(0.f);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        sum = ff_add(sum, ff{__shfl_sync(0xffffffffu, F.hi, base + k * 2 * TT), __shfl_sync(0xffffffffu, F.lo, base + k * 2 * TT)});
      const ff wk = ff_mul(s.rho, F);
      q.w[1] = wk.hi + wk.lo;
      q.w[0] = rest_weight32(s.rho, sum, d);
      eq32_polynomial(s, d, q);
      return q;
    }
  };
  Eq32 e;
  if (kind == PCLB_BC_DIRICHLET) e = factors(g);

  if (!ready()) return;   // uniform: the tile is given up
  const float* fn = sm + row * kWinR + cw + (layer == 0 ? 0 : step);
  State32 m;
  if constexpr (!kShare) {
    m = state32(fn, PL, d);
  } else {
    const int k = group + 1;   // groups: shells 1; 2 + 3; 3; 4
    float S, X, Xl, Y, Yl;
    group_sums32(fn + (1 + (k - 1) * kNDirs) * PL, group == 1 ? fn + (1 + 2 * kNDirs) * PL : nullptr, PL, d, S, X, Xl, Y, Yl);
    const ff v = group == 2 ? ff{d.dv23, d.dv23_lo} : ff{d.speed[k], d.speed_lo[k]};
    const ff h = group == 2 ? ff{d.dh23, d.dh23_lo} : ff{d.half_v2[k], d.half_v2_lo[k]};
    const ff tx = ff_mul(v, ff{X, Xl}), ty = ff_mul(v, ff{Y, Yl}), te = ff_mul(h, ff_of(S));
    ff rho = ff_of(fn[0]), jx = ff_of(0.f), jy = jx, en = jx;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int from = base + i * 2 * TT;
      auto get = [&](float x) { return __shfl_sync(0xffffffffu, x, from); };
      const float Si = get(S);
      if (i != 2) rho = ff_add(rho, ff_of(Si));
      jx = ff_add(jx, ff{get(tx.hi), get(tx.lo)});
      jy = ff_add(jy, ff{get(ty.hi), get(ty.lo)});
      en = ff_add(en, ff{get(te.hi), get(te.lo)});
    }
    m = state32_of(rho, jx, jy, en);
  }
  // the other node's state (lane a holds a, lane b holds b)
  auto other = [&](ff x) { return ff{__shfl_xor_sync(0xffffffffu, x.hi, TT), __shfl_xor_sync(0xffffffffu, x.lo, TT)}; };
  const State32 o{other(m.rho), other(m.ux), other(m.uy), other(m.E),
                  __shfl_xor_sync(0xffffffffu, (int)m.ok, TT) != 0};
  const State32 a = layer == 0 ? m : o, b = layer == 0 ? o : m;
  // Eq. (39), applied twice: g0 = 2a - b, g1 = 2 g0 - a = 3a - 2b.
  auto extrapolated = [&](ff xa, ff xb) {
    const ff g0 = ff_add(ff_scale(xa, 2.f), ff_neg(xb));
    return layer == 0 ? g0 : ff_add(ff_scale(g0, 2.f), ff_neg(xa));
  };
  if (kind != PCLB_BC_DIRICHLET) {
    g.rho = extrapolated(a.rho, b.rho);
    g.E = extrapolated(a.E, b.E);
    if (kind == PCLB_BC_EXTRAP) {
      g.ux = extrapolated(a.ux, b.ux);
      g.uy = extrapolated(a.uy, b.uy);
    }
    e = factors(g);
  }
  // equilibrium of the wall node, for the departure it hands to its ghosts
  Eq32 ea{};
  if (neq) ea = factors(a);
  const int col = cw - step * (1 + layer);
  if (t0 + lane % TT >= p.n_theta) return;
  if (!(a.ok && b.ok && g.rho.hi > 0.f && g.E.hi > 0.f)) atomicOr(p.status, PCLB_FLAG_NONPHYS);
  if (col < 0 || col >= kWinR) return;
  const float* fa = sm + row * kWinR + cw;
  float* gp = sm + row * kWinR + col;
  if (group == 0) gp[0] = feq32(e, d, 0, 0, 1.f) + (neq ? fa[0] - feq32(ea, d, 0, 0, 1.f) : 0.f);
#pragma unroll 1
  for (int k = kShare ? group + 1 : 1; k <= (kShare ? group + 1 : 4); ++k)
#pragma unroll
    for (int i = 0; i < kHalf; ++i) {
      const int q = 1 + (k - 1) * kNDirs + i, kw = kShare ? 1 : k;
      float v1 = feq32_weighted(e, d, e.w[kw], k, i, 1.f), v2 = feq32_weighted(e, d, e.w[kw], k, i, -1.f);
      if (neq) {
        v1 += fa[q * PL] - feq32_weighted(ea, d, ea.w[kw], k, i, 1.f);
        v2 += fa[(q + kHalf) * PL] - feq32_weighted(ea, d, ea.w[kw], k, i, -1.f);
      }
      gp[q * PL] = v1;
      gp[(q + kHalf) * PL] = v2;
    }
}

__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Limiter part of the MWB increment of both nodes, |D| (D - Dp) / (|D| + |Dp|)
// (0 when D = Dp = 0), Eq. (28) in upwind form.
__device__ __forceinline__ f2 limiter2(f2 D, f2 Dp) {
  const f2 aD = abs2(D);
  const f2 den = add2(aD, abs2(Dp));
  const f2 rr = mk2(rcp_approx(fmaxf(den.x, 1e-30f)), rcp_approx(fmaxf(den.y, 1e-30f)));
  return mul2(mul2(aD, rr), sub2(D, Dp));
}

}  // namespace

template <int SCH, int TT>
__global__ void __launch_bounds__(F32Size<TT>::threads, kCtasPerSm32)
    step_kernel_f32(const __grid_constant__ CUtensorMap tmap_in, float* __restrict__ f_out,
                    const __grid_constant__ StepParams p, const __grid_constant__ DvmConst<float> d, int ty0) {
  using SZ = F32Size<TT>;
  constexpr int PL = SZ::plane, SPLIT = SZ::split;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float* sm = reinterpret_cast<float*>(smem_raw);
  float4* tab = reinterpret_cast<float4*>(smem_raw + SZ::planes_bytes);
  f2* xch = reinterpret_cast<f2*>(smem_raw + SZ::planes_bytes + SZ::tab_bytes);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + SZ::planes_bytes + SZ::tab_bytes + SZ::exchange_bytes);

  const int r0 = blockIdx.x * kTileR;
  const int t0 = (blockIdx.y + ty0) * TT;   // ty0: first tile row of the launch
  const int tid = threadIdx.x;

  // Thread 0 initialises the barriers and issues the copies at once; the
  // block barrier below (after the table fill) makes the initialised
  // barriers visible to the other threads before their first wait.
  if (tid == 0) {
    tma_prefetch_desc(&tmap_in);
    for (int g = 0; g < kGroups; ++g) mbar_init(&bar[g], 1);
    mbar_fence_init();
  }
  const int warp = tid >> 5, lane = tid & 31;
  const int cw_out = p.n_r - 1 - r0 + kLeft;
  const bool inner = r0 == 0, outer = cw_out <= kLeft + kTileR;   // tiles at a wall
  bool ok = true;
  auto ready = [&](int g) {
    if (ok) ok = p.wait_ns != 0 && mbar_wait_bounded(&bar[g], 0, p.wait_ns);   // 0: give up at once
  };
  if constexpr (SPLIT > 1) {
    if (warp >= kStepThreads32 / 32) {   // the ghost columns' warps: one per wall
      const int side = warp - kStepThreads32 / 32;
      const bool active = side == 0 ? inner : outer;
      bool joined = false;
      auto all = [&]() {   // after what does not depend on f
        pdl_wait();
        block_barrier();   // barriers initialised
        joined = true;
        for (int g = 0; g < kGroups; ++g) ready(g);
        return ok = __all_sync(0xffffffffu, ok);
      };
      if (active) ghost_columns_f32<TT>(sm, lane, side, side == 0 ? kLeft : cw_out, t0, p, d, all);
      if (!joined) block_barrier();
      if (inner || outer) __syncthreads_or(!ok);
      return;
    }
  }
  // Courant entries of the tile rows: table layout [pair][row] (read before
  // the wait: no step writes them)
  const int te_pair = tid / TT, te_row = tid % TT;
  float4 te;
  if (tid < kPairs * TT) te = p.courant[(size_t)(min(t0 + te_row, p.n_theta - 1) + kGhostRows) * kPairs + te_pair];
  pdl_wait();      // the step before this one has written f and read f_out
  pdl_launch();    // the next one may start its set-up
  if (tid == 0) {
#pragma unroll 1
    for (int g = 0; g < kGroups; ++g) {
      const int q0 = group_first(g), n = group_planes(g);
      mbar_arrive_expect_tx(&bar[g], (uint32_t)(n * PL * 4));
#pragma unroll 1
      for (int q = q0; q < q0 + n; ++q) tma_load_3d(sm + q * PL, &tmap_in, r0 - kLeft, t0, q, &bar[g]);
    }
  }
  if (tid < kPairs * TT) tab[te_pair * TT + te_row] = te;
  block_barrier();   // table visible (while the copies are still landing)

  // ---- per-thread nodes: row rl, radial cells j2 and j2 + 1 -----------------
  const int rl = (2 * warp + (lane >> 4)) % TT;    // tile row
  const int split = SPLIT == 1 ? 0 : warp / (TT / 2);   // SPLIT > 1: shell split + 1; the two warps after those: ghost columns
  const int j2 = 2 * (lane & 15);                  // even radial offset 0..30
  const int row = rl + 2;                          // window row
  const int col = kLeft + j2;                      // window column of the first node
  const int t = t0 + rl;
  const int r = r0 + j2;
  const bool row_ok = t < p.n_theta;
  const bool v0 = row_ok && r < p.n_r, v1 = row_ok && r + 1 < p.n_r;
  const float* win = sm + row * kWinR + col;

  Eq2 eq;
  const int ip = (warp & (TT / 2 - 1)) * 32 + lane;   // node pair of the tile (SPLIT > 1)
  {
    State2 s;
    if constexpr (SPLIT == 1) {
      s = state2<PL>(win, d, ready);
    } else {
      s = state2_split<PL>(win, d, split, xch, SZ::pairs, ip, ready, [&]() { ok = !barrier_or(1, kStepThreads32, !ok); });
    }
    const bool ok0 = s.rho.hi.x > 0.f && s.E.hi.x > 0.f && isfinite(s.E.hi.x) && isfinite(s.ux.hi.x) &&
                     isfinite(s.uy.hi.x);
    const bool ok1 = s.rho.hi.y > 0.f && s.E.hi.y > 0.f && isfinite(s.E.hi.y) && isfinite(s.ux.hi.y) &&
                     isfinite(s.uy.hi.y);
    if (ok && ((v0 && !ok0) || (v1 && !ok1))) atomicOr(p.status, PCLB_FLAG_NONPHYS);
    // keep lanes without a valid node finite (their results are never stored)
    if (!v0) { s.rho.hi.x = 1.f; s.rho.lo.x = 0.f; s.E.hi.x = 1.f; s.E.lo.x = 0.f;
               s.ux.hi.x = 0.f; s.ux.lo.x = 0.f; s.uy.hi.x = 0.f; s.uy.lo.x = 0.f; }
    if (!v1) { s.rho.hi.y = 1.f; s.rho.lo.y = 0.f; s.E.hi.y = 1.f; s.E.lo.y = 0.f;
               s.ux.hi.y = 0.f; s.ux.lo.y = 0.f; s.uy.hi.y = 0.f; s.uy.lo.y = 0.f; }
    if constexpr (SPLIT == 1) {
      eq = eq2(s, d);
    } else {   // this thread's shell only; the first thread of a pair also needs the sum of all four
      const ff2 F = shell_weight2(s.E, d, split + 1);
      xch[(29 + 2 * split) * SZ::pairs + ip] = F.hi;
      xch[(30 + 2 * split) * SZ::pairs + ip] = F.lo;
      eq.w[1] = ff2_round(ff2_mul(s.rho, F));
      eq2_polynomial(s, eq);
      barrier_or(1, kStepThreads32, false);
      if (split == 0) {
        ff2 sum = ff2_of(bc2(0.f));
#pragma unroll
        for (int k = 0; k < 4; ++k)
          sum = ff2_add(sum, ff2{xch[(29 + 2 * k) * SZ::pairs + ip], xch[(30 + 2 * k) * SZ::pairs + ip]});
        eq.w[0] = rest_weight2(s.rho, sum, d);
      }
    }
  }

  // ---- radial ghost columns (tiles at a wall only) ----------------------------
  if (inner || outer) {
    if constexpr (SPLIT == 1) {
      const bool here = __all_sync(0xffffffffu, ok);
      auto landed = [&]() { return here; };
      if (inner && warp == 0) ghost_columns_f32<TT>(sm, lane, 0, kLeft, t0, p, d, landed);
      if (outer && warp == 1) ghost_columns_f32<TT>(sm, lane, 1, cw_out, t0, p, d, landed);
    }
    if (__syncthreads_or(!ok)) {   // ghost columns visible; a copy that timed out stops the tile
      if (tid == 0) {
        atomicOr(p.status, PCLB_FLAG_TIMEOUT);
        for (int g = 0; g < kGroups; ++g) mbar_wait_bounded(&bar[g], 0, kDefaultWaitNs);
      }
      return;
    }
  } else if (!ok) {
    // a copy did not land in time: report it, give the copies a bounded time
    // to finish, and leave (no barrier follows in this tile)
    atomicOr(p.status, PCLB_FLAG_TIMEOUT);
    for (int g = 0; g < kGroups; ++g) mbar_wait_bounded(&bar[g], 0, kDefaultWaitNs);
    return;
  }

  // ---- update ----------------------------------------------------------------
  const f2 invr = mk2(v0 ? p.inv_r_f[r] : 1.f, v1 ? p.inv_r_f[r + 1] : 1.f);
  const f2 decay = bc2((float)p.decay);
  const size_t plane_out = (size_t)p.rows * p.pitch;
  float* out_row = f_out + (size_t)(t + kGhostRows) * p.pitch + r;
  // tiles away from the radial walls and the seam take the plain store
  const bool plain_tile = r0 + kTileR <= p.n_r && t0 >= 2 && t0 + TT <= p.n_theta - 2;
  auto store = [&](int q, f2 o) {
    if (plain_tile) {
      __stcs(reinterpret_cast<float2*>(out_row + (size_t)q * plane_out), o);   // not read again before the next step
      return;
    }
    // seam and ragged tiles: the seam rows' ghost copies, formed here so
    // that plain tiles keep no registers for them
    const bool lo_ghost = row_ok && t >= p.n_theta - 2;
    const bool hi_ghost = row_ok && t < 2;
    float* out_lo = f_out + (size_t)max(t - (p.n_theta - 2), 0) * p.pitch + r;
    float* out_hi = f_out + (size_t)(p.n_theta + kGhostRows + t) * p.pitch + r;
    if (v1) {
      *reinterpret_cast<float2*>(out_row + (size_t)q * plane_out) = o;
      if (lo_ghost) *reinterpret_cast<float2*>(out_lo + (size_t)d.recv_lo[q] * plane_out) = o;
      if (hi_ghost) *reinterpret_cast<float2*>(out_hi + (size_t)d.recv_hi[q] * plane_out) = o;
    } else if (v0) {
      out_row[(size_t)q * plane_out] = o.x;
      if (lo_ghost) out_lo[(size_t)d.recv_lo[q] * plane_out] = o.x;
      if (hi_ghost) out_hi[(size_t)d.recv_hi[q] * plane_out] = o.x;
    }
  };

  if (split == 0) {  // rest velocity: no convection
    const f2 f0 = ld2(win);
    const f2 e0 = mul2(eq.w[0], eq.a0);
    store(0, fma2(sub2(f0, e0), decay, e0));
  }

  // One velocity of a pair.  sr = +1 if its upwind neighbour in r is at
  // larger r, st the same for theta (rows); fe is its equilibrium.
  // nar, nkr, nat, nkt: the negated a = |C| and K = |C|(1 - |C|) in r and
  // theta.  Increments in upwind form (D, Dp the upwind differences):
  // MWB a D + K h(D, Dp); WB a D + K (D - Dp)/2; LW a D + K (Dd - D)/2 with
  // Dd the downwind difference; second-order upwind a D + a (D - Dp)/2.
  auto update = [&](int q, int sr, int st, f2 nar, f2 nkr, f2 nat, f2 nkt, f2 fe) {
    const float* w = win + q * PL;
    const f2 C = ld2(w);
    const f2 S = ld2(w + 2 * sr);                 // (j-2, j-1) or (j+2, j+3)
    const f2 T1 = ld2(w + st * kWinR);
    const f2 T2 = ld2(w + 2 * st * kWinR);
    const f2 u1 = sr < 0 ? mk2(S.y, C.x) : mk2(C.y, S.x);   // first upwind neighbours
    const f2 Dr = sub2(C, u1), Dt = sub2(C, T1);
    // the convection increments summed first (small), then added once to
    // the relaxed value (one rounding at the magnitude of f for them)
    f2 dc = mul2(nar, Dr);
    dc = fma2(nat, Dt, dc);
    if constexpr (SCH == PCLB_SCHEME_MWB) {
      dc = fma2(nkr, limiter2(Dr, sub2(u1, S)), dc);
      dc = fma2(nkt, limiter2(Dt, sub2(T1, T2)), dc);
    } else if constexpr (SCH == PCLB_SCHEME_WB) {
      dc = fma2(mul2(bc2(0.5f), nkr), sub2(Dr, sub2(u1, S)), dc);
      dc = fma2(mul2(bc2(0.5f), nkt), sub2(Dt, sub2(T1, T2)), dc);
    } else if constexpr (SCH == PCLB_SCHEME_UPWIND2) {
      dc = fma2(mul2(bc2(0.5f), nar), sub2(Dr, sub2(u1, S)), dc);
      dc = fma2(mul2(bc2(0.5f), nat), sub2(Dt, sub2(T1, T2)), dc);
    } else {
      const f2 X = ld2(w - 2 * sr);               // the pair on the downwind side
      const f2 d1 = sr < 0 ? mk2(C.y, X.x) : mk2(X.y, C.x);   // first downwind neighbours
      const f2 Td = ld2(w - st * kWinR);
      dc = fma2(mul2(bc2(0.5f), nkr), sub2(sub2(d1, C), Dr), dc);
      dc = fma2(mul2(bc2(0.5f), nkt), sub2(sub2(Td, C), Dt), dc);
    }
    store(q, add2(fma2(sub2(C, fe), decay, fe), dc));
  };

  // Shells run as a loop (keeps the hot body small for the instruction
  // cache); the four direction pairs of a shell are unrolled.
#pragma unroll 1
  for (int k = SPLIT == 1 ? 1 : split + 1; k <= (SPLIT == 1 ? 4 : split + 1); ++k) {
    const f2 sh = bc2(d.speed[k]), sl = bc2(d.speed_lo[k]);
    const f2 wk = SPLIT > 1 || k == 1 ? eq.w[1] : (k == 2 ? eq.w[2] : (k == 3 ? eq.w[3] : eq.w[4]));
    const int qb = 1 + (k - 1) * kNDirs;
#pragma unroll
    for (int i = 0; i < kHalf; ++i) {
      const int q = qb + i;
      const float4 tb = tab[((k - 1) * kHalf + i) * TT + rl];
      const int fl = __float_as_int(tb.w);
      const int sr = (fl & 1) ? 1 : -1;            // v_r < 0: upwind at larger r
      const int st = (fl & 2) ? 1 : -1;            // v_theta < 0: upwind at larger theta
      const f2 nar = bc2(-tb.x), nkr = bc2(-tb.y);
      const f2 nat = mul2(bc2(-tb.z), invr);
      const f2 nkt = fma2(nat, nat, nat);            // -(a - a^2) with a = -nat
      f2 fp, fm;   // equilibrium of the pair
      feq_pair2(eq, sh, sl, i, wk, fp, fm);
      update(q, sr, st, nar, nkr, nat, nkt, fp);
      update(q + kHalf, -sr, -st, nar, nkr, nat, nkt, fm);
    }
  }
}

template <int SCH, int TT>
static cudaError_t launch_tile_rows_f32(const CUtensorMap* tmap_in, float* f_out, const StepParams& p,
                                        const DvmConst<float>& d, cudaStream_t stream, int ty_begin, int ty_end) {
  static std::atomic<unsigned long long> configured{0};   // per instantiation and device
  {
    const cudaError_t e = set_smem_once(step_kernel_f32<SCH, TT>, F32Size<TT>::smem, configured);
    if (e != cudaSuccess) return e;
  }
  const dim3 grid((p.n_r + kTileR - 1) / kTileR, ty_end - ty_begin);
  return launch_overlapped(step_kernel_f32<SCH, TT>, grid, F32Size<TT>::threads, F32Size<TT>::smem, stream, *tmap_in,
                           f_out, p, d, ty_begin);
}

template <int SCH>
static cudaError_t launch_scheme_f32(const CUtensorMap* tmap_in, float* f_out, const StepParams& p,
                                     const DvmConst<float>& d, cudaStream_t stream, int ty_begin, int ty_end) {
  if (p.tile_rows == kTileT32)
    return launch_tile_rows_f32<SCH, kTileT32>(tmap_in, f_out, p, d, stream, ty_begin, ty_end);
  constexpr int per = kTileT32 / kTileTSmall;
  const int last = (p.n_theta + kTileTSmall - 1) / kTileTSmall;
  return launch_tile_rows_f32<SCH, kTileTSmall>(tmap_in, f_out, p, d, stream, ty_begin * per,
                                                ty_end * per < last ? ty_end * per : last);
}

// Tile rows [ty_begin, ty_end) of the grid, kTileT32 nodes each (ty_end < 0:
// to the last tile row); an empty range launches nothing.  tmap_in: boxes of
// p.tile_rows + 4 window rows.
cudaError_t launch_step_f32(const CUtensorMap* tmap_in, float* f_out, const StepParams& p,
                            const DvmConst<float>& d, cudaStream_t stream, int ty_begin, int ty_end) {
  if (ty_end < 0) ty_end = (p.n_theta + kTileT32 - 1) / kTileT32;
  if (ty_begin < 0 || ty_end <= ty_begin) return cudaSuccess;
  switch (p.scheme) {
    case PCLB_SCHEME_WB: return launch_scheme_f32<PCLB_SCHEME_WB>(tmap_in, f_out, p, d, stream, ty_begin, ty_end);
    case PCLB_SCHEME_LW: return launch_scheme_f32<PCLB_SCHEME_LW>(tmap_in, f_out, p, d, stream, ty_begin, ty_end);
    case PCLB_SCHEME_UPWIND2:
      return launch_scheme_f32<PCLB_SCHEME_UPWIND2>(tmap_in, f_out, p, d, stream, ty_begin, ty_end);
    default: return launch_scheme_f32<PCLB_SCHEME_MWB>(tmap_in, f_out, p, d, stream, ty_begin, ty_end);
  }
}

}  // namespace pclb
