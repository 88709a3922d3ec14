// The FP64 step (Eq. 38) on small grids, where the time of one
// tile is the time of the step: tiles of 32 (r) x TT (theta) nodes, TT = 2 or 4.
//
// As in step_kernel_f64.cu the sums and the convection increments are formed in
// 64-bit fixed point (fixed64.cuh), here on the exponent of the five values of
// each stencil (or of a shell's values at a node), so that no pass over the
// window comes first; FP64 keeps the states, the equilibrium and the final sums.
// What is left is a chain of latencies, so the CTA's warps work side by side:
//   * 16 pair warps, 16 / TT per row, own a shell (TT = 4) or half a shell (TT =
//     2) each: they form the shells' sums, then d f - M_r - M_theta of their
//     labels, and add (1 - d) f^eq when the state is there;
//   * TT state warps, one per row, form the node state and the equilibrium
//     factors from the shells' sums, and the rest velocity;
//   * two ghost warps, one per wall, form the ghost layers' states and factors
//     (Sec. II C 1) from the same sums; the pair warps turn them into values.
// 100 x 20 with non-equilibrium walls: 16.8 us per step (206 us with all of it in
// FP64 and the ghost columns row by row; 15.4 us with conversions and products
// that dropped what is below a unit); 64 x 128: 16.4 us.
#include <cuda.h>
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "fixed64.cuh"
#include "pclb_internal.h"

namespace pclb {

namespace {

constexpr int kPairsSm = 4 * kHalfDirs;
constexpr int kPairWarps = 16;

template <int SCH>
struct SmTab {
  FxCoef<SCH> r;    // radial
  uint64_t at;      // |C_theta| at the tile's first column, units of 2^-63
  int64_t fl;       // bit 0: v_r < 0, bit 1: v_theta < 0 for the first label of the pair
};

template <int SCH, int TT>
struct SmSize {
  static constexpr int split = kPairWarps / TT;             // warps per row: 4 or 8
  static constexpr int dirs = split == 4 ? 4 : 2;           // direction pairs of its shell per warp
  static constexpr int threads = 32 * (kPairWarps + TT + 2);
  static constexpr int plane = kWinR * (TT + 4);
  static constexpr int planes_bytes = kQ * plane * 8;
  static constexpr int tab_bytes = kPairsSm * TT * (int)sizeof(SmTab<SCH>);
  // per node the shells' sums (S, X, Y), the equilibrium factors w_1 .. w_4, a0, a1, u / E
  static constexpr int node_bytes = TT * 32 * (12 + 8) * 8;
  // per wall, slot (ghost layer 0, 1, wall node) and row the factors w_0 .. w_4, a0, a1, a1h, u / E
  static constexpr int ghost_bytes = 2 * 3 * TT * 10 * 8;
  static constexpr int kept_bytes = 2 * dirs * 32 * kPairWarps * 8;
  static constexpr int smem = planes_bytes + tab_bytes + node_bytes + ghost_bytes + kept_bytes + 128;
  static_assert((plane * 8) % 128 == 0, "TMA destinations must stay 128-byte aligned");
};

// Named barriers (0 is the block's): warps that only hand something over
// arrive, those that need it wait.
constexpr int kBarSums = 1, kBarFactors = 2, kBarGhosts = 3, kBarState = 4;
__device__ __forceinline__ void bar_arrive(int id, int threads) {
  __syncwarp();
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void bar_wait(int id, int threads) {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}

}  // namespace

template <int SCH, int TT>
__global__ void __launch_bounds__(SmSize<SCH, TT>::threads, 1)
    step_small_f64(const __grid_constant__ CUtensorMap tmap_in, double* __restrict__ f_out,
                   const __grid_constant__ StepParams p, const __grid_constant__ DvmConst<double> d, int ty0) {
  using SZ = SmSize<SCH, TT>;
  constexpr int PLANE = SZ::plane, SPLIT = SZ::split, DIRS = SZ::dirs;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  double* sm = reinterpret_cast<double*>(smem_raw);
  SmTab<SCH>* tab = reinterpret_cast<SmTab<SCH>*>(smem_raw + SZ::planes_bytes);            // [pair][row]
  double* sums = reinterpret_cast<double*>(smem_raw + SZ::planes_bytes + SZ::tab_bytes);   // [row][lane][12]
  double* fac = sums + TT * 32 * 12;                                                         // [row][lane][8]
  double* gfac = fac + TT * 32 * 8;                                                          // [side][slot][row][10]
  double* kept = gfac + 2 * 3 * TT * 10;                                                     // [label][pair thread]
  uint64_t* bar = reinterpret_cast<uint64_t*>(kept + 2 * SZ::dirs * 32 * kPairWarps);

  const int r0 = blockIdx.x * kTileR;
  const int t0 = (blockIdx.y + ty0) * TT;   // ty0: first tile row of the launch
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int cw_out = p.n_r - 1 - r0 + kLeft;
  const bool inner = r0 == 0, outer = cw_out <= kLeft + kTileR;   // tiles at a wall
  const int n_ghost = (inner ? 1 : 0) + (outer ? 1 : 0);           // ghost warps at work
  // threads at each named barrier
  constexpr int kValWarps = TT * 64 / 32;                          // pair warps that store ghost values: an item per thread
  const int n_sums = 32 * (4 * TT + TT + n_ghost), n_factors = 32 * (kValWarps + n_ghost);
  constexpr int n_values = 32 * kPairWarps, n_state = 32 * (kPairWarps + TT);

  if (tid == 0) {
    tma_prefetch_desc(&tmap_in);
    mbar_init(bar, 1);
    mbar_fence_init();
  }
  const double inv_r0 = p.inv_r[r0];
  if (tid < kPairsSm * TT) {   // Courant entries of the tile rows
    const int pair = tid / TT, rl = tid % TT;
    const double* e = p.courant64 + ((size_t)(min(t0 + rl, p.n_theta - 1) + kGhostRows) * kPairsSm + pair) * 4;
    SmTab<SCH> t;
    t.r = fx_coef<SCH>(fx_fraction(e[0]));
    t.at = fx_fraction(e[2] * inv_r0);
    t.fl = (int64_t)e[3];
    tab[pair * TT + rl] = t;
  }

  // ---- ghost warps: lane (slot or node, row); what does not depend on f first
  const int side = warp - kPairWarps - TT;          // ghost warps: 0 inner, 1 outer
  const bool ghosts = side >= 0 && (side == 0 ? inner : outer);
  const int grow = lane % TT, slot = lane / TT;     // slots: ghost layers 0, 1, wall node
  const int kind = p.bc_kind[side == 1] & ~PCLB_BC_NEQ;
  double g[4] = {1.0, 0.0, 0.0, 1.0};               // rho, u_x, u_y, E of the slot
  if (ghosts && slot < 2 && kind != PCLB_BC_EXTRAP) {
    const int t = min(t0 + grow, p.n_theta - 1);
    const double c = p.cos_t[t], s = p.sin_t[t];
    const double* v = p.bc_vals + (size_t)((side * 2 + slot) * 4) * p.n_theta + t;
    const double ur = v[1 * p.n_theta], ut = v[2 * p.n_theta];
    g[1] = ur * c - ut * s;
    g[2] = ur * s + ut * c;
    if (kind == PCLB_BC_DIRICHLET) {
      g[0] = v[0];
      g[3] = v[3 * p.n_theta];
    }
  }

  pdl_wait();      // the step before this one has written f and read f_out
  pdl_launch();    // the next one may start its set-up
  if (tid == 0) {  // window rows [t0-2, t0+TT+2) are stored rows [t0, t0+TT+4)
    mbar_arrive_expect_tx(bar, (uint32_t)SZ::planes_bytes);
#pragma unroll 1
    for (int q = 0; q < kQ; ++q) tma_load_3d(sm + q * PLANE, &tmap_in, r0 - kLeft, t0, q, bar);
  }
  __syncthreads();
  // The whole block gives the tile up if any thread's wait ran out (barriers
  // follow, so the decision must be uniform); thread 0 then gives the copies
  // one more bounded chance to land before the block exits.
  if (__syncthreads_or(p.wait_ns == 0 || !mbar_wait_bounded(bar, 0, p.wait_ns))) {   // 0: give up at once
    if (tid == 0) {
      atomicOr(p.status, PCLB_FLAG_TIMEOUT);
      mbar_wait_bounded(bar, 0, kDefaultWaitNs);
    }
    return;
  }

  const double decay = p.decay, omd = 1.0 - decay;
  const int rl = warp < kPairWarps ? warp % TT : warp - kPairWarps;   // tile row of a pair or state warp
  const int r = r0 + lane, t = t0 + rl;
  // threads without a node repeat the last one's (what TMA fills in for them is out of fixed point's range)
  const int node = (min(rl, p.n_theta - 1 - t0) + 2) * kWinR + kLeft + min(lane, p.n_r - 1 - r0);
  const bool valid = r < p.n_r && t < p.n_theta;
  const size_t plane_out = (size_t)p.rows * p.pitch;
  auto store = [&](int q, double v) {
    f_out[(size_t)q * plane_out + (size_t)(t + kGhostRows) * p.pitch + r] = v;
    if (t >= p.n_theta - 2)   // also the low ghost rows (theta <= 0) of the receiving label
      f_out[(size_t)d.recv_lo[q] * plane_out + (size_t)(t - (p.n_theta - 2)) * p.pitch + r] = v;
    if (t < 2)                // and the high ghost rows (theta > 2 pi n_f / n_dirs)
      f_out[(size_t)d.recv_hi[q] * plane_out + (size_t)(p.n_theta + kGhostRows + t) * p.pitch + r] = v;
  };

  if (warp >= kPairWarps + TT) {   // ---- ghost warps ----------------------------
    if (!ghosts) return;
    bar_wait(kBarSums, n_sums);
    // the state of node slot (0 the wall node a, 1 the next node b); a wall
    // node outside the tile's own columns has no sums yet
    NodeState<double> m;
    m.rho = m.E = 1.0; m.ux = m.uy = 0.0; m.ok = true;
    const int step = side == 0 ? 1 : -1, ca = side == 0 ? kLeft : cw_out;
    const bool row_ok = t0 + grow < p.n_theta;
    if (slot < 2 && row_ok) {
      const int col = ca + slot * step;
      const double* f = sm + (grow + 2) * kWinR + col;
      double own[12];
      const double* s = sums + (grow * 32 + col - kLeft) * 12;
      if (col < kLeft || col >= kLeft + kTileR) {
#pragma unroll 1
        for (int k = 1; k <= 4; ++k) shell_sums64(f + (1 + (k - 1) * kNDirs) * PLANE, PLANE, d, own + 3 * (k - 1));
        s = own;
      }
      m = state_of_sums(f[0], s, d);
    }
    const double v[4] = {m.rho, m.ux, m.uy, m.E};
    double a[4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      a[j] = __shfl_sync(0xffffffffu, v[j], grow);
      const double b = __shfl_sync(0xffffffffu, v[j], TT + grow);
      // Eq. (39), applied twice: g0 = 2a - b, g1 = 2 g0 - a
      const double g0 = 2.0 * a[j] - b;
      const bool extrapolate = (j == 0 || j == 3) ? kind != PCLB_BC_DIRICHLET : kind == PCLB_BC_EXTRAP;
      if (extrapolate) g[j] = slot == 0 ? g0 : 2.0 * g0 - a[j];
      if (slot == 2) g[j] = a[j];
    }
    if (slot < 2 && row_ok && !(m.ok && positive64(g[0]) && positive64(g[3]))) atomicOr(p.status, PCLB_FLAG_NONPHYS);
    const EqParams<double> e = eq_params<double>(g[0], g[1], g[2], g[3], d);
    if (slot < 3) {
      double* o = gfac + ((side * 3 + slot) * TT + grow) * 10;
#pragma unroll
      for (int k = 0; k < 5; ++k) o[k] = e.w[k];
      o[5] = e.a0; o[6] = e.a1; o[7] = e.a1h; o[8] = e.uxE; o[9] = e.uyE;
    }
    bar_arrive(kBarFactors, n_factors);
    return;
  }
  double* nfac = fac + (rl * 32 + lane) * 8;
  if (warp >= kPairWarps) {        // ---- state warps ----------------------------
    const double f0 = sm[node];
    bar_wait(kBarSums, n_sums);
    const NodeState<double> m = state_of_sums(f0, sums + (rl * 32 + lane) * 12, d);
    if (valid && !m.ok) atomicOr(p.status, PCLB_FLAG_NONPHYS);
    const EqParams<double> e = eq_params<double>(omd * m.rho, m.ux, m.uy, m.E, d);   // w_k = (1 - d) rho F_k
#pragma unroll
    for (int k = 1; k <= 4; ++k) nfac[k - 1] = e.w[k];
    nfac[4] = e.a0; nfac[5] = e.a1; nfac[6] = e.uxE; nfac[7] = e.uyE;
    bar_arrive(kBarState, n_state);
    if (valid) store(0, fma(decay, f0, e.w[0] * e.a0));   // rest velocity: no convection
    return;
  }

  // ---- pair warps ------------------------------------------------------------
  const int part = warp / TT, k = part / (SPLIT / 4) + 1, i_first = part % (SPLIT / 4) * DIRS;
  if (i_first == 0) {
    double s[3];
    shell_sums64(sm + (1 + (k - 1) * kNDirs) * PLANE + node, PLANE, d, s);
    double* o = sums + (rl * 32 + lane) * 12 + 3 * (k - 1);
    o[0] = s[0]; o[1] = s[1]; o[2] = s[2];
    bar_arrive(kBarSums, n_sums);
  }
  if (n_ghost > 0) {
    // ghost values: a wall, layer, row and pair per thread
    if (warp < kValWarps) {
      bar_wait(kBarFactors, n_factors);
      const int row = tid % TT, lay = tid / TT & 1, sd = tid / (2 * TT) & 1, pair = tid / (4 * TT);
      const int ca = sd == 0 ? kLeft : cw_out, col = ca - (sd == 0 ? 1 : -1) * (1 + lay);
      if ((sd == 0 ? inner : outer) && t0 + row < p.n_theta && col >= 0 && col < kWinR) {
        const int kk = 1 + pair / kHalfDirs, q1 = 1 + (kk - 1) * kNDirs + pair % kHalfDirs, q2 = q1 + kHalfDirs;
        double* w = sm + (row + 2) * kWinR;
        auto feq = [&](int sl, double& fp, double& fm) {   // P(+-x) = ev +- od (Eq. 10)
          const double* x = gfac + ((sd * 3 + sl) * TT + row) * 10;
          const double y = d.vx[q1] * x[8] + d.vy[q1] * x[9], y2 = y * y;
          const double ev = x[5] + y2 * (x[7] + y2 * (1.0 / 24.0)), od = y * (x[6] + y2 * (1.0 / 6.0));
          fp = x[kk] * (ev + od);
          fm = x[kk] * (ev - od);
        };
        double fp, fm;
        feq(lay, fp, fm);
        if (p.bc_kind[sd] & PCLB_BC_NEQ) {   // the wall node's departure
          double ap, am;
          feq(2, ap, am);
          fp += w[(size_t)q1 * PLANE + ca] - ap;
          fm += w[(size_t)q2 * PLANE + ca] - am;
        }
        w[(size_t)q1 * PLANE + col] = fp;
        w[(size_t)q2 * PLANE + col] = fm;
      }
    }
    bar_wait(kBarGhosts, n_values);
  }
  // d f - M_r - M_theta of this thread's labels, kept in shared memory so that the loop
  // stays rolled (unrolled, the compared schemes took 13% more on 64 x 64, now 16.3 us a step)
  double* mine = kept + tid;
  const uint64_t dfx = fx_fraction(fabs(decay));
  const int64_t dsign = decay < 0.0 ? -1 : 0;
  const double inv_r = p.inv_r[min(r, p.n_r - 1)];
  const uint64_t ratio = fx_fraction(inv_r * recip_newton(inv_r0));   // 1/r relative to the tile's first column
  const double* c64 = p.courant64 + ((size_t)(min(t, p.n_theta - 1) + kGhostRows) * kPairsSm + (k - 1) * kHalfDirs) * 4;
#pragma unroll 1
  for (int j = 0; j < DIRS; ++j) {
    const int i = i_first + j, q1 = 1 + (k - 1) * kNDirs + i;
    const SmTab<SCH>& te = tab[((k - 1) * kHalfDirs + i) * TT + rl];
    const FxCoef<SCH> cr = te.r, ct = fx_coef<SCH>(fx_mul_frac(te.at, ratio));
    const int fl = (int)te.fl;
#pragma unroll
    for (int L = 0; L < 2; ++L) {
      constexpr int far = SCH == PCLB_SCHEME_LW ? -1 : 2;
      const int s_r = ((fl & 1) != 0) != (L != 0) ? 1 : -1;               // v_r < 0: upwind at larger r
      const int s_t = ((fl & 2) != 0) != (L != 0) ? kWinR : -kWinR;       // v_theta < 0: upwind at larger theta
      const double* x = sm + (q1 + L * kHalfDirs) * PLANE + node;
      mine[(2 * j + L) * 32 * kPairWarps] = fx_carried<SCH>(x[0], x[s_r], x[far * s_r], x[s_t], x[far * s_t], cr, ct, dfx,
                                                            dsign, decay, c64 + 4 * i, inv_r);
    }
  }
  bar_wait(kBarState, n_state);
  if (!valid) return;
  // (1 - d) f^eq of the pairs: ev +- od, ev = A + y^2 (B + y^2 C), od = y (O1 + y^2 O3)
  const double w = nfac[k - 1], a0 = nfac[4], a1 = nfac[5], uxE = nfac[6], uyE = nfac[7], wa = w * a1;
  const double A = w * a0, B = wa * d.half_v2[k], C = w * d.v4_24[k], O1 = wa * d.speed[k], O3 = w * d.v3_6[k];
#pragma unroll
  for (int j = 0; j < DIRS; ++j) {
    const int i = i_first + j, q1 = 1 + (k - 1) * kNDirs + i;
    double y = i == 0 ? uxE : uyE;                                   // directions (1,0), (s,s), (0,1), (-s,s)
    if (i & 1) y = d.cx[2] * (i == 1 ? uyE + uxE : uyE - uxE);
    const double y2 = y * y, ev = fma(y2, fma(y2, C, B), A), z = fma(y2, O3, O1);
    store(q1, fma(y, z, ev + mine[2 * j * 32 * kPairWarps]));
    store(q1 + kHalfDirs, fma(-y, z, ev + mine[(2 * j + 1) * 32 * kPairWarps]));
  }
}

template <int SCH, int TT>
static cudaError_t launch_small(const CUtensorMap* tmap_in, double* f_out, const StepParams& p, const DvmConst<double>& d,
                                cudaStream_t stream, int ty_begin, int ty_end) {
  static std::atomic<unsigned long long> configured{0};   // per instantiation and device
  constexpr int smem = SmSize<SCH, TT>::smem, threads = SmSize<SCH, TT>::threads;
  const cudaError_t e = set_smem_once(step_small_f64<SCH, TT>, smem, configured);
  if (e != cudaSuccess) return e;
  const dim3 grid((p.n_r + kTileR - 1) / kTileR, ty_end - ty_begin);
  return launch_overlapped(step_small_f64<SCH, TT>, grid, threads, smem, stream, *tmap_in, f_out, p, d, ty_begin);
}

// Tile rows [ty_begin, ty_end) of p.tile_rows nodes each.
template <int SCH>
cudaError_t launch_step_small_f64(const CUtensorMap* tmap_in, double* f_out, const StepParams& p,
                                  const DvmConst<double>& d, cudaStream_t stream, int ty_begin, int ty_end) {
  return p.tile_rows == 2 ? launch_small<SCH, 2>(tmap_in, f_out, p, d, stream, ty_begin, ty_end)
                          : launch_small<SCH, 4>(tmap_in, f_out, p, d, stream, ty_begin, ty_end);
}
#define PCLB_SMALL(SCH)                                                                                             \
  template cudaError_t launch_step_small_f64<SCH>(const CUtensorMap*, double*, const StepParams&,                   \
                                                  const DvmConst<double>&, cudaStream_t, int, int);
PCLB_SMALL(PCLB_SCHEME_MWB)
PCLB_SMALL(PCLB_SCHEME_WB)
PCLB_SMALL(PCLB_SCHEME_LW)
PCLB_SMALL(PCLB_SCHEME_UPWIND2)
#undef PCLB_SMALL

}  // namespace pclb
