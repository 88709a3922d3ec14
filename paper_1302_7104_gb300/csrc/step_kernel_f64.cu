// Fused FP64 time step (Eq. 38 with the MWB increments of Eq. 28 or those of
// the compared schemes): one launch advances every node.
//
// What bounds it: FP64 issue.  A quarter SM starts one warp-wide FP64
// operation per 64-76 cycles (measured), so the ~34 FP64 operations per update
// of a plain evaluation took 34 ms on 4096 x 4096, where HBM needs 1.3 ms.
// Everything that is a sum, a difference or a convection increment is
// therefore done in 64-bit fixed point (fixed64.cuh) on the integer and float
// pipes; FP64 keeps the node state, the equilibrium factors and the final
// sums (~7 operations per update), so results keep double precision.
//
// Tile work (one CTA, 512 threads; kTileR x kTileT nodes, one per thread):
//   1. one thread issues 33 TMA box copies (one per velocity plane) of the
//      window [r0-4, r0+36) x [t0-2, t0+18) into shared memory;
//   2. tiles at a wall form the radial ghost columns in the window, in FP64
//      (ghost_cols.cuh);
//   3. the block finds the largest exponent of each shell's planes and
//      converts the shells' windows in place to fixed point;
//   4. the sums of Eqs. 3-5 per shell as integers, then the node state and the
//      equilibrium factors in FP64;
//   5. per pair of opposite velocities: d f - M_r - M_theta in fixed point,
//      turned to double once, plus (1 - d) f^eq in FP64; rows next to the
//      azimuthal seam also store the output's ghost rows (Eq. 40).
// The window's exponents serve a shell of a node only where the node's values
// are not far below the window's largest: down to 2^5, where the unit, 2^-58 of the
// largest, reaches the rounding of double arithmetic at the node.  The node's
// scale is its largest value of the shell, or (1 - d) rho times the largest
// term of F_k(T) if that is more: f^eq carries the rounding of those terms (F_k
// is their difference and passes through 0 within the usual range of T).  A
// row in which a shell falls short takes that shell from the doubles in global
// memory, on the exponent of each stencil as in step_small_f64.cu; so do all
// shells, and the state, of a row where the unit is coarse for a density, a node is
// not physical, or the window holds NaN, infinity or exponents near the
// ends of the range.  Tiles at a wall, whose ghost columns are in the window
// only, load it again for that.  (The line had been the density alone, 2^8 below
// the window's largest value: a shell of cold gas beside hot gas could be
// wrong by 2^-49 of its scale.  And what left fixed point was done in FP64: a
// 512 x 1024 step with a density jump of 1000 in every tile took 1.73 ms, now
// 1.04 ms; with a jump of 20, 351 us.)
//
// Grids that do not fill the chip with such tiles run step_small_f64.cu.
// Consecutive steps overlap their set-up (programmatic dependent launch).
#include <cuda.h>
#include <cuda_runtime.h>

#include "device_common.cuh"
#include "fixed64.cuh"
#include "ghost_cols.cuh"
#include "pclb_internal.h"

namespace pclb {

namespace {

constexpr int kThreadsFx = 512;
constexpr int kPairsFx = 4 * kNDirs / 2;   // pairs of opposite velocities
constexpr int kThinHi = 1 << (26 - 5);     // high word of a fixed-point value 2^5 below the largest

template <int SCH>
struct FxTab {
  FxCoef<SCH> r;    // radial
  uint64_t at;      // |C_theta| at the tile's first column, units 2^-63
  int fl, pad;      // bit 0: v_r < 0, bit 1: v_theta < 0 for the first label of the pair
};

template <int SCH>
struct FxSize {
  static constexpr int plane = kWinR * (kTileT + 4);
  static constexpr int planes_bytes = kQ * plane * 8;
  static constexpr int tab_bytes = kPairsFx * kTileT * (int)sizeof(FxTab<SCH>);
  static constexpr int scratch = kGhostScratch64<kTileT> * 8;
  static constexpr int smem = planes_bytes + tab_bytes + scratch + 128;
  static_assert((plane * 8) % 128 == 0, "TMA destinations must stay 128-byte aligned");
  static_assert(smem <= 232448, "shared memory of one CTA");
};

// Where a node's results go: label q at (t, r), and the azimuthal ghost rows it
// feeds (Eq. 40).
struct NodeOut {
  double* f;
  int t, r;
  __device__ __forceinline__ void store(int q, double v, const StepParams& p, const DvmConst<double>& d) const {
    const size_t plane = (size_t)p.rows * p.pitch;
    f[(size_t)q * plane + (size_t)(t + kGhostRows) * p.pitch + r] = v;
    if (t >= p.n_theta - 2)   // the low ghost rows (theta <= 0) of the receiving label
      f[(size_t)d.recv_lo[q] * plane + (size_t)(t - (p.n_theta - 2)) * p.pitch + r] = v;
    if (t < 2)                // the high ghost rows (theta > 2 pi n_f / n_dirs)
      f[(size_t)d.recv_hi[q] * plane + (size_t)(p.n_theta + kGhostRows + t) * p.pitch + r] = v;
  }
};

// The pairs of shell k at one node from doubles: w the node, planes `plane` and
// rows `row` apart; eq of (1 - d) rho; tab the tile's entries at the node's row (TT
// apart), ratio and inv_r its 1/r.
template <int SCH, int TT>
__device__ __noinline__ void stencil_shell(const double* w, size_t plane, int row, int k, const EqParams<double>& eq,
                                           const FxTab<SCH>* tab, uint64_t ratio, const StepParams& p,
                                           const DvmConst<double>& d, NodeOut out) {
  const uint64_t dfx = fx_fraction(fabs(p.decay));
  const int64_t dsign = p.decay < 0.0 ? -1 : 0;
  const double* c64 = p.courant64 + (size_t)(out.t + kGhostRows) * kPairsFx * 4;
  const double inv_r = p.inv_r[out.r];
#pragma unroll 1
  for (int pair = (k - 1) * kHalfDirs; pair < k * kHalfDirs; ++pair) {
    const int q1 = 1 + (k - 1) * kNDirs + pair % kHalfDirs;
    const FxTab<SCH>& te = tab[pair * TT];
    const FxCoef<SCH> cr = te.r, ct = fx_coef<SCH>(fx_mul_frac(te.at, ratio));
    const double x = d.vx[q1] * eq.uxE + d.vy[q1] * eq.uyE, x2 = x * x;
    const double ev = eq.a0 + x2 * (eq.a1h + x2 * (1.0 / 24.0)), od = x * (eq.a1 + x2 * (1.0 / 6.0));
#pragma unroll 1
    for (int L = 0; L < 2; ++L) {
      constexpr int far = SCH == PCLB_SCHEME_LW ? -1 : 2;
      const int q = q1 + L * kHalfDirs;
      const int s_r = ((te.fl & 1) != 0) != (L != 0) ? 1 : -1, s_t = ((te.fl & 2) != 0) != (L != 0) ? row : -row;
      const double* f = w + (size_t)q * plane;
      const double g = fx_carried<SCH>(f[0], f[s_r], f[far * s_r], f[s_t], f[far * s_t], cr, ct, dfx, dsign, p.decay,
                                       c64 + 4 * pair, inv_r);
      out.store(q, fma(eq.w[k], L ? ev - od : ev + od, g), p, d);
    }
  }
}

// The node's state and (1 - d) f^eq factors from doubles.
__device__ __noinline__ bool stencil_state(const double* w, size_t plane, double omd, const DvmConst<double>& d,
                                           EqParams<double>& eq) {
  double s[12];
#pragma unroll 1
  for (int k = 1; k <= 4; ++k) shell_sums64(w + (1 + (k - 1) * kNDirs) * plane, plane, d, s + 3 * (k - 1));
  const NodeState<double> m = state_of_sums(w[0], s, d);
  eq = eq_params<double>(omd * m.rho, m.ux, m.uy, m.E, d);
  return m.ok;
}

}  // namespace

template <int SCH>
__global__ void __launch_bounds__(kThreadsFx, 1)
    step_kernel_f64(const __grid_constant__ CUtensorMap tmap_in, const double* f_in, double* __restrict__ f_out,
                    const __grid_constant__ StepParams p, const __grid_constant__ DvmConst<double> d, int ty0) {
  using SZ = FxSize<SCH>;
  constexpr int PLANE = SZ::plane, TT = kTileT;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  double* sm = reinterpret_cast<double*>(smem_raw);
  int64_t* fx = reinterpret_cast<int64_t*>(smem_raw);
  FxTab<SCH>* tab = reinterpret_cast<FxTab<SCH>*>(smem_raw + SZ::planes_bytes);          // [pair][row]
  double* scratch = reinterpret_cast<double*>(smem_raw + SZ::planes_bytes + SZ::tab_bytes);
  uint64_t* bar = reinterpret_cast<uint64_t*>(smem_raw + SZ::planes_bytes + SZ::tab_bytes + SZ::scratch);
  int* top = reinterpret_cast<int*>(bar + 2);   // [4] largest high words of the shells

  const int r0 = blockIdx.x * kTileR;
  const int t0 = (blockIdx.y + ty0) * TT;   // ty0: first tile row of the launch
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;

  auto load = [&](uint64_t* b) {   // thread 0: window rows [t0-2, t0+TT+2) are stored rows [t0, t0+TT+4)
    mbar_arrive_expect_tx(b, (uint32_t)(kQ * PLANE * 8));
#pragma unroll 1
    for (int q = 0; q < kQ; ++q) tma_load_3d(sm + q * PLANE, &tmap_in, r0 - kLeft, t0, q, b);
  };
  if (tid == 0) {
    tma_prefetch_desc(&tmap_in);
    mbar_init(&bar[0], 1);
    mbar_init(&bar[1], 1);
    mbar_fence_init();
  }
  const double inv_r0 = p.inv_r[r0];
  if (tid < kPairsFx * TT) {   // Courant entries of the tile rows
    const int pair = tid / TT, rl = tid % TT;
    const double* e = p.courant64 + ((size_t)(min(t0 + rl, p.n_theta - 1) + kGhostRows) * kPairsFx + pair) * 4;
    FxTab<SCH> t;
    t.r = fx_coef<SCH>(fx_fraction(e[0]));
    t.at = fx_fraction(e[2] * inv_r0);
    t.fl = (int)e[3];
    t.pad = 0;
    tab[pair * TT + rl] = t;
  }
  if (tid < 4) top[tid] = 0;
  pdl_wait();      // the step before this one has written f and read f_out
  pdl_launch();    // the next one may start its set-up
  if (tid == 0) load(&bar[0]);
  // The whole block gives the tile up if any thread's wait ran out (block
  // barriers follow, so the decision must be uniform); thread 0 then gives
  // the copies one more bounded chance to land before the block exits.
  __syncthreads();
  auto wait = [&](uint64_t* b) {
    if (__syncthreads_or(p.wait_ns == 0 || !mbar_wait_bounded(b, 0, p.wait_ns))) {   // 0: give up at once
      if (tid == 0) {
        atomicOr(p.status, PCLB_FLAG_TIMEOUT);
        mbar_wait_bounded(b, 0, kDefaultWaitNs);
      }
      return false;
    }
    return true;
  };
  if (!wait(&bar[0])) return;

  const bool wall_tile = r0 == 0 || p.n_r - 1 - r0 <= kTileR;
  if (wall_tile) ghost_columns_f64<TT, PLANE>(sm, scratch, r0, t0, p, d);

  // ---- largest exponent of each shell, then its window in fixed point (the
  // rest plane stays as it is: no convection) ------------------------------------
  {
    const int* hi = reinterpret_cast<const int*>(sm) + 1;
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int first = (1 + g * kNDirs) * PLANE, n = kNDirs * PLANE;
      int m = 0;
      for (int i = tid; i < n; i += kThreadsFx) m = max(m, hi[2 * (first + i)] & 0x7fffffff);
      m = __reduce_max_sync(0xffffffffu, (unsigned)m);
      if (lane == 0) atomicMax(&top[g], m);
    }
  }
  __syncthreads();
  int ek[4];
  bool range = true;   // uniform over the block
#pragma unroll
  for (int g = 0; g < 4; ++g) {
    ek[g] = top[g] >> 20;
    range = range && ek[g] >= kFxMinExp && ek[g] <= kFxMaxExp;
  }
  if (range) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const int first = (1 + g * kNDirs) * PLANE, n = kNDirs * PLANE;
      for (int i = tid; i < n; i += kThreadsFx) fx[first + i] = fx_from_double(sm[first + i], ek[g]);
    }
  }
  __syncthreads();

  // ---- the node state and the equilibrium factors ------------------------------
  const int rl = warp;   // tile row
  const int r = r0 + lane, t = t0 + rl;
  const int node = (rl + 2) * kWinR + kLeft + lane;
  const bool valid = r < p.n_r && t < p.n_theta;
  const double decay = p.decay, omd = 1.0 - decay;
  EqParams<double> eq;
  double f0 = 0.0;
  auto shell_exp = [&](int k) { return k == 1 ? ek[0] : (k == 2 ? ek[1] : (k == 3 ? ek[2] : ek[3])); };
  unsigned slow = 1;   // bit k: shell k of this row from doubles; bit 0: the state and all shells
  if (range) {
    f0 = sm[node];
    double s0 = f0, sx = 0.0, sy = 0.0, se = 0.0;
    unsigned thin = 0;   // bit k: the node's values of shell k lie more than 2^5 below the largest
#pragma unroll 1
    for (int k = 1; k <= 4; ++k) {   // S, X = sum c_x f, Y: directions (1,0), (s,s), (0,1), (-s,s)
      const int64_t* f = fx + (1 + (k - 1) * kNDirs) * PLANE + node;
      int64_t S = 0, D[kHalfDirs];
      int most = 0;
#pragma unroll
      for (int i = 0; i < kHalfDirs; ++i) {
        const int64_t a = f[i * PLANE], b = f[(i + kHalfDirs) * PLANE];
        S += a + b;
        D[i] = a - b;
        const int ha = (int)(a >> 32), hb = (int)(b >> 32);
        most |= (ha ^ (ha >> 31)) | (hb ^ (hb >> 31));
      }
      if (most < kThinHi) thin |= 1u << k;
      const int e = shell_exp(k);
      const double Sd = fx_to_double(S, e);
      s0 += Sd;
      sx = fma(d.speed[k], fx_to_double(D[0] + fx_diagonal(D[1] - D[3]), e), sx);
      sy = fma(d.speed[k], fx_to_double(D[2] + fx_diagonal(D[1] + D[3]), e), sy);
      se = fma(d.half_v2[k], Sd, se);
    }
    // factors of (1 - d) f^eq: w_k = (1 - d) rho F_k
    const NodeState<double> m = node_state64(s0, sx, sy, se);
    eq = valid ? eq_params<double>(omd * m.rho, m.ux, m.uy, m.E, d) : eq_params<double>(1.0, 0.0, 0.0, 1.0, d);
    slow = 0;
    if (valid && thin) {   // the shells where (1 - d) rho times the largest term of F_k is no larger either
      const double E = m.E, w = fabs(omd) * m.rho;
#pragma unroll 1
      for (int k = 1; k <= 4; ++k) {
        if (!(thin >> k & 1)) continue;
        const double(&c)[4] = d.Fc[k];
        const double F = fmax(fmax(fabs(c[0]), fabs(c[1]) * E), fmax(fabs(c[2]), fabs(c[3]) * E) * E * E) * E;
        const int least = shell_exp(k) - 5;
        if (fx_exponent(__double2hiint(w * F)) < least) slow |= 1u << k;
        if ((slow >> k & 1) && fx_exponent(__double2hiint(m.rho)) < least) slow |= 1;
      }
    }
    if (valid && !m.ok) slow |= 1;
    slow = __reduce_or_sync(0xffffffffu, slow);
  }
  if (slow & 1) slow = 31;

  // ---- rows with shells from doubles: from global memory, or (tiles at a wall) from the window loaded again
  const size_t plane_out = (size_t)p.rows * p.pitch;
  const double* w64 = f_in + (size_t)(t + kGhostRows) * p.pitch + r;
  size_t plane64 = plane_out;
  int row64 = p.pitch;
  if (wall_tile && __syncthreads_or(slow != 0)) {
    if (tid == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      load(&bar[1]);
    }
    if (!wait(&bar[1])) return;
    ghost_columns_f64<TT, PLANE>(sm, scratch, r0, t0, p, d);
    w64 = sm + node;
    plane64 = PLANE;
    row64 = kWinR;
    slow = 31;
  }
  if (!valid) return;
  const uint64_t ratio = fx_fraction(p.inv_r[r] * recip_newton(inv_r0));   // 1/r relative to the tile's first column
  const NodeOut node_out{f_out, t, r};
  if (slow) {
    EqParams<double> e = eq;   // a copy in memory: the functions take it by reference
    if (slow & 1) {
      if (!stencil_state(w64, plane64, omd, d, e)) atomicOr(p.status, PCLB_FLAG_NONPHYS);
      f0 = w64[0];
      eq = e;
    }
#pragma unroll 1
    for (int k = 1; k <= 4; ++k)
      if (slow >> k & 1) stencil_shell<SCH, TT>(w64, plane64, row64, k, e, tab + rl, ratio, p, d, node_out);
  }

  // ---- output ------------------------------------------------------------------
  double* out = f_out + (size_t)(t + kGhostRows) * p.pitch + r;
  auto store = [&](int q, double v) {
    out[(size_t)q * plane_out] = v;
    if (t >= p.n_theta - 2)   // also the low ghost rows (theta <= 0) of the receiving label
      f_out[(size_t)d.recv_lo[q] * plane_out + (size_t)(t - (p.n_theta - 2)) * p.pitch + r] = v;
    if (t < 2)                // and the high ghost rows (theta > 2 pi n_f / n_dirs)
      f_out[(size_t)d.recv_hi[q] * plane_out + (size_t)(p.n_theta + kGhostRows + t) * p.pitch + r] = v;
  };
  store(0, fma(decay, f0, eq.w[0] * eq.a0));   // rest velocity: no convection
  const uint64_t dfx = fx_fraction(fabs(decay));
  const int64_t dsign = decay < 0.0 ? -1 : 0;
  const double c45 = d.cx[2];
  const double y1 = c45 * (eq.uyE + eq.uxE), y3 = c45 * (eq.uyE - eq.uxE);
  // A pair's results are stored one pair later, so that the FP64 pipe works
  // on them beside the next pair's integer part.
  int q_last = 0;
  double o1, o2;
#pragma unroll 1
  for (int k = 1; k <= 4; ++k) {
    if (slow >> k & 1) continue;
    const int e = shell_exp(k);
    // (1 - d) f^eq of the shell's pairs: ev +- od, ev = A + y^2 (B + y^2 C), od = y (O1 + y^2 O3)
    const double w = k == 1 ? eq.w[1] : (k == 2 ? eq.w[2] : (k == 3 ? eq.w[3] : eq.w[4])), wa = w * eq.a1;
    const double A = w * eq.a0, B = wa * d.half_v2[k], C = w * d.v4_24[k], O1 = wa * d.speed[k], O3 = w * d.v3_6[k];
#pragma unroll 1
    for (int i = 0; i < kHalfDirs; ++i) {
      const int q1 = 1 + (k - 1) * kNDirs + i, q2 = q1 + kHalfDirs;
      const double y = i == 0 ? eq.uxE : (i == 1 ? y1 : (i == 2 ? eq.uyE : y3)), y2 = y * y;
      const double ev = fma(y2, fma(y2, C, B), A), z = fma(y2, O3, O1);
      const FxTab<SCH>& te = tab[((k - 1) * kHalfDirs + i) * TT + rl];
      const FxCoef<SCH> cr = te.r, ct = fx_coef<SCH>(fx_mul_frac(te.at, ratio));
      const int fl = te.fl;
      const int sr = (fl & 1) ? 1 : -1;               // v_r < 0 for q1: upwind at larger r
      const int st = (fl & 2) ? kWinR : -kWinR;       // v_theta < 0 for q1: upwind at larger theta
      // d f - M_r - M_theta of a label whose upwind neighbours sit at s_r and s_t
      auto carried = [&](const int64_t* x, int s_r, int s_t) {
        const int64_t x0 = x[0];
        const int64_t keep = fx_signed(fx_mul(fx_abs(x0), dfx), (x0 >> 63) ^ dsign);
        return fx_to_double(keep - fx_increment<SCH>(x0, x[s_r], x[2 * s_r], x[-s_r], cr) -
                                fx_increment<SCH>(x0, x[s_t], x[2 * s_t], x[-s_t], ct), e);
      };
      const double g1 = carried(fx + q1 * PLANE + node, sr, st), g2 = carried(fx + q2 * PLANE + node, -sr, -st);
      if (q_last) {
        store(q_last, o1);
        store(q_last + kHalfDirs, o2);
      }
      o1 = fma(y, z, ev + g1);
      o2 = fma(-y, z, ev + g2);
      q_last = q1;
    }
  }
  if (q_last) {
    store(q_last, o1);
    store(q_last + kHalfDirs, o2);
  }
}

template <int SCH>
cudaError_t launch_step_small_f64(const CUtensorMap*, double*, const StepParams&, const DvmConst<double>&, cudaStream_t,
                                  int, int);

template <int SCH>
static cudaError_t launch_scheme(const CUtensorMap* tmap_in, const double* f_in, double* f_out, const StepParams& p,
                                 const DvmConst<double>& d, cudaStream_t stream, int ty_begin, int ty_end) {
  if (p.tile_rows != kTileT) {
    const int per = kTileT / p.tile_rows, last = (p.n_theta + p.tile_rows - 1) / p.tile_rows;
    return launch_step_small_f64<SCH>(tmap_in, f_out, p, d, stream, ty_begin * per, std::min(ty_end * per, last));
  }
  static std::atomic<unsigned long long> configured{0};   // per instantiation and device
  const cudaError_t e = set_smem_once(step_kernel_f64<SCH>, FxSize<SCH>::smem, configured);
  if (e != cudaSuccess) return e;
  const dim3 grid((p.n_r + kTileR - 1) / kTileR, ty_end - ty_begin);
  return launch_overlapped(step_kernel_f64<SCH>, grid, kThreadsFx, FxSize<SCH>::smem, stream, *tmap_in, f_in, f_out,
                           p, d, ty_begin);
}

// Tile rows [ty_begin, ty_end) of the grid, kTileT nodes each (ty_end < 0: to
// the last tile row); an empty range launches nothing.  tmap_in: f_in in boxes
// of p.tile_rows + 4 window rows.
template <class T>
cudaError_t launch_step(const CUtensorMap* tmap_in, const T* f_in, T* f_out, const StepParams& p,
                        const DvmConst<T>& d, cudaStream_t stream, int ty_begin, int ty_end) {
  if (ty_end < 0) ty_end = (p.n_theta + kTileT - 1) / kTileT;
  if (ty_begin < 0 || ty_end <= ty_begin) return cudaSuccess;
  switch (p.scheme) {
    case PCLB_SCHEME_WB: return launch_scheme<PCLB_SCHEME_WB>(tmap_in, f_in, f_out, p, d, stream, ty_begin, ty_end);
    case PCLB_SCHEME_LW: return launch_scheme<PCLB_SCHEME_LW>(tmap_in, f_in, f_out, p, d, stream, ty_begin, ty_end);
    case PCLB_SCHEME_UPWIND2: return launch_scheme<PCLB_SCHEME_UPWIND2>(tmap_in, f_in, f_out, p, d, stream, ty_begin, ty_end);
    default: return launch_scheme<PCLB_SCHEME_MWB>(tmap_in, f_in, f_out, p, d, stream, ty_begin, ty_end);
  }
}

template cudaError_t launch_step<double>(const CUtensorMap*, const double*, double*, const StepParams&,
                                         const DvmConst<double>&, cudaStream_t, int, int);

}  // namespace pclb
