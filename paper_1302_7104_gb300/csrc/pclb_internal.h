// Internal types shared by the host side of the C ABI and the kernels.
// Not part of the public interface (include/pclb.h).
#pragma once

#include <atomic>
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "pclb.h"

namespace pclb {

// The discrete velocity model built here: N_k = 4 shells of kNDirs directions
// plus the rest velocity (Eq. 2), Q = 33 for the octagon.
constexpr int kNDirs = 8;
constexpr int kQ = 1 + 4 * kNDirs;

// Tiling of the fused step kernel.  A tile is kTileR x kTileT interior nodes;
// its shared-memory window holds every velocity plane over
// [r0 - 4, r0 + kTileR + 4) x [t0 - 2, t0 + kTileT + 2): the +-2 stencil halo
// in both directions, with the radial start rounded down to a 16-byte
// boundary so the TMA box starts aligned.
constexpr int kTileR = 32;
constexpr int kTileT = 16;
// FP32 step kernel: tile rows, threads (two radially adjacent nodes each) and
// CTAs per SM
constexpr int kTileT32 = 16;
constexpr int kStepThreads32 = 16 * kTileT32;
constexpr int kCtasPerSm32 = 2;
// The octagon's steps on small grids: tiles of kTileTSmall rows on at most
// kSmallGridTiles tiles of 32 x 16 (two waves of the 152 SMs), in FP64 of two
// rows on at most kTinyGridTiles64 (one wave).  FP64, us per step with tiles
// of 2 / 4 / 16 rows: 64 x 128 (16 tiles) 16.4 / 24.2 / 53.2, 64 x 256 (32)
// 32.5 / 24.5 / 53.3, 128 x 304 (76) 65.2 / 48.5 / 53.3, 128 x 608 (152)
// 123 / 96.7 / 54.2.  FP32, us per step with 4 / 16: 64 x 128 7.5 / 13.1, 64 x
// 608 (76) 8.9 / 13.3, 128 x 400 (100) 15.0 / 13.5.
constexpr int kTileTSmall = 4;
constexpr int kSmallGridTiles = 76, kTinyGridTiles64 = 19;
constexpr int kWinR = kTileR + 8;   // 40 columns
constexpr int kLeft = 4;            // column of interior r0 inside the window
constexpr int kPitchAlign = 32;     // row pitch in elements (128 B for float)
constexpr int kGhostRows = 2;       // azimuthal ghost rows stored on each side
// Tile rows of the adjoint kernel (its window holds f and lam for all labels).
constexpr int kAdjRows32 = 16;
constexpr int kAdjRows64 = 8;
constexpr int kAdjRows64Small = 4;    // FP64 on grids of at most kSmallGridTilesAdj tiles of 8 rows
// us per adjoint step with tiles of 4 / 8 rows: 64 x 304 (76 tiles of 8) 104 /
// 154, 128 x 304 (152) 157 / 154, 128 x 400 (200) 213 / 256, 128 x 608 (304) 281 /
// 258: up to three of the small ones per SM (152 SMs, two at a time).  With
// more than 152 of the large ones some SMs hold two and take as long as 304 do.
constexpr int kSmallGridTilesAdj = 228;
// 2 rows on at most kTinyGridTilesAdj (one of their blocks to an SM): 64 x 152
// (38) 73.4 us against 104 with 4 rows, 64 x 304 (76) 104 against 104.
constexpr int kAdjRows64Tiny = 2;
constexpr int kTinyGridTilesAdj = 38;
// Time a kernel waits for the TMA copies of its own window (mbarrier phase)
// before it reports PCLB_FLAG_TIMEOUT and gives the tile up; the copies of a
// tile given up get the default limit again to land before the CTA exits.
// The step kernels take their first wait's limit from StepParams::wait_ns
// (pclb_set_wait_limit); every other wait uses the default.
constexpr uint64_t kDefaultWaitNs = 2000000000ull;   // 2 s
constexpr uint64_t kMaxWaitNs = 60000000000ull;      // 60 s

// Per-velocity constants, in the arithmetic type T of the kernel, plus the
// double-precision ones the moment / temperature recovery uses.
template <class T>
struct DvmConst {
  T vx[kQ], vy[kQ];           // Cartesian components v_qx, v_qy
  T cx[kQ], cy[kQ];           // unit direction (cos phi_i, sin phi_i); 0 for q = 0
  T speed[5];                 // v_k
  T half_v2[5];               // v_k^2 / 2
  T v3_6[5], v4_24[5];        // v_k^3 / 6, v_k^4 / 24
  T Fc[5][4];                 // F_k(E) = sum_{n=1..4} Fc[k][n-1] E^n, k = 1..4 (Eq. 11a)
  T Fc_lo[5][4];              // Fc - (double)Fc rounded to T: the low part of a float-float pair
  // Low parts (value - (double)hi, rounded to T) of the velocity constants, so
  // that the FP32 path can use them as float-float pairs; zero for double.
  T vx_lo[kQ], vy_lo[kQ], cx_lo[kQ], cy_lo[kQ];
  T speed_lo[5], half_v2_lo[5];
  // v_3 - v_2 and (v_3^2 - v_2^2)/2 as float-float pairs: the FP32 moments sum
  // shells 2 and 3 direction by direction (their speeds are close and their
  // weights opposite), then correct with these differences.
  T dv23, dv23_lo, dh23, dh23_lo;
  T B0;                       // F_0 = 1 - B0 (F_1 + .. + F_4) (Eq. 11b)
  int8_t shell[kQ];           // k of label q
  int8_t recv_lo[kQ];         // label whose low ghost rows copy rows n_theta-2.. of label q
  int8_t recv_hi[kQ];         // label whose high ghost rows copy rows 0, 1 of label q
};

// Velocity sets with N_i = 16 or 24 (Table I), for the generic kernels; all
// constants in double.
constexpr int kMaxQ = 1 + 4 * 24;
struct DvmG {
  double vx[kMaxQ], vy[kMaxQ];
  double half_v2[5];          // v_k^2 / 2
  double Fc[5][4];            // F_k(E) = sum_{n=1..4} Fc[k][n-1] E^n, k = 1..4 (Eq. 11a)
  double B0;                  // F_0 = 1 - B0 (F_1 + .. + F_4) (Eq. 11b)
  int shell[kMaxQ];
  int recv_lo[kMaxQ], recv_hi[kMaxQ];   // as in DvmConst
  int n_dirs, q;
};

struct StepParams {
  int n_r, n_theta;           // interior nodes
  int pitch;                  // elements per stored row (multiple of kPitchAlign)
  int rows;                   // stored rows per plane: n_theta + 4
  double dt_dr;               // dt / dr
  double dt_dth;              // dt / dtheta
  double decay;               // exp(-dt / tau), Eq. (19), or 1 - dt / tau (forward Euler)
  int bc_kind[2];
  int scheme;                 // pclb_scheme of the convection increments
  const double* cos_t;        // [n_theta] cos(theta_i), host-computed in double
  const double* sin_t;        // [n_theta]
  const double* inv_r;        // [n_r] 1 / r_i
  const double* bc_vals;      // [2 sides][2 layers][4 fields][n_theta] or unused
  const float4* courant;      // [n_theta + 4][4 n_dirs / 2] (stored rows, ghosts included): per
                              // opposite-velocity pair (first label
                              // q of the pair) |C_r|, |C_r|(1 - |C_r|), |v_theta| dt / dtheta,
                              // flags (bit 0: v_r < 0, bit 1: v_theta < 0) as int bits
  const double* courant64;    // the same table in double: [n_theta + 4][pairs][4] (flags as value)
  const float* inv_r_f;       // [n_r] 1 / r_i in float
  const float4* cs_ff;        // [n_theta] cos theta_i, sin theta_i as float-float pairs (hi, lo, hi, lo)
  int tile_rows;              // tile rows of the step: kTileT, kTileTSmall or (FP64) 2
  int adj_rows;               // tile rows of the adjoint
  uint32_t* status;           // device status word (PCLB_FLAG_*)
  uint64_t wait_ns;           // a step's wait for its own window copies before it gives the tile up
};

// Workspace layout (byte offsets from the caller's base pointer).
struct Layout {
  size_t f[2];                // two ping-pong distributions [Q][rows][pitch]
  size_t adj_f;               // a state copy for pclb_adjoint_step
  size_t lam[2];              // ping-pong adjoint variables, same layout as f
  size_t f_bytes;
  size_t cos_t, sin_t, inv_r, bc_vals, courant, courant64, inv_r_f, cs_ff;
  size_t status;              // uint32 status word (+ padding)
  size_t partials;            // double [kDiagBlocks][8] reduction partials
  size_t diag_out;            // double [8]
  size_t stage;               // host-I/O staging: 8 fields [n_theta][n_r]
  size_t adj_scratch;         // the adjoint's wall scratch (adjoint_walls.cuh)
  size_t gen_ghost;           // N_i = 16, 24, FP64: radial ghost values [side][layer][n_theta][Q]
  size_t total;
};

// Raises kernel fn's dynamic shared-memory limit to `bytes` once per device
// (the attribute belongs to each device's context); `done` holds one bit per
// device ordinal.
template <class F>
inline cudaError_t set_smem_once(F* fn, int bytes, std::atomic<unsigned long long>& done) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  const unsigned long long bit = dev < 64 ? (1ull << dev) : 0ull;
  if (bit && (done.load(std::memory_order_acquire) & bit)) return cudaSuccess;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e == cudaSuccess && bit) done.fetch_or(bit, std::memory_order_release);
  return e;
}

constexpr int kOwnSmBytes = 116 * 1024;   // more than half of an SM's 228 KB

// Launches fn so that its start overlaps the end of the kernel before it on
// the stream (programmatic dependent launch): fn calls pdl_wait() before it
// touches anything that kernel reads or writes.
template <class... P, class... A>
inline cudaError_t launch_overlapped(void (*fn)(P...), dim3 grid, int threads, int smem, cudaStream_t stream,
                                     const A&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = (size_t)smem;
  cfg.stream = stream;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fn, args...);
}

// Shared memory of an adjoint launch of that many blocks, each needing smem.
// Its blocks are placed while the step before it still holds most SMs, and
// would pile up on the free ones; where there is an SM for each (152), they ask
// for more than half of one.  A step and an adjoint step, without and with: FP64
// 64 x 128 121 and 92 us, 64 x 256 182 and 129; FP32 128 x 304 69.6 and 51.6.
// Contexts on streams of their own lose nothing by it (adjoint steps of four, FP64
// 64 x 128: 60 us each, FP32 128 x 304: 14.4).
inline int adjoint_smem(int smem, int blocks) { return blocks <= 152 && smem < kOwnSmBytes ? kOwnSmBytes : smem; }

size_t adjoint_scratch_bytes(int n_theta, int elem);

constexpr int kDiagBlocks = 304;    // 2 x 152 SMs

// Adds up the blocks' partials of the global integrals (field_kernels.cu).
cudaError_t launch_diag_final(const double* partials, int n_blocks, double* out, double n_nodes, cudaStream_t s);

// Host helpers shared by the C-ABI translation units (defined in pclb_abi.cu).
pclb_status validate_problem(const pclb_grid* g, const pclb_dvm* d, pclb_precision prec);
template <class T>
void fill_dvm(DvmConst<T>& c, const pclb_dvm& d, const pclb_grid& g);
void set_thread_error(const char* msg);   // text returned by pclb_last_error(NULL)

// Element size of a precision.
inline size_t elem_size(pclb_precision p) { return p == PCLB_FP64 ? 8 : 4; }

}  // namespace pclb

// Host context behind the opaque pclb_ctx handle.
struct pclb_ctx {
  pclb_grid grid;
  pclb_dvm dvm;
  pclb_precision prec;
  double tau, dt;
  int32_t bc_kind[2];   // pclb_bc_kind, possibly with PCLB_BC_NEQ
  int32_t scheme = 0;       // pclb_scheme
  int32_t relaxation = 0;   // pclb_relaxation
  cudaStream_t stream;
  cudaStream_t capture = nullptr;     // private stream for capturing step graphs
  struct StepGraph {
    int32_t n, cur;                   // steps and starting buffer of the captured sequence
    cudaGraphExec_t exec;
  } graphs[4] = {};
  int32_t n_graphs = 0;
  // pclb_run_host with page-locked buffers: the host transfers of each
  // azimuthal slab run on two copy streams and its set-state kernel on a
  // third stream while the steps of other slabs run on `stream` and io_alt
  // (created on first use)
  static constexpr int kIoSlabs = 16;
  cudaStream_t io_in = nullptr, io_set = nullptr, io_out = nullptr, io_alt = nullptr;
  cudaEvent_t io_start = nullptr, io_done = nullptr;
  cudaEvent_t io_loaded[kIoSlabs] = {}, io_isset[kIoSlabs] = {}, io_ready[kIoSlabs] = {};
  unsigned char* ws;
  pclb::Layout lay;
  int cur;                    // which of the two f buffers holds the state
  bool has_state;
  CUtensorMap tmap[2];        // TMA descriptors of the two f buffers
  CUtensorMap tmap_adj[5];    // adjoint-window descriptors: f[0], f[1], adj_f, lam[0], lam[1]
  CUtensorMap tmap_node[5];   // FP32 adjoint node-phase descriptors (tile boxes) of the same buffers
  int cur_lam;                // which lam buffer holds the adjoint variable
  bool has_lam;
  pclb::StepParams sp;
  pclb::DvmConst<float> dvm32;
  pclb::DvmConst<double> dvm64;
  pclb::DvmG dvmg;            // N_i = 16, 24 (the generic kernels)
  char err[512];
};
