// Float tables of the N_i = 16 and 24 velocity sets (Table I) for their FP32
// step (dvm_tiled32.cu), beside the double constants of DvmG; and the entry
// points of the steps of these sets.
#pragma once

#include "pclb.h"
#include "pclb_internal.h"

namespace pclb {

constexpr int kMaxPairsG = kMaxQ / 8;   // N_i / 2 <= 12 opposite-direction pairs per shell

// Float-float constants are pairs (h, l) with h + l the double value.
struct DvmG32 {
  float vx[kMaxQ], vy[kMaxQ];                  // v_q rounded to float
  float cxh[kMaxPairsG], cxl[kMaxPairsG];      // unit vector of direction i < N_i / 2 (Eq. 2)
  float cyh[kMaxPairsG], cyl[kMaxPairsG];
  float sph[5], spl[5], hvh[5], hvl[5];        // v_k and v_k^2 / 2
  float dv23h, dv23l, dh23h, dh23l;            // v_3 - v_2 and (v_3^2 - v_2^2) / 2
  float Fch[5][4], Fcl[5][4];                  // F_k(E) = sum_n Fc[k][n-1] E^n (Eq. 11a)
  float B0h, B0l;                              // F_0 = 1 - B0 sum_k F_k (Eq. 11b)
  // For sums in integers (gen_state.cuh): v_k = fx_speed[k-1] 2^(fx_exp_v - 63), v_k^2 / 2
  // = fx_half_v2[k-1] 2^(fx_exp_hv - 63), the unit vectors' |x| and y in 2^-63; fx_neg_x bit
  // i: x < 0; fx_ok: the speeds are such that this holds.
  uint64_t fx_speed[4], fx_half_v2[4], fx_cx[kMaxPairsG], fx_cy[kMaxPairsG];
  int fx_exp_v, fx_exp_hv, fx_neg_x, fx_ok;
};

void fill_dvm_generic32(DvmG32& c, const pclb_dvm& d, const DvmG& g);

// f^eq of the fields in FP64 (dvm_step_f64.cu).
cudaError_t gen_launch_set_state_f64(double* f, const double* rho, const double* ur, const double* ut,
                                     const double* temp, const StepParams& p, const DvmG& d, cudaStream_t s);

// One FP64 step of the N_i = 16 or 24 set (dvm_step_f64.cu): the radial ghost
// layers into ghost [side][layer][n_theta][Q], then the nodes.
cudaError_t gen_launch_step_f64(const double* f, double* f_out, double* ghost, const StepParams& p, const DvmG& d,
                                cudaStream_t s);

// One FP32 step of the N_i = 16 or 24 set (the tiled kernel); tmap describes f
// (box kWinR x (kTileT32 + 4) x 1 over Q planes).
cudaError_t gen_tiled_step_f32(const CUtensorMap* tmap, const float* f, float* f_out, const StepParams& p,
                               const DvmG& d, const DvmG32& c, cudaStream_t s);

}  // namespace pclb
