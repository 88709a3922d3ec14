// Copies between the packed [Q][n_theta][n_r] layout and the stored layout
// (azimuthal ghost rows, padded rows), for every velocity set.
//
// Bound: HBM (one read and one write of the distribution).  One warp moves
// one piece of a row, every lane kCopyUnroll (16-byte) or 2 kCopyUnroll
// (element) accesses of which all loads are issued before the first store,
// so that a few thousand CTAs keep ~64 KB per SM in flight.  One element per
// thread (535k CTAs on 1999 x 1013, FP32) had taken 270 us per copy there, 30% of
// the copy rate; this form is bound by HBM.  16-byte accesses where both sides
// allow them (the packed array 16-byte aligned and n_r whole vectors);
// the stored rows always are aligned.
#pragma once

#include <cuda_runtime.h>

#include "pclb_internal.h"

namespace pclb {

constexpr int kCopyThreads = 256;
constexpr int kCopyUnroll = 8;

template <class T, class V>
struct CopyPiece {
  static constexpr int kPer = sizeof(V) / sizeof(T);                            // elements per access
  static constexpr int kAcc = sizeof(V) == 16 ? kCopyUnroll : 2 * kCopyUnroll;   // accesses per lane
  static constexpr int kLen = 32 * kPer * kAcc;                                 // elements per warp
};

// Labels whose azimuthal ghost rows copy the seam rows of label q (Eq. 40).
struct RecvLabels {
  int8_t recv_lo[kMaxQ], recv_hi[kMaxQ];
};

template <class D>
inline RecvLabels recv_labels(const D& d, int n_labels) {
  RecvLabels r{};
  for (int q = 0; q < n_labels; ++q) {
    r.recv_lo[q] = (int8_t)d.recv_lo[q];
    r.recv_hi[q] = (int8_t)d.recv_hi[q];
  }
  return r;
}

// UNPACK: packed -> stored with the seam rows' ghost copies (Eq. 40),
// else stored -> packed.
template <class T, class V, bool UNPACK>
__global__ void __launch_bounds__(kCopyThreads)
    copy_rows_kernel(const T* __restrict__ src, T* __restrict__ dst, int pieces, size_t items,
                     const __grid_constant__ StepParams p, const __grid_constant__ RecvLabels d) {
  using P = CopyPiece<T, V>;
  const size_t item = (size_t)blockIdx.x * (kCopyThreads / 32) + (threadIdx.x >> 5);
  if (item >= items) return;
  const size_t row = item / pieces;
  const int q = (int)(row / p.n_theta), t = (int)(row % p.n_theta);
  const int r0 = (int)(item % pieces) * P::kLen + (threadIdx.x & 31) * P::kPer;
  const size_t plane = (size_t)p.rows * p.pitch;
  const size_t packed = row * p.n_r, stored = (size_t)q * plane + (size_t)(t + kGhostRows) * p.pitch;
  const T* s = src + (UNPACK ? packed : stored);
  V v[P::kAcc];
#pragma unroll
  for (int i = 0; i < P::kAcc; ++i) {
    const int r = r0 + i * 32 * P::kPer;
    if (r < p.n_r) v[i] = *reinterpret_cast<const V*>(s + r);
  }
  auto put = [&](T* o) {
#pragma unroll
    for (int i = 0; i < P::kAcc; ++i) {
      const int r = r0 + i * 32 * P::kPer;
      if (r < p.n_r) *reinterpret_cast<V*>(o + r) = v[i];
    }
  };
  put(dst + (UNPACK ? stored : packed));
  if constexpr (UNPACK) {
    if (t >= p.n_theta - 2) put(dst + (size_t)d.recv_lo[q] * plane + (size_t)(t - (p.n_theta - 2)) * p.pitch);
    if (t < 2) put(dst + (size_t)d.recv_hi[q] * plane + (size_t)(p.n_theta + kGhostRows + t) * p.pitch);
  }
}

template <class T, bool UNPACK>
cudaError_t launch_copy_rows(const T* src, T* dst, int n_labels, const StepParams& p, const RecvLabels& d,
                             cudaStream_t s) {
  const void* packed = UNPACK ? static_cast<const void*>(src) : static_cast<const void*>(dst);
  auto go = [&](auto vec) {
    using V = decltype(vec);
    const int pieces = (p.n_r + CopyPiece<T, V>::kLen - 1) / CopyPiece<T, V>::kLen;
    const size_t items = (size_t)n_labels * p.n_theta * pieces;
    const size_t blocks = (items + kCopyThreads / 32 - 1) / (kCopyThreads / 32);
    copy_rows_kernel<T, V, UNPACK><<<(unsigned)blocks, kCopyThreads, 0, s>>>(src, dst, pieces, items, p, d);
    return cudaGetLastError();
  };
  const bool wide = reinterpret_cast<uintptr_t>(packed) % 16 == 0 && (size_t)p.n_r * sizeof(T) % 16 == 0;
  return wide ? go(float4{}) : go(T{});
}

}  // namespace pclb
