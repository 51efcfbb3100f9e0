// 3x3 complex matrices in host layout (18 doubles each, consecutive) staged
// through shared memory: a CTA moves one contiguous chunk of matrices with
// coalesced 16-byte accesses, one thread per matrix works on its staged row.
// The pitch of 19 doubles keeps the per-thread 8-byte accesses free of bank
// conflicts.  The host-layout side may be host memory that the device reads
// or writes directly (pinned memory over NVLink-C2C): every byte crosses
// once, coalesced.
#pragma once

#include "lgf_common.cuh"

namespace lgf {

constexpr int kStageMats = 256;   // links per CTA of the link loads and stores
constexpr int kStagePitch = 19;   // doubles per staged matrix

// n matrices from the first'th on, into sm
__device__ __forceinline__ void stage_in(const double* __restrict__ aos, double* sm, int64_t first, int n) {
  const double2* src = reinterpret_cast<const double2*>(aos + first * 18);
  for (int j = threadIdx.x; j < n * 9; j += blockDim.x) {
    const double2 v = src[j];  // doubles 2j and 2j+1 of the chunk: one matrix, entries k and k+1
    const int m = (2 * j) / 18, k = (2 * j) - m * 18;
    sm[m * kStagePitch + k] = v.x;
    sm[m * kStagePitch + k + 1] = v.y;
  }
}

__device__ __forceinline__ void stage_out(const double* sm, double* __restrict__ aos, int64_t first, int n) {
  double2* dst = reinterpret_cast<double2*>(aos + first * 18);
  for (int j = threadIdx.x; j < n * 9; j += blockDim.x) {
    const int m = (2 * j) / 18, k = (2 * j) - m * 18;
    dst[j] = make_double2(sm[m * kStagePitch + k], sm[m * kStagePitch + k + 1]);
  }
}

// this thread's matrix into its staged row
template <class T>
__device__ __forceinline__ void stage_matrix(double* sm, const M3<T>& m) {
  double* d = sm + threadIdx.x * kStagePitch;
#pragma unroll
  for (int q = 0; q < 9; ++q) {
    d[2 * q] = (double)m.e[q / 3][q % 3].re;
    d[2 * q + 1] = (double)m.e[q / 3][q % 3].im;
  }
}

}  // namespace lgf
