// The FP32 z-t plane kernel of the plane pipelines (k_fft_zt.cu describes the pass
// and instantiates the shapes with tuned schedules; k_zt_pairs.cu the other
// pairs of common extents): one CTA per field and run of BX consecutive (x, y)
// columns, which are contiguous at every (z, t) whatever Lx; a run may cross
// from one y to the next, and the last one may be ragged.
#pragma once

#include "fft_reg.cuh"
#include "lgf_df.cuh"
#include "lgf_kernels.cuh"

namespace lgf {

// pitch of one t slice: BX*LZ plus padding that shifts consecutive t slices
// by one run of BX elements across the 32 shared-memory banks
template <class T, int LZ, int BX>
constexpr int zt_pitch() {
  constexpr int W = (int)sizeof(cx<T>) / 4;  // banks per element
  for (int pad = 0; pad < 32; ++pad)
    if ((((BX * LZ + pad) * W) % 32) == ((BX * W) % 32)) return BX * LZ + pad;
  return BX * LZ;
}

template <int LZ, int LT, int BX>
constexpr int zt_threads() {
  return BX * (LZ > LT ? LZ : LT);
}

// a thread holds a whole t line through the forward transform, the factor and
// the inverse: FP32 lines up to 32 run 3 CTAs of 128 threads per SM at BX = 4
// (up to 170 registers, no spills; 4 CTAs at 128 registers spilled 56 bytes
// per thread and took 22.6 instead of 21.7 us at 32^4, 5 and 6 CTAs took
// 23.9 and 28.9 us), 2 of 256 at BX = 8
template <int LZ, int LT, int BX>
constexpr int zt_min_blocks() {
  return LZ <= 32 && LT <= 32 ? (BX <= 4 ? 3 : 2) : 1;
}

template <class T, int LZ, int LT, int BX>
constexpr size_t zt_smem_bytes() {
  return (size_t)zt_pitch<T, LZ, BX>() * LT * sizeof(cx<T>);
}

// the low parts of s2p[0] (x, y, z) and of c_over_V, for factors rounded once
constexpr int kS2Low = 3 * 4 * kMaxL;
constexpr int kCLow = kS2Low + 3 * kMaxL;

// the x, y and z terms of p2(k) as hi + lo
__device__ __forceinline__ df p2_xyz(const float* __restrict__ s2p, int x, int y, int z) {
  const df xy = two_sum(__ldg(s2p + x), __ldg(s2p + kMaxL + y));
  df a = two_sum(xy.h, __ldg(s2p + 2 * kMaxL + z));
  a.l += xy.l + (__ldg(s2p + kS2Low + x) + __ldg(s2p + kS2Low + kMaxL + y) + __ldg(s2p + kS2Low + 2 * kMaxL + z));
  return a;
}

// p2_max / (V p2(k)) at position P of a t line (radix order 0)
template <int LT, int P>
__device__ __forceinline__ float factor_rounded(df c, df a) {
  constexpr double s2 = regfft::MomentumSq<LT, P>::value;
  constexpr float h = (float)s2, l = (float)(s2 - (double)h);
  return df_quotient(c, a, {h, l});
}

// FP32: factor from s2p[RO][axis][position] and c_over_V = p2_max / V, 0 at
// k = 0.  EXACT (RO 0): rounded once from hi + lo parts, 6e-8 of it, for the
// shapes whose factor has always been formed in FP64 and rounded; the tuned
// shapes' is formed in FP32, up to 2e-7.
template <int LZ, int LT, int BX, int RO, bool EXACT = false>
__global__ void __launch_bounds__(zt_threads<LZ, LT, BX>(), zt_min_blocks<LZ, LT, BX>())
    k_plane_zt(cx<float>* __restrict__ D, int Lx, int Ly, const float* __restrict__ s2p, float c_over_V,
               const DevState* __restrict__ st) {
  using T = float;
  pdl_wait();
  if (st != nullptr && st->done) return;
  constexpr int PT = zt_pitch<T, LZ, BX>();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* tile = reinterpret_cast<cx<T>*>(smem_raw);  // [t][z][xb], t pitch PT
  const int q0 = blockIdx.x * BX;
  const int f = blockIdx.y;
  const int LxLy = Lx * Ly;
  const int V = LxLy * LZ * LT;
  const int xb = threadIdx.x % BX, row = threadIdx.x / BX;
  const bool inside = q0 + xb < LxLy;
  cx<T>* Df = D + (f * V + q0);
  // forward z: line (xb, t) straight from global memory (for each z a warp
  // reads BX consecutive x at 32 / BX values of t: whole 32-byte sectors)
  if (inside && row < LT) {
    const int t = row;
    cx<T>* line = tile + t * PT + xb;
    const cx<T>* g = Df + (xb + LxLy * LZ * t);
    cx<T> v[LZ];
#pragma unroll
    for (int p = 0; p < LZ; ++p) {  // running pointer: one address register
      v[p] = *g;
      g += LxLy;
    }
    regfft::forward<T, LZ, RO>(v);
#pragma unroll
    for (int p = 0; p < LZ; ++p) line[p * BX] = v[p];
  }
  __syncthreads();
  // t lines (xb, z): forward, acceleration factor, inverse
  if (inside && row < LZ) {
    const int z = row;
    cx<T>* line = tile + z * BX + xb;
    cx<T> v[LT];
#pragma unroll
    for (int p = 0; p < LT; ++p) v[p] = line[p * PT];
    regfft::forward<T, LT, RO>(v);
    const int q = q0 + xb, y = q / Lx, x = q - y * Lx;
    // the t contribution at each position is a compile-time constant
    const bool origin = (x | y | z) == 0;
    if constexpr (EXACT) {
      const df a = p2_xyz(s2p, x, y, z), c = {c_over_V, __ldg(s2p + kCLow)};
      regfft::static_for<0, LT>([&](auto pc) {
        constexpr int p = decltype(pc)::value;
        v[p] = scale(v[p], p == 0 && origin ? 0.0f : factor_rounded<LT, p>(c, a));
      });
    } else {
      const float a = __ldg(s2p + x) + __ldg(s2p + kMaxL + y) + __ldg(s2p + RO * 4 * kMaxL + 2 * kMaxL + z);
      regfft::static_for<0, LT>([&](auto pc) {
        constexpr int p = decltype(pc)::value;
        constexpr float s2t = (float)regfft::MomentumSq<LT, p, RO>::value;
        float kf = c_over_V * rcp_approx(a + s2t);
        if (p == 0 && origin) kf = 0.0f;
        v[p] = scale(v[p], (T)kf);
      });
    }
    regfft::inverse<T, LT, RO>(v);
#pragma unroll
    for (int p = 0; p < LT; ++p) line[p * PT] = v[p];
  }
  __syncthreads();
  // inverse z, stored straight to global memory
  if (inside && row < LT) {
    const int t = row;
    const cx<T>* line = tile + t * PT + xb;
    cx<T>* g = Df + (xb + LxLy * LZ * t);
    cx<T> v[LZ];
#pragma unroll
    for (int p = 0; p < LZ; ++p) v[p] = line[p * BX];
    regfft::inverse<T, LZ, RO>(v);
#pragma unroll
    for (int p = 0; p < LZ; ++p) {
      *g = v[p];
      g += LxLy;
    }
  }
}

}  // namespace lgf
