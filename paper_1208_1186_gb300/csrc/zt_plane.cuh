// The FP32 z-t plane kernel of the plane pipelines (k_fft_zt.cu describes the pass
// and instantiates the shapes with tuned schedules; k_zt_pairs.cu the other
// pairs of common extents): one CTA per field and run of BX consecutive (x, y)
// columns, which are contiguous at every (z, t) whatever Lx; a run may cross
// from one y to the next, and the last one may be ragged.
#pragma once

#include "fft_reg.cuh"
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

// TABLE: the CTAs per SM that the lines' registers leave without the loads of
// the factors, which otherwise would be kept in flight in more registers (20 x
// 40: 148 instead of 127, two CTAs per SM for three).  us with the factor formed in
// FP32 and from the table: 18 x 40 16.6 and 17.1, 20 x 40 12.6 and 12.4, 10 x 24 7.9
// and 7.8, 30 x 10 12.4 and 12.4; lines of 36 lose a CTA, 24 x 36 13.6 and 17.1 (held
// to four they spill: 18 x 36 10.6, 10.9 and 14).
template <int LZ, int LT, int BX>
constexpr int zt_table_min_blocks() {
  constexpr int m = LZ > LT ? LZ : LT;
  return m <= 24 ? zt_min_blocks<LZ, LT, BX>() : m <= 32 ? 5 : m <= 40 ? 3 : m <= 48 ? 2 : 1;
}

template <class T, int LZ, int LT, int BX>
constexpr size_t zt_smem_bytes() {
  return (size_t)zt_pitch<T, LZ, BX>() * LT * sizeof(cx<T>);
}

// factor from s2p[RO][axis][position] and c_over_V = p2_max / V, formed in FP32,
// 0 at k = 0 (up to 2e-7 off).  TABLE (RO 0): from kfac, formed in FP64 and
// rounded, for the shapes whose factor has always been.
template <int LZ, int LT, int BX, int RO, bool TABLE = false>
__global__ void __launch_bounds__(zt_threads<LZ, LT, BX>(), TABLE ? zt_table_min_blocks<LZ, LT, BX>()
                                                                  : zt_min_blocks<LZ, LT, BX>())
    k_plane_zt(cx<float>* __restrict__ D, int Lx, int Ly, const float* __restrict__ s2p, float c_over_V,
               const float* __restrict__ kfac, const DevState* __restrict__ st) {
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
    if constexpr (TABLE) {
      const float* k = kfac + (q + LxLy * z);
#pragma unroll
      for (int p = 0; p < LT; ++p) {
        v[p] = scale(v[p], __ldg(k));
        k += LxLy * LZ;
      }
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
