// Geometry and launchers of the plane kernels whose extents are run-time values:
// fft_any.cuh (FP32, a thread per line), fft_fx.cuh (FP64 lines up to 32) and
// k_fft_long.cu (two steps a line).
#pragma once

#include "lgf_kernels.cuh"

namespace lgf {
namespace anyfft {

// quotient by a run-time divisor d: exact for n < 2^32 / d with rcp = ceil(2^32 / d)
struct Div {
  unsigned d, rcp;
};
inline Div make_div(int d) { return {(unsigned)d, 0xFFFFFFFFu / (unsigned)d + 1u}; }
__device__ __forceinline__ int quot(int n, const Div& v) { return v.d == 1 ? n : (int)__umulhi((unsigned)n, v.rcp); }

struct XyGeom {
  int Lx, Ly, P, N;  // extents, padded row pitch, Lx Ly
  int V, ntiles, tpc;  // sites, (plane, field) tiles, tiles per CTA
  Div x;               // by Lx
};

struct ZtGeom {
  int Lz, Lt;
  int S, V;       // Lx Ly columns, sites
  int bx, lbx;    // columns per tile (a power of two) and its logarithm
  int PT;         // padded t pitch of a tile
};

constexpr int kXyThreads = 128;

// threads of a z-t CTA: bx max(Lz, Lt) at most
template <int kMaxLen>
constexpr int zt_max_threads() {
  return 4 * kMaxLen;
}

// the FP32 kernels for extents up to kMaxLen
template <class T, int kMaxLen>
struct Xy {
  static cudaError_t init(int smem);
  static cudaError_t launch(void* D, const XyGeom& g, size_t smem, bool inverse, const DevState* st, cudaStream_t s);
};
template <class T, int kMaxLen>
struct Zt {
  static cudaError_t init(int smem);
  static cudaError_t launch(void* D, const ZtGeom& g, size_t smem, int threads, const void* kfac, const DevState* st,
                            cudaStream_t s);
};

}  // namespace anyfft

namespace longfft {

// plane passes of any extents in two steps a line (k_fft_long.cu)
template <class T>
cudaError_t init(int smem);
template <class T>
cudaError_t launch_xy(void* D, const anyfft::XyGeom& g, size_t smem, bool inverse, const DevState* st, cudaStream_t s);
template <class T>
cudaError_t launch_zt(void* D, const anyfft::ZtGeom& g, size_t smem, const void* kfac, const DevState* st,
                      cudaStream_t s);

}  // namespace longfft

namespace fxfft {

// the FP64 passes of extents up to 32 in block floating point (fft_fx.cuh)
constexpr int kFxThreads = 128;
cudaError_t init(int smem);
cudaError_t launch_xy(void* D, const anyfft::XyGeom& g, size_t smem, int threads, bool inverse, const DevState* st,
                      cudaStream_t s);
cudaError_t launch_zt(void* D, const anyfft::ZtGeom& g, size_t smem, int threads, const double* kfac,
                      int kmax_exponent, const DevState* st, cudaStream_t s);

}  // namespace fxfft
}  // namespace lgf
