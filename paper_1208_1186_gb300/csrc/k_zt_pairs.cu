// z-t plane kernels (zt_plane.cuh) for every pair of common extents, for the
// shapes that have no tuned instance in k_fft_zt.cu.  One kernel per pair, not
// one kernel that picks its line lengths at run time: at the same instruction
// count and occupancy the latter spent twice the time (24^3 x 48: 33 against 18
// us), waiting for instructions (4.6 cycles per issue against 0.7, ncu) -- a
// kernel of 27 KB of straight-line code is fetched ahead, a path through one of
// many hundred KB is not.  The price is code: 225 kernels make 71 MB of objects (the
// library is 102 MB) and 5 of the 14 CPU minutes of its build.  FP32 only: FP64 planes run
// in 64-bit block floating point (k_fft_fx.cu) or in two steps a line
// (k_fft_long.cu).  Compiled once per z extent (build.py).
#include "zt_plane.cuh"

namespace lgf {

namespace {

// 32 bytes of consecutive columns per run, 64 where both lines are short
constexpr int pair_bx(int m) { return m <= 8 ? 8 : 4; }

template <int LZ, int LT>
cudaError_t pair_init() {
  constexpr int BX = pair_bx(LZ > LT ? LZ : LT);
  constexpr size_t sm = zt_smem_bytes<float, LZ, LT, BX>();
  if constexpr (sm > 48 * 1024)
    return cudaFuncSetAttribute(k_plane_zt<LZ, LT, BX, 0, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
  return cudaSuccess;
}

template <int LZ, int LT>
cudaError_t pair_launch(void* D, int Lx, int Ly, const float* kfac, const DevState* st, cudaStream_t s) {
  constexpr int BX = pair_bx(LZ > LT ? LZ : LT);
  constexpr size_t sm = zt_smem_bytes<float, LZ, LT, BX>();
  dim3 grid((unsigned)((Lx * Ly + BX - 1) / BX), 4);
  return launch_pdl(k_plane_zt<LZ, LT, BX, 0, true>, grid, zt_threads<LZ, LT, BX>(), sm, s,
                    static_cast<cx<float>*>(D), Lx, Ly, nullptr, 0.f, kfac, st);
}

}  // namespace

template <int LZ>
cudaError_t zt_pair_init(int Lt) {
  switch (Lt) {
#define LGF_CASE(LT) \
  case LT: return pair_init<LZ, LT>();
    LGF_PAIR_EXTENTS(LGF_CASE)
#undef LGF_CASE
    default: return cudaSuccess;
  }
}

template <int LZ>
cudaError_t launch_zt_pair(int Lt, void* D, int Lx, int Ly, const float* kfac, const DevState* st, cudaStream_t s) {
  switch (Lt) {
#define LGF_CASE(LT) \
  case LT: return pair_launch<LZ, LT>(D, Lx, Ly, kfac, st, s);
    LGF_PAIR_EXTENTS(LGF_CASE)
#undef LGF_CASE
    default: return cudaErrorInvalidValue;
  }
}

template cudaError_t zt_pair_init<LGF_PAIR_Z>(int);
template cudaError_t launch_zt_pair<LGF_PAIR_Z>(int, void*, int, int, const float*, const DevState*, cudaStream_t);

}  // namespace lgf
