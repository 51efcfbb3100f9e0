// Instances and dispatch of the FP64 passes in block floating point
// (fft_fx.cuh).  Compiled once per part (build.py): 0 the dispatch, 1 and 2 the x-y
// and z-t kernels of all lengths, 3 and 4 those with their extents compiled in.
//
// The code of the latter is small enough to be fetched ahead, where a path
// through the kernel of all lengths is not (z-t of 16^3 x 32: 53 against 72 us,
// 16^4: 20.0 against 22.5; x-y of 32^4: 90 against 97).  Not the z-t planes of
// equal extents from 20 on, whose z and t lines share one function there (32^4:
// 171 us against 220 with two copies).  The list is LGF_ZT_F64 (lgf_kernels.cuh)
// without those; it is not complete: other short pairs would gain as 16 x 32 does,
// at a kernel each.
#include "fft_fx.cuh"

#define LGF_FX_EQUAL_WARP(X) X(4) X(6) X(8) X(10) X(12) X(16)
#define LGF_FX_EQUAL(X) X(20) X(24) X(32)
#define LGF_FX_PAIRS(X) X(4, 4) X(6, 6) X(8, 8) X(12, 12) X(16, 16) X(32, 8) X(32, 16) X(16, 32)

namespace lgf {
namespace fxfft {

struct XyArgs {
  cx<double>* D;
  const anyfft::XyGeom& g;
  size_t smem;
  int threads;
  bool inverse;
  const DevState* st;
  cudaStream_t s;
};
struct ZtArgs {
  cx<double>* D;
  const anyfft::ZtGeom& g;
  size_t smem;
  int threads;
  const double* kfac;
  int kmax_exponent;
  const DevState* st;
  cudaStream_t s;
};
// per part: raise the kernels' shared memory limits, launch one
cudaError_t xy_any_init(int smem);
cudaError_t xy_any(const XyArgs& a);
cudaError_t xy_equal_init(int smem);
bool xy_equal(const XyArgs& a, cudaError_t* e);  // false: no kernel for these extents
cudaError_t zt_any_init(int smem);
cudaError_t zt_any(const ZtArgs& a);
cudaError_t zt_pair_init(int smem);
bool zt_pair(const ZtArgs& a, cudaError_t* e);

#if LGF_FX_PART == 0

cudaError_t init(int smem) {
  smem -= 1024;  // the kernels' own shared variables
  cudaError_t e = xy_any_init(smem);
  if (e == cudaSuccess) e = xy_equal_init(smem);
  if (e == cudaSuccess) e = zt_any_init(smem);
  if (e == cudaSuccess) e = zt_pair_init(smem);
  return e;
}

cudaError_t launch_xy(void* D, const anyfft::XyGeom& g, size_t smem, int threads, bool inverse, const DevState* st,
                      cudaStream_t s) {
  const XyArgs a{static_cast<cx<double>*>(D), g, smem, threads, inverse, st, s};
  cudaError_t e = cudaSuccess;
  return g.Lx == g.Ly && xy_equal(a, &e) ? e : xy_any(a);
}

cudaError_t launch_zt(void* D, const anyfft::ZtGeom& g, size_t smem, int threads, const double* kfac,
                      int kmax_exponent, const DevState* st, cudaStream_t s) {
  const ZtArgs a{static_cast<cx<double>*>(D), g, smem, threads, kfac, kmax_exponent, st, s};
  cudaError_t e = cudaSuccess;
  return zt_pair(a, &e) ? e : zt_any(a);
}

#elif LGF_FX_PART == 2

cudaError_t zt_any_init(int smem) {
  return cudaFuncSetAttribute(k_fx_zt<>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}
cudaError_t zt_any(const ZtArgs& a) {
  const dim3 grid((unsigned)((a.g.S + a.g.bx - 1) / a.g.bx), 4);
  return launch_pdl(k_fx_zt<>, grid, a.threads, a.smem, a.s, a.D, a.g, a.kfac, a.kmax_exponent, a.st);
}

#elif LGF_FX_PART == 4

cudaError_t zt_pair_init(int smem) {
  cudaError_t e = cudaSuccess;
#define LGF_CASE(A, B)  \
  if (e == cudaSuccess) \
    e = cudaFuncSetAttribute(k_fx_zt<A, B>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  LGF_FX_PAIRS(LGF_CASE)
#undef LGF_CASE
  return e;
}
bool zt_pair(const ZtArgs& a, cudaError_t* e) {
  const dim3 grid((unsigned)((a.g.S + a.g.bx - 1) / a.g.bx), 4);
#define LGF_CASE(A, B)                                                                                              \
  if (a.g.Lz == A && a.g.Lt == B) {                                                                                 \
    *e = launch_pdl(k_fx_zt<A, B>, grid, a.threads, a.smem, a.s, a.D, a.g, a.kfac, a.kmax_exponent, a.st);          \
    return true;                                                                                                    \
  }
  LGF_FX_PAIRS(LGF_CASE)
#undef LGF_CASE
  return false;
}

#else  // parts 1 and 3: x-y

template <int N>
static cudaError_t xy_init(int smem) {
  const cudaError_t e =
      cudaFuncSetAttribute(k_fx_xy<false, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return e != cudaSuccess ? e
                          : cudaFuncSetAttribute(k_fx_xy<true, N>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

template <int N>
static cudaError_t xy_launch(const XyArgs& a) {
  const unsigned nb = (unsigned)((a.g.ntiles + a.g.tpc - 1) / a.g.tpc);
  if (a.inverse) return launch_pdl(k_fx_xy<true, N>, nb, a.threads, a.smem, a.s, a.D, a.g, a.st);
  return launch_pdl(k_fx_xy<false, N>, nb, a.threads, a.smem, a.s, a.D, a.g, a.st);
}

#if LGF_FX_PART == 1

cudaError_t xy_any_init(int smem) { return xy_init<0>(smem); }
cudaError_t xy_any(const XyArgs& a) { return xy_launch<0>(a); }

#else

namespace {

// x-y planes of equal small extents: as k_plane_xy_warp, L lanes own a tile from
// load to store, lines in registers, the tile's exponent agreed by shuffles.
// Small lattices are bound by the latency of the phases, of which k_fx_xy has
// more (8^4: 8.6 against 10.4 us, 16^4: 12.6 against 16.6); from 20 on the
// unrolled code is the longer wait (32^4: 128 against 97).
template <int L>
__device__ __forceinline__ int registers_sum(const cx<I> (&v)[L]) {
  int m = 0;
#pragma unroll
  for (int p = 0; p < L; ++p) m += size_of(v[p].re) + size_of(v[p].im);
  return m;
}

template <int L, bool INV>
__global__ void __launch_bounds__(32) k_fx_xy_warp(cx<double>* __restrict__ D, int V, int ntiles,
                                                   const DevState* __restrict__ st) {
  pdl_wait();
  if (st != nullptr && st->done) return;
  constexpr int G = 32 / L, P = L + 1, N = L * L;
  __shared__ cx<I> tiles[G * L * P];
  const int g = threadIdx.x / L, r = threadIdx.x % L;
  const int tile_id = blockIdx.x * G + g;  // = 4 plane + field
  const bool active = g < G && tile_id < ntiles;
  // the lanes of this tile (the lanes past the last whole group: one another)
  const unsigned mask = g < G ? ((1u << L) - 1u) << (g * L) : ~0u << ((G * L) & 31);
  cx<I>* tile = tiles + (active ? g : 0) * L * P;
  cx<double>* src = D + (active ? (tile_id & 3) * V + (tile_id >> 2) * N : 0);
  cx<I> v[L];
  int E = 0;
  if (active) {
#pragma unroll
    for (int p = 0; p < L; ++p) {
      const longlong2 b = bits_at(src + p * L + r);
      v[p] = mk<I>(I::from(b.x), I::from(b.y));
      E = max(E, max(exponent(b.x), exponent(b.y)));
    }
  }
  E = __reduce_max_sync(mask, E);
  int m = 0;
  if (active) {
#pragma unroll
    for (int p = 0; p < L; ++p) m += size_of_bits(v[p].re.v, E) + size_of_bits(v[p].im.v, E);
  }
  const int s0 = shift_for(__reduce_max_sync(mask, m), 43);
  if (active) {  // y-line r, transformed, into column r
#pragma unroll
    for (int p = 0; p < L; ++p)
      v[p] = mk<I>(I::from(from_bits(v[p].re.v, E, s0)), I::from(from_bits(v[p].im.v, E, s0)));
    if (INV)
      regfft::inverse<I, L>(v);
    else
      regfft::forward<I, L>(v);
#pragma unroll
    for (int p = 0; p < L; ++p) tile[p * P + r] = v[p];
  }
  __syncwarp();
  m = 0;
  if (active) {  // x-line r from row r
#pragma unroll
    for (int p = 0; p < L; ++p) v[p] = tile[r * P + p];
    m = registers_sum<L>(v);
  }
  const int s1 = shift_for(__reduce_max_sync(mask, m), 44);
  if (active) {
    const long long half = (1ll << s1) >> 1;
#pragma unroll
    for (int p = 0; p < L; ++p) v[p] = mk<I>(shifted(v[p].re, s1, half), shifted(v[p].im, s1, half));
    if (INV)
      regfft::inverse<I, L>(v);
    else
      regfft::forward<I, L>(v);
    cx<double>* row = reinterpret_cast<cx<double>*>(tile) + r * P;
    const int X = E - 1022 - 61 + s0 + s1;
#pragma unroll
    for (int p = 0; p < L; ++p) row[p] = out(v[p], X, E == 0x7ff);
  }
  __syncwarp();
  if (active) {
    const cx<double>* o = reinterpret_cast<const cx<double>*>(tile);
#pragma unroll
    for (int k = 0; k < L; ++k) src[k * L + r] = o[k * P + r];
  }
}

template <int L>
cudaError_t warp_launch(const XyArgs& a) {
  const unsigned nb = (unsigned)((a.g.ntiles + 32 / L - 1) / (32 / L));
  if (a.inverse) return launch_pdl(k_fx_xy_warp<L, true>, nb, 32, 0, a.s, a.D, a.g.V, a.g.ntiles, a.st);
  return launch_pdl(k_fx_xy_warp<L, false>, nb, 32, 0, a.s, a.D, a.g.V, a.g.ntiles, a.st);
}

}  // namespace

cudaError_t xy_equal_init(int smem) {
  cudaError_t e = cudaSuccess;
#define LGF_CASE(N) \
  if (e == cudaSuccess) e = xy_init<N>(smem);
  LGF_FX_EQUAL(LGF_CASE)
#undef LGF_CASE
  return e;
}
bool xy_equal(const XyArgs& a, cudaError_t* e) {
  switch (a.g.Lx) {
#define LGF_CASE(N) \
  case N: *e = warp_launch<N>(a); return true;
    LGF_FX_EQUAL_WARP(LGF_CASE)
#undef LGF_CASE
#define LGF_CASE(N) \
  case N: *e = xy_launch<N>(a); return true;
    LGF_FX_EQUAL(LGF_CASE)
#undef LGF_CASE
    default: return false;
  }
}

#endif
#endif

}  // namespace fxfft
}  // namespace lgf
