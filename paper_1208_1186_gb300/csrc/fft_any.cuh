// FP32 plane passes of any accepted extents (products of 2, 3 and 5 up to 64) with
// in-register line FFTs (fft_reg.cuh), for the shapes that have no kernel of their
// own (k_fft.cu chooses):
//
//   k_any_xy(fwd) -> k_any_zt (fwd z, fwd t, x p2_max/(V p2), inv t, inv z)
//   -> k_any_xy(inv)
//
// the paper's "2D plus 2D" split (Sec. 2.2).  The extents are run-time values, and
// each line's transform, whose length is a template constant, is picked by a
// switch that is uniform over the CTA.  Only the index arithmetic is run-time; it
// goes by multiply-high reciprocals.
//
// Staged butterflies in shared memory with run-time radices, strides and
// divisions took 170 us per acceleration of 20 x 30 x 18 x 40, now 45 (its z-t
// plane by k_zt_pairs.cu).
#pragma once

#include "fft_any_geom.cuh"
#include "fft_reg.cuh"

namespace lgf {
namespace anyfft {

#define LGF_LINE_LENGTHS(X) \
  X(2) X(3) X(4) X(5) X(6) X(8) X(9) X(10) X(12) X(15) X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32) \
  X(36) X(40) X(45) X(48) X(50) X(54) X(60) X(64)

// f(std::integral_constant<int, L>) for the line length L <= kMaxLen
template <int kMaxLen, class F>
__device__ __forceinline__ void with_length(int L, F&& f) {
  switch (L) {
#define LGF_CASE(N)                                                            \
  case N:                                                                      \
    if constexpr (N <= kMaxLen) f(std::integral_constant<int, N>{});           \
    break;
    LGF_LINE_LENGTHS(LGF_CASE)
#undef LGF_CASE
  }
}

// The line transforms are functions of their own, called from the switch:
// inlined, all lengths shared one register allocation with spills, and the x-y
// pass of 20 x 30 x 18 x 40 took 16.3 instead of 14.4 us.
template <int L, class T, bool INV>
__device__ __noinline__ void y_line(const cx<T>* src, int pitch, cx<T>* col, int P) {
  cx<T> v[L];
#pragma unroll
  for (int i = 0; i < L; ++i) {
    v[i] = *src;
    src += pitch;
  }
  if (INV)
    regfft::inverse<T, L>(v);
  else
    regfft::forward<T, L>(v);
#pragma unroll
  for (int i = 0; i < L; ++i) {
    *col = v[i];
    col += P;
  }
}

template <int L, class T, bool INV>
__device__ __noinline__ void x_line(cx<T>* row) {
  cx<T> v[L];
#pragma unroll
  for (int i = 0; i < L; ++i) v[i] = row[i];
  if (INV)
    regfft::inverse<T, L>(v);
  else
    regfft::forward<T, L>(v);
#pragma unroll
  for (int i = 0; i < L; ++i) row[i] = v[i];
}

// forward t, times the acceleration factor (the table at kl, step apart),
// inverse t
template <int L, class T>
__device__ __noinline__ void t_line(cx<T>* line, int PT, const T* kl, int step) {
  T k[L];  // loaded before the transform
#pragma unroll
  for (int i = 0; i < L; ++i) {
    k[i] = __ldg(kl);
    kl += step;
  }
  cx<T> v[L];
  cx<T>* p = line;
#pragma unroll
  for (int i = 0; i < L; ++i) {
    v[i] = *p;
    p += PT;
  }
  regfft::forward<T, L>(v);
#pragma unroll
  for (int i = 0; i < L; ++i) v[i] = scale(v[i], k[i]);
  regfft::inverse<T, L>(v);
  p = line;
#pragma unroll
  for (int i = 0; i < L; ++i) {
    *p = v[i];
    p += PT;
  }
}

template <int L, class T>
__device__ __noinline__ void z_line_out(const cx<T>* line, int bx, cx<T>* dst, int pitch) {
  cx<T> v[L];
#pragma unroll
  for (int i = 0; i < L; ++i) {
    v[i] = *line;
    line += bx;
  }
  regfft::inverse<T, L>(v);
#pragma unroll
  for (int i = 0; i < L; ++i) {
    *dst = v[i];
    dst += pitch;
  }
}

// lines of kMaxLen complex numbers: as many CTAs as their registers leave
template <int kMaxLen>
constexpr int xy_min_blocks() {
  return kMaxLen <= 32 ? 4 : 2;
}

// tpc tiles (one field of one (z, t) plane each: tile = 4 plane + field) per
// CTA.  One thread per y-line loads it straight into registers (for each y the
// threads of a tile read one contiguous row), transforms it and hands the
// x-lines through shared memory to one thread each; the rows then leave
// shared memory as they came.  (The two 1D transforms commute.)  The row pitch
// is odd, so no phase has bank conflicts.
template <class T, bool INV, int kMaxLen>
__global__ void __launch_bounds__(kXyThreads, (xy_min_blocks<kMaxLen>()))
    k_any_xy(cx<T>* __restrict__ D, const XyGeom g, const DevState* __restrict__ st) {
  pdl_wait();
  if (st != nullptr && st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* tiles = reinterpret_cast<cx<T>*>(smem_raw);  // [tile][y][x], row pitch P
  const int t0 = blockIdx.x * g.tpc;
  const int nt = g.ntiles - t0 < g.tpc ? g.ntiles - t0 : g.tpc;
  for (int l = threadIdx.x; l < nt * g.Lx; l += kXyThreads) {
    const int j = quot(l, g.x), x = l - j * g.Lx, tile = t0 + j;
    const cx<T>* src = D + ((tile & 3) * g.V + (tile >> 2) * g.N + x);
    cx<T>* col = tiles + j * g.Ly * g.P + x;
    with_length<kMaxLen>(g.Ly, [&](auto n) { y_line<decltype(n)::value, T, INV>(src, g.Lx, col, g.P); });
  }
  __syncthreads();
  for (int l = threadIdx.x; l < nt * g.Ly; l += kXyThreads)
    with_length<kMaxLen>(g.Lx, [&](auto n) { x_line<decltype(n)::value, T, INV>(tiles + l * g.P); });
  __syncthreads();
  for (int l = threadIdx.x; l < nt * g.Lx; l += kXyThreads) {
    const int j = quot(l, g.x), x = l - j * g.Lx, tile = t0 + j;
    cx<T>* dst = D + ((tile & 3) * g.V + (tile >> 2) * g.N + x);
    const cx<T>* col = tiles + j * g.Ly * g.P + x;
#pragma unroll 4
    for (int i = 0; i < g.Ly; ++i) dst[i * g.Lx] = col[i * g.P];
  }
}

template <int kMaxLen>
constexpr int zt_min_blocks() {
  return kMaxLen <= 32 ? 3 : 1;
}

// One CTA per field and run of bx consecutive (x, y) columns, whatever Lx: the
// columns of a (z, t) site are contiguous, and a run may cross from one y to
// the next.  z lines come from global memory into registers, go to the t lines
// through shared memory, and are stored from registers after the inverse.
// The factor comes from the per-site table kfac.
template <class T, int kMaxLen>
__global__ void __launch_bounds__((zt_max_threads<kMaxLen>()), (zt_min_blocks<kMaxLen>()))
    k_any_zt(cx<T>* __restrict__ D, const ZtGeom g, const T* __restrict__ kfac, const DevState* __restrict__ st) {
  pdl_wait();
  if (st != nullptr && st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* tile = reinterpret_cast<cx<T>*>(smem_raw);  // [t][z][column], t pitch PT
  const int q0 = blockIdx.x * g.bx;
  const int xb = threadIdx.x & (g.bx - 1), row = threadIdx.x >> g.lbx;
  const int q = q0 + xb;
  const bool inside = q < g.S;
  cx<T>* Dq = D + (blockIdx.y * g.V + q);
  if (inside && row < g.Lt)  // forward z of line (column, t = row)
    with_length<kMaxLen>(g.Lz, [&](auto n) {
      y_line<decltype(n)::value, T, false>(Dq + g.S * g.Lz * row, g.S, tile + row * g.PT + xb, g.bx);
    });
  __syncthreads();
  if (inside && row < g.Lz)  // t line (column, z = row): forward, factor, inverse
    with_length<kMaxLen>(g.Lt, [&](auto n) {
      t_line<decltype(n)::value, T>(tile + row * g.bx + xb, g.PT, kfac + (q + g.S * row), g.S * g.Lz);
    });
  __syncthreads();
  if (inside && row < g.Lt)  // inverse z, to global memory
    with_length<kMaxLen>(g.Lz, [&](auto n) {
      z_line_out<decltype(n)::value, T>(tile + row * g.PT + xb, g.bx, Dq + g.S * g.Lz * row, g.S);
    });
}

// shared memory beyond 48 KB has to be allowed per kernel (once per device, at
// handle creation)
template <class T, int kMaxLen>
cudaError_t Xy<T, kMaxLen>::init(int smem) {
  const cudaError_t e =
      cudaFuncSetAttribute(k_any_xy<T, false, kMaxLen>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return e != cudaSuccess ? e
                          : cudaFuncSetAttribute(k_any_xy<T, true, kMaxLen>,
                                                 cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

template <class T, int kMaxLen>
cudaError_t Xy<T, kMaxLen>::launch(void* D, const XyGeom& g, size_t smem, bool inverse, const DevState* st,
                                   cudaStream_t s) {
  const unsigned nb = (unsigned)((g.ntiles + g.tpc - 1) / g.tpc);
  const auto d = static_cast<cx<T>*>(D);
  if (inverse) return launch_pdl(k_any_xy<T, true, kMaxLen>, nb, kXyThreads, smem, s, d, g, st);
  return launch_pdl(k_any_xy<T, false, kMaxLen>, nb, kXyThreads, smem, s, d, g, st);
}

template <class T, int kMaxLen>
cudaError_t Zt<T, kMaxLen>::init(int smem) {
  return cudaFuncSetAttribute(k_any_zt<T, kMaxLen>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
}

template <class T, int kMaxLen>
cudaError_t Zt<T, kMaxLen>::launch(void* D, const ZtGeom& g, size_t smem, int threads, const void* kfac,
                                   const DevState* st, cudaStream_t s) {
  const dim3 grid((unsigned)((g.S + g.bx - 1) / g.bx), 4);
  return launch_pdl(k_any_zt<T, kMaxLen>, grid, threads, smem, s, static_cast<cx<T>*>(D), g,
                    static_cast<const T*>(kfac), st);
}

}  // namespace anyfft
}  // namespace lgf
