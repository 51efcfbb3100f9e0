// Pipeline 1, plane passes of any extents: each pass by the kernel instantiated
// for its extents where there is one (x-y planes of equal extents in
// k_fft_plane.cu, FP32 z-t planes of common extents in k_zt_pairs.cu), else by
// the run-time kernels of fft_any.cuh, whose tiling is chosen here.
#include "fft_any_geom.cuh"
#include "fft_reg.cuh"

namespace lgf {

namespace {

using anyfft::XyGeom;
using anyfft::ZtGeom;

constexpr int kSms = 152;
constexpr size_t kXyTileBytes = 56 * 1024;  // four CTAs share an SM's 227 KB (three with tiles of up to 75 KB in FP64)

// As many (plane, field) tiles per CTA as give its 128 threads a line each, if
// four CTAs still fit an SM and every SM still gets a CTA.
XyGeom xy_geom(int prec, const int L[4], size_t* smem) {
  XyGeom g;
  g.Lx = L[0];
  g.Ly = L[1];
  g.P = L[0] | 1;
  g.N = L[0] * L[1];
  g.V = g.N * L[2] * L[3];
  g.ntiles = 4 * L[2] * L[3];
  g.x = anyfft::make_div(g.Lx);
  const size_t tile = (size_t)g.Ly * g.P * 2 * prec;
  int t = anyfft::kXyThreads / (g.Lx > g.Ly ? g.Lx : g.Ly);
  if (t > (int)(kXyTileBytes / tile)) t = (int)(kXyTileBytes / tile);
  if (t > g.ntiles / kSms) t = g.ntiles / kSms;
  g.tpc = t < 1 ? 1 : t;
  *smem = g.tpc * tile;
  return g;
}

// 32 bytes of consecutive columns per tile (4 FP32, 2 FP64 complex numbers), or
// more where the z and t lines are short, as long as two CTAs per SM remain.
ZtGeom zt_geom(int prec, const int L[4], size_t* smem, int* threads) {
  ZtGeom g;
  g.Lz = L[2];
  g.Lt = L[3];
  g.S = L[0] * L[1];
  g.V = g.S * L[2] * L[3];
  const int m = g.Lz > g.Lt ? g.Lz : g.Lt;
  g.bx = prec == 4 ? 4 : 2;
  while (2 * g.bx * m <= 128 && 4 * ((g.S + 2 * g.bx - 1) / (2 * g.bx)) >= 2 * kSms) g.bx *= 2;
  g.lbx = 0;
  while ((1 << g.lbx) < g.bx) ++g.lbx;
  // consecutive t slices shift by one run of columns across the banks
  const int words = 2 * prec / 4;
  g.PT = g.bx * g.Lz;
  while ((g.PT * words) % 32 != (g.bx * words) % 32) ++g.PT;
  *smem = (size_t)g.PT * g.Lt * 2 * prec;
  *threads = (g.bx * m + 31) & ~31;
  return g;
}

// the acceleration factor of every site, formed in FP64, in the positions the
// forward passes leave the modes (an FP64 division per mode and iteration would
// cost more than reading it)
template <class T>
__global__ void __launch_bounds__(256) k_kfac(const double* __restrict__ s2, double p2max, T* __restrict__ kfac, int Lx,
                                              int Ly, int Lz, int V) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= V) return;
  const int x = s % Lx, r = s / Lx, y = r % Ly, zt = r / Ly, z = zt % Lz, t = zt / Lz;
  const double p2 = s2[x] + s2[kMaxL + y] + s2[2 * kMaxL + z] + s2[3 * kMaxL + t];
  kfac[s] = s ? (T)(p2max / (p2 * (double)V)) : (T)0;
}

}  // namespace

cudaError_t launch_kfac(int prec, const int L[4], const double* s2, double p2max, void* kfac, cudaStream_t s) {
  const int V = L[0] * L[1] * L[2] * L[3];
  const unsigned nb = (unsigned)((V + 255) / 256);
  if (prec == 8)
    k_kfac<<<nb, 256, 0, s>>>(s2, p2max, static_cast<double*>(kfac), L[0], L[1], L[2], V);
  else
    k_kfac<<<nb, 256, 0, s>>>(s2, p2max, static_cast<float*>(kfac), L[0], L[1], L[2], V);
  return cudaPeekAtLastError();
}

bool zt_pair_supported(int prec, int Lz, int Lt) {
  if (prec != 4) return false;
  bool z = false, t = false;
#define LGF_IS(N)     \
  z = z || Lz == N;   \
  t = t || Lt == N;
  LGF_PAIR_EXTENTS(LGF_IS)
#undef LGF_IS
  return z && t;
}

bool extents_supported(const int L[4], int prec, size_t smem_limit) {
  for (int a = 0; a < 4; ++a)
    if (L[a] < 2 || L[a] > kMaxL || !regfft::supported(L[a])) return false;
  // the range of planes this library has always taken: two copies of an x-y
  // plane and of a z-t plane of bx columns (with the factor beside it) in one
  // CTA's shared memory
  int bx = prec == 8 ? 2 : 4;
  while (L[0] % bx != 0) bx /= 2;
  const size_t c = 2 * (size_t)prec, tile = (size_t)bx * (L[2] + 1) * L[3];
  return (2 * (size_t)(L[0] + 1) * L[1] + 2 * kMaxL) * c <= smem_limit &&
         (2 * tile + 4 * kMaxL) * c + tile * prec <= smem_limit;
}

cudaError_t fft_any_init(int smem) {
  cudaError_t e = anyfft::Xy<float, 32>::init(smem);
  if (e == cudaSuccess) e = anyfft::Xy<float, 64>::init(smem);
  if (e == cudaSuccess) e = fxfft::init(smem);
  if (e == cudaSuccess) e = anyfft::Xy<double, 64>::init(smem);
  if (e == cudaSuccess) e = anyfft::Zt<float, 32>::init(smem);
  if (e == cudaSuccess) e = anyfft::Zt<float, 64>::init(smem);
  if (e == cudaSuccess) e = anyfft::Zt<double, 64>::init(smem);
  return e;
}

cudaError_t zt_pair_init(int Lz, int Lt) {
  switch (Lz) {
#define LGF_CASE(N) \
  case N: return zt_pair_init<N>(Lt);
    LGF_PAIR_EXTENTS(LGF_CASE)
#undef LGF_CASE
    default: return cudaSuccess;
  }
}

cudaError_t launch_fft_xy(int prec, const int L[4], void* D, int inverse, const DevState* st, cudaStream_t s) {
  if (prec == 4 && plane_xy_supported(L[0], L[1]))
    return launch_plane_xy(L[0], D, (int64_t)L[0] * L[1] * L[2] * L[3], L[2], L[3], inverse, st, s);
  size_t sm = 0;
  const XyGeom g = xy_geom(prec, L, &sm);
  const int m = g.Lx > g.Ly ? g.Lx : g.Ly;
  const bool inv = inverse != 0;
  if (prec == 8) {
    const int thr = g.tpc * m >= fxfft::kFxThreads ? fxfft::kFxThreads : (g.tpc * m + 31) & ~31;
    if (m <= 32) return fxfft::launch_xy(D, g, sm, thr, inv, st, s);
    return anyfft::Xy<double, 64>::launch(D, g, sm, inv, st, s);
  }
  if (m <= 32) return anyfft::Xy<float, 32>::launch(D, g, sm, inv, st, s);
  return anyfft::Xy<float, 64>::launch(D, g, sm, inv, st, s);
}

cudaError_t launch_fft_zt(int prec, const int L[4], void* D, const void* kfac, int kmax_exponent, const DevState* st,
                          cudaStream_t s) {
  if (zt_pair_supported(prec, L[2], L[3])) {
    switch (L[2]) {
#define LGF_CASE(N) \
  case N: return launch_zt_pair<N>(L[3], D, L[0], L[1], static_cast<const float*>(kfac), st, s);
      LGF_PAIR_EXTENTS(LGF_CASE)
#undef LGF_CASE
    }
  }
  size_t sm = 0;
  int thr = 0;
  const ZtGeom g = zt_geom(prec, L, &sm, &thr);
  const int m = g.Lz > g.Lt ? g.Lz : g.Lt;
  if (prec == 8) {
    if (m <= 32)
      return fxfft::launch_zt(D, g, sm, thr, static_cast<const double*>(kfac), kmax_exponent, st, s);
    return anyfft::Zt<double, 64>::launch(D, g, sm, thr, kfac, st, s);
  }
  if (m <= 32) return anyfft::Zt<float, 32>::launch(D, g, sm, thr, kfac, st, s);
  return anyfft::Zt<float, 64>::launch(D, g, sm, thr, kfac, st, s);
}

}  // namespace lgf
