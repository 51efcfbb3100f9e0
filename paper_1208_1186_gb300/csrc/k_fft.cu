// Pipeline 1, plane passes of any extents: each pass by the kernel instantiated
// for its extents where there is one (x-y planes of equal extents in
// k_fft_plane.cu, FP32 z-t planes of common extents in k_zt_pairs.cu), else by
// the run-time kernels: a thread per line in fft_any.cuh (FP32) and fft_fx.cuh
// (FP64 lines up to 32), two steps a line in k_fft_long.cu.  The kernel and its
// tiling are chosen here.
#include "fft_any_geom.cuh"
#include "fft_reg.cuh"

namespace lgf {

namespace {

using anyfft::XyGeom;
using anyfft::ZtGeom;

constexpr int kSms = 152;
constexpr size_t kXyTileBytes = 56 * 1024;  // four CTAs share an SM's 227 KB (three with tiles of up to 75 KB in FP64)
constexpr size_t kZtTileBytes = 48 * 1024;

// kernels with a thread per 16 points of a line (k_fft_long.cu): a round of
// 128 threads
constexpr int kLongPoints = 128 * 16;

// As many (plane, field) tiles per CTA as asked for, if four CTAs still fit an SM
// and every SM still gets a CTA.
XyGeom xy_geom(int prec, const int L[4], int tiles, size_t* smem) {
  XyGeom g;
  g.Lx = L[0];
  g.Ly = L[1];
  g.P = L[0] | 1;
  g.N = L[0] * L[1];
  g.V = g.N * L[2] * L[3];
  g.ntiles = 4 * L[2] * L[3];
  g.x = anyfft::make_div(g.Lx);
  const size_t tile = (size_t)g.Ly * g.P * 2 * prec;
  int t = tiles;
  if (t > (int)(kXyTileBytes / tile)) t = (int)(kXyTileBytes / tile);
  if (t > g.ntiles / kSms) t = g.ntiles / kSms;
  g.tpc = t < 1 ? 1 : t;
  *smem = g.tpc * tile;
  return g;
}

// Planes of lines in two steps a line (k_fft_long.cu): lines above 32 in FP64; in
// FP32 where the longer lines are so few that one thread each leaves most of a
// warp idle, and x-y lines above 40.  Steps against lines, us: z-t of 48^3 x 2 23
// and 74, of 9 x 12 x 60 x 16 25 and 16; x-y of 45 x 45 34 and 36, of 60 x 4 18 and
// 21, of 20 x 36 24 and 20; an update of 64 x 64 x 8 x 8 64 and 81, of 48 x 32^3 283
// and 271.
bool xy_in_steps(int prec, int Lx, int Ly) {
  const int m = Lx > Ly ? Lx : Ly, n = Lx < Ly ? Lx : Ly;
  return m > 32 && (prec == 8 || m > 40 || m > 4 * n);
}
bool zt_in_steps(int prec, int Lz, int Lt) {
  const int m = Lz > Lt ? Lz : Lt, n = Lz < Lt ? Lz : Lt;
  return prec == 8 ? m > 32 : m > 6 * n;
}

// 32 bytes of consecutive columns per tile (4 FP32, 2 FP64 complex numbers), or
// more where the z and t lines are short, as long as two CTAs per SM remain.
ZtGeom zt_geom(int prec, const int L[4], size_t* smem, int* threads) {
  ZtGeom g;
  g.Lz = L[2];
  g.Lt = L[3];
  g.S = L[0] * L[1];
  g.V = g.S * L[2] * L[3];
  const int m = g.Lz > g.Lt ? g.Lz : g.Lt, N = g.Lz * g.Lt;
  g.bx = prec == 4 ? 4 : 2;
  auto wants_more = [&] {
    if (!zt_in_steps(prec, g.Lz, g.Lt)) return 2 * g.bx * m <= 128;
    return g.bx * N < kLongPoints && 2 * g.bx * (size_t)N * 2 * prec <= kZtTileBytes;
  };
  while (wants_more() && 4 * ((g.S + 2 * g.bx - 1) / (2 * g.bx)) >= 2 * kSms) g.bx *= 2;
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
  if (e == cudaSuccess) e = anyfft::Xy<float, 40>::init(smem);
  if (e == cudaSuccess) e = fxfft::init(smem);
  if (e == cudaSuccess) e = anyfft::Zt<float, 32>::init(smem);
  if (e == cudaSuccess) e = anyfft::Zt<float, 64>::init(smem);
  if (e == cudaSuccess) e = longfft::init<double>(smem);
  if (e == cudaSuccess) e = longfft::init<float>(smem);
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
  const bool inv = inverse != 0;
  const int m = L[0] > L[1] ? L[0] : L[1];
  if (xy_in_steps(prec, L[0], L[1])) {
    const XyGeom g = xy_geom(prec, L, (kLongPoints + L[0] * L[1] - 1) / (L[0] * L[1]), &sm);
    if (prec == 8) return longfft::launch_xy<double>(D, g, sm, inv, st, s);
    return longfft::launch_xy<float>(D, g, sm, inv, st, s);
  }
  const XyGeom g = xy_geom(prec, L, anyfft::kXyThreads / m, &sm);  // a line for each thread
  if (prec == 8) {
    const int thr = g.tpc * m >= fxfft::kFxThreads ? fxfft::kFxThreads : (g.tpc * m + 31) & ~31;
    return fxfft::launch_xy(D, g, sm, thr, inv, st, s);
  }
  if (m <= 32) return anyfft::Xy<float, 32>::launch(D, g, sm, inv, st, s);
  return anyfft::Xy<float, 40>::launch(D, g, sm, inv, st, s);
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
  const int m = L[2] > L[3] ? L[2] : L[3];
  const ZtGeom g = zt_geom(prec, L, &sm, &thr);
  if (zt_in_steps(prec, L[2], L[3])) {
    if (prec == 8) return longfft::launch_zt<double>(D, g, sm, kfac, st, s);
    return longfft::launch_zt<float>(D, g, sm, kfac, st, s);
  }
  if (prec == 8) return fxfft::launch_zt(D, g, sm, thr, static_cast<const double*>(kfac), kmax_exponent, st, s);
  if (m <= 32) return anyfft::Zt<float, 32>::launch(D, g, sm, thr, kfac, st, s);
  return anyfft::Zt<float, 64>::launch(D, g, sm, thr, kfac, st, s);
}

}  // namespace lgf
