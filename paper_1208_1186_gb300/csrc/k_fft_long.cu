// Plane passes for planes of long or of few lines (pipeline 1; k_fft.cu draws the
// line): each line in two steps of at most 16 points through shared memory.
//
// A line of L = A B points is A-point transforms at stride B, twiddles, and
// B-point transforms of the A blocks, every one of them a thread's: a plane of
// few long lines (48^3 x 2: two z lines a column) still fills its warps, which
// bounds an FP64 pass, because the FP64 pipe serves a warp in the same time
// however few of its lanes have work.  A and B split the radix sequence of
// regfft's transform of L, so that the frequencies come to rest at the same
// positions (digit_rev) as anywhere else.
//
// In FP64 a line of up to 64 complex numbers in one thread's registers spilled, and
// lanes without a line idled.  us by line -> in two steps (in brackets: radix-4, 2, 3,
// 5 stages in shared memory, which ran before both): z-t pass of 48^3 x 2 829 -> 81
// (124), 36^3 x 6 407 -> 146 (209), 48^3 x 8 929 -> 358 (498); both x-y passes of
// 48^3 x 8 776 -> 499 (683), 2 x 64 x 15 x 54 466 -> 63 (61), 64 x 2 x 2 x 2 82 -> 27
// (21).
#include "fft_any_geom.cuh"
#include "fft_reg.cuh"

namespace lgf {
namespace longfft {

namespace {

constexpr int kThreads = 128;

// L = a b: the split of L's radix sequence with the shortest longer part
constexpr int split_a(int L) {
  int best = L, a = 1, rem = L;
  while (rem > 1) {
    const int r = regfft::next_radix(rem);
    a *= r;
    rem /= r;
    const int m = a > rem ? a : rem, bm = best > L / best ? best : L / best;
    if (m < bm) best = a;
  }
  return best;
}

template <int L>
struct Shape {
  static constexpr int A = L <= 16 ? L : split_a(L), B = L / A;
  static_assert(A <= 16 && B <= 16, "a step fits a thread's registers");
};

// W_L^m, m < L
template <class T, int L>
struct Twiddles {
  T v[2 * L];
  constexpr Twiddles() : v{} {
    for (int m = 0; m < L; ++m) {
      v[2 * m] = (T)regfft::turn_cs(m, L, 0);
      v[2 * m + 1] = (T)-regfft::turn_cs(m, L, 1);
    }
  }
};
template <class T, int L>
__device__ const Twiddles<T, L> kTwiddles{};

template <class T, int L>
__device__ __forceinline__ cx<T> twiddle(int m) {
  if constexpr (sizeof(T) == 8) {
    const double2 w = __ldg(reinterpret_cast<const double2*>(kTwiddles<T, L>.v) + m);
    return mk<T>(w.x, w.y);
  } else {
    const float2 w = __ldg(reinterpret_cast<const float2*>(kTwiddles<T, L>.v) + m);
    return mk<T>(w.x, w.y);
  }
}

// n lines in shared memory: line l starts at (l % na) sa + (l / na) sb, its
// elements are es apart
template <class T>
struct Lines {
  cx<T>* p;
  int n, na, sa, sb, es;
  __device__ __forceinline__ cx<T>* at(int l) const {
    const int o = (unsigned)l / (unsigned)na;
    return p + (l - o * na) * sa + o * sb;
  }
};

// the A-point step: a thread per (line, b), forward with its twiddles after it,
// inverse with their conjugates before it
template <class T, int L, bool INV>
__device__ __forceinline__ void step_a(const Lines<T>& ln) {
  constexpr int A = Shape<L>::A, B = Shape<L>::B;
  for (int w = threadIdx.x; w < ln.n * B; w += blockDim.x) {
    const int b = (unsigned)w / (unsigned)ln.n;
    cx<T>* p = ln.at(w - b * ln.n) + b * ln.es;
    const int es = B * ln.es;
    cx<T> v[A];
#pragma unroll
    for (int a = 0; a < A; ++a) v[a] = p[a * es];
    if constexpr (INV) {
      if constexpr (B > 1) {
        regfft::static_for<1, A>([&](auto ac) {
          constexpr int a = decltype(ac)::value;
          v[a] = mul_cj(v[a], twiddle<T, L>(b * regfft::digit_rev(A, a)));
        });
      }
      regfft::inverse<T, A>(v);
    } else {
      regfft::forward<T, A>(v);
      if constexpr (B > 1) {
        regfft::static_for<1, A>([&](auto ac) {
          constexpr int a = decltype(ac)::value;
          v[a] = v[a] * twiddle<T, L>(b * regfft::digit_rev(A, a));
        });
      }
    }
#pragma unroll
    for (int a = 0; a < A; ++a) p[a * es] = v[a];
  }
}

// the B-point step: a thread per (line, block), forward or inverse, or (MID)
// forward, times k at positions ks apart from each line's first, and inverse
enum Mode { kForward, kInverse, kMid };
template <class T, int L, Mode M, class K>
__device__ __forceinline__ void step_b(const Lines<T>& ln, const K& k, int ks) {
  constexpr int A = Shape<L>::A, B = Shape<L>::B;
  if constexpr (B > 1 || M == kMid) {
    for (int w = threadIdx.x; w < ln.n * A; w += blockDim.x) {
      const int a = (unsigned)w / (unsigned)ln.n, l = w - a * ln.n;
      cx<T>* p = ln.at(l) + a * B * ln.es;
      cx<T> v[B];
#pragma unroll
      for (int b = 0; b < B; ++b) v[b] = p[b * ln.es];
      if constexpr (M != kInverse && B > 1) regfft::forward<T, B>(v);
      if constexpr (M == kMid) {
        const T* f = k(l) + a * B * ks;
#pragma unroll
        for (int b = 0; b < B; ++b) v[b] = scale(v[b], __ldg(f + b * ks));
      }
      if constexpr (M != kForward && B > 1) regfft::inverse<T, B>(v);
#pragma unroll
      for (int b = 0; b < B; ++b) p[b * ln.es] = v[b];
    }
  }
}

template <class T, int L, bool INV>
__device__ __noinline__ void transform(const Lines<T> ln) {
  auto none = [](int) { return (const T*)nullptr; };
  if constexpr (INV) {
    step_b<T, L, kInverse>(ln, none, 0);
    if (Shape<L>::B > 1) __syncthreads();
    step_a<T, L, true>(ln);
  } else {
    step_a<T, L, false>(ln);
    if (Shape<L>::B > 1) __syncthreads();
    step_b<T, L, kForward>(ln, none, 0);
  }
}

// forward, times the table, inverse; line l is column l % bx (of nx) at z = l / bx
template <class T, int L>
__device__ __noinline__ void accelerate(const Lines<T> ln, const T* kfac, int S, int nx, int bx, int lbx, int ks) {
  step_a<T, L, false>(ln);
  __syncthreads();
  auto k = [&](int l) {
    const int xb = l & (bx - 1);
    return kfac + (xb < nx ? xb : nx - 1) + S * (l >> lbx);
  };
  step_b<T, L, kMid>(ln, k, ks);
  __syncthreads();
  step_a<T, L, true>(ln);
}

#define LGF_LONG_LENGTHS(X) \
  X(2) X(3) X(4) X(5) X(6) X(8) X(9) X(10) X(12) X(15) X(16) X(18) X(20) X(24) X(25) X(27) X(30) X(32) \
  X(36) X(40) X(45) X(48) X(50) X(54) X(60) X(64)

template <class T, bool INV>
__device__ __forceinline__ void any_transform(int L, const Lines<T>& ln) {
  switch (L) {
#define LGF_CASE(N) \
  case N: transform<T, N, INV>(ln); break;
    LGF_LONG_LENGTHS(LGF_CASE)
#undef LGF_CASE
  }
}

// The x-y pass: tpc tiles (one field of one plane each, tile = 4 plane + field)
// per CTA, [tile][y][x] with an odd row pitch.
template <class T, bool INV>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 8 ? 4 : 6)
    k_long_xy(cx<T>* __restrict__ D, const anyfft::XyGeom g, const DevState* __restrict__ st) {
  pdl_wait();
  if (st != nullptr && st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* tiles = reinterpret_cast<cx<T>*>(smem_raw);
  const int t0 = blockIdx.x * g.tpc;
  const int nt = g.ntiles - t0 < g.tpc ? g.ntiles - t0 : g.tpc;
  // rows of all tiles, a row's elements on neighbouring threads
  auto rows = [&](auto&& move) {
    for (int e = threadIdx.x; e < nt * g.N; e += kThreads) {
      const int r = anyfft::quot(e, g.x), x = e - r * g.Lx;  // row of the CTA
      const int j = (unsigned)r / (unsigned)g.Ly, y = r - j * g.Ly, tile = t0 + j;
      move(D + ((tile & 3) * g.V + (tile >> 2) * g.N + y * g.Lx + x), tiles + r * g.P + x);
    }
  };
  rows([](cx<T>* d, cx<T>* s) { *s = *d; });
  __syncthreads();
  any_transform<T, INV>(g.Ly, Lines<T>{tiles, nt * g.Lx, g.Lx, 1, g.Ly * g.P, g.P});
  __syncthreads();
  any_transform<T, INV>(g.Lx, Lines<T>{tiles, nt * g.Ly, nt * g.Ly, g.P, 0, 1});
  __syncthreads();
  rows([](cx<T>* d, cx<T>* s) { *d = *s; });
}

// The z-t pass: one CTA per field and run of bx columns, [t][z][column] with a
// padded t pitch; the factor from the per-site table.
template <class T>
__global__ void __launch_bounds__(kThreads, sizeof(T) == 8 ? 4 : 6)
    k_long_zt(cx<T>* __restrict__ D, const anyfft::ZtGeom g, const T* __restrict__ kfac,
              const DevState* __restrict__ st) {
  pdl_wait();
  if (st != nullptr && st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<T>* tile = reinterpret_cast<cx<T>*>(smem_raw);
  const int q0 = blockIdx.x * g.bx;
  cx<T>* Df = D + (blockIdx.y * g.V + q0);
  const int nx = g.S - q0 < g.bx ? g.S - q0 : g.bx;  // a ragged last run: the columns past it are zeros
  auto sites = [&](auto&& move) {
    for (int e = threadIdx.x; e < g.bx * g.Lz * g.Lt; e += kThreads) {
      const int xb = e & (g.bx - 1), r = e >> g.lbx;  // r = z + Lz t
      const int t = (unsigned)r / (unsigned)g.Lz, z = r - t * g.Lz;
      move(xb < nx, Df + xb + g.S * r, tile + t * g.PT + z * g.bx + xb);
    }
  };
  sites([](bool in, cx<T>* d, cx<T>* s) { *s = in ? *d : mk<T>(0, 0); });
  __syncthreads();
  const Lines<T> zl{tile, g.bx * g.Lt, g.bx, 1, g.PT, g.bx};
  const Lines<T> tl{tile, g.bx * g.Lz, g.bx * g.Lz, 1, 0, g.PT};
  any_transform<T, false>(g.Lz, zl);
  __syncthreads();
  switch (g.Lt) {
#define LGF_CASE(N) \
  case N: accelerate<T, N>(tl, kfac + q0, g.S, nx, g.bx, g.lbx, g.S * g.Lz); break;
    LGF_LONG_LENGTHS(LGF_CASE)
#undef LGF_CASE
  }
  __syncthreads();
  any_transform<T, true>(g.Lz, zl);
  __syncthreads();
  sites([](bool in, cx<T>* d, cx<T>* s) {
    if (in) *d = *s;
  });
}

}  // namespace

template <class T>
cudaError_t init(int smem) {
  cudaError_t e = cudaFuncSetAttribute(k_long_xy<T, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_long_xy<T, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(k_long_zt<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  return e;
}

template <class T>
cudaError_t launch_xy(void* D, const anyfft::XyGeom& g, size_t smem, bool inverse, const DevState* st,
                      cudaStream_t s) {
  const unsigned nb = (unsigned)((g.ntiles + g.tpc - 1) / g.tpc);
  const auto d = static_cast<cx<T>*>(D);
  if (inverse) return launch_pdl(k_long_xy<T, true>, nb, kThreads, smem, s, d, g, st);
  return launch_pdl(k_long_xy<T, false>, nb, kThreads, smem, s, d, g, st);
}

template <class T>
cudaError_t launch_zt(void* D, const anyfft::ZtGeom& g, size_t smem, const void* kfac, const DevState* st,
                      cudaStream_t s) {
  const dim3 grid((unsigned)((g.S + g.bx - 1) / g.bx), 4);
  return launch_pdl(k_long_zt<T>, grid, kThreads, smem, s, static_cast<cx<T>*>(D), g, static_cast<const T*>(kfac),
                    st);
}

template cudaError_t init<LGF_LONG_T>(int);
template cudaError_t launch_xy<LGF_LONG_T>(void*, const anyfft::XyGeom&, size_t, bool, const DevState*, cudaStream_t);
template cudaError_t launch_zt<LGF_LONG_T>(void*, const anyfft::ZtGeom&, size_t, const void*, const DevState*,
                                           cudaStream_t);

}  // namespace longfft
}  // namespace lgf
