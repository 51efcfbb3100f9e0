// FP64 line transforms in 64-bit block floating point.
//
// The FP64 pipe does two operations a clock and SM, 1/62 of the FP32 rate, and
// bounds an FP64 FFT pass at an eighth of what memory allows; the integer pipes
// add 64-bit numbers at 32 a clock and SM and multiply 32 x 32 + 64 at 32.  A
// tile of lines therefore takes one exponent and is transformed as 64-bit
// integers: additions are exact, a twiddle product is off by about one unit.
// Before each axis the tile is scaled so that the largest sum of |re| + |im|
// over one of its lines is just below 2^62.  That sum bounds every number of the
// line's transform, and where a few large modes dominate (as after the
// acceleration) it leaves almost all bits to the numbers themselves: an FP64
// transform rounds each number at 53 bits, this one all of them at 62 bits below
// the line's sum.
//
// The exponent is the CTA's: the tiles of an x-y CTA (fields and planes) and the
// columns of a z-t CTA share it, so numbers far below the CTA's largest are cut off
// at 2^-61 of it, not at their own 53 bits.
//
// regfft's transforms (fft_reg.cuh) run on this type as they do on float and
// double: the same stages and order, with twiddles and factors of 62 bits.  Error
// of the whole acceleration against extended precision, FP64 -> this: 8^4 3.9e-16 ->
// 1.1e-16, 16^4 4.8e-16 -> 1.3e-16, 24^3 x 12 7.1e-16 -> 1.4e-16, 32 x 32 x 8 x 8
// 5.6e-16 -> 1.8e-16 (with twiddles of 53 bits, some units off, and factors of 60 2.7,
// 3.3, 5.9 and 3.8e-16).
#pragma once

#include "fft_any.cuh"
#include "fft_reg.cuh"
#include "lgf_fx.cuh"

namespace lgf {
namespace fxfft {

// data: a tile's integers; constants (twiddles, |c| <= 1): c 2^62
struct I {
  long long v;
  I() = default;
  __host__ __device__ constexpr explicit I(double c)
      : v((long long)(c * 4611686018427387904.0 + (c < 0 ? -0.5 : 0.5))) {}
  __device__ constexpr I operator-() const { return from(-v); }
  __host__ __device__ static constexpr I from(long long x) {
    I r(0.0);
    r.v = x;
    return r;
  }
};
// the constant's 62 bits, of which a double has 53
constexpr I constant(regfft::dd c) {
  const double S = 4611686018427387904.0, x = c.h * S;
  const long long n = (long long)x;
  const double r = (x - (double)n) + c.l * S;
  return I::from(n + (long long)(r + (r < 0 ? -0.5 : 0.5)));
}
}  // namespace fxfft

namespace regfft {
template <>
struct Constant<fxfft::I> {
  static constexpr fxfft::I of(dd c) { return fxfft::constant(c); }
};
}  // namespace regfft

namespace fxfft {

__device__ __forceinline__ I operator+(I a, I b) { return I::from(a.v + b.v); }
__device__ __forceinline__ I operator-(I a, I b) { return I::from(a.v - b.v); }

// a number as hi 2^32 + lo, both signed
struct Split {
  int hi, lo;
};
__device__ __forceinline__ Split split(long long x) { return {(int)((x + 0x80000000ll) >> 32), (int)x}; }

// sums of at most two products a c / 2^62, the low x low parts (below one unit)
// left out; in range for |a|, or the sum of the two |a|, up to 2^62 and |c| <= 2^62
struct Acc {
  long long hi = 0, mid = 1ll << 29;  // rounds value(): a floor would add up over a line
  __device__ __forceinline__ void add(Split a, Split c) {
    hi += (long long)a.hi * c.hi;
    mid += (long long)a.hi * c.lo + (long long)a.lo * c.hi;
  }
  __device__ __forceinline__ void sub(Split a, Split c) {
    hi -= (long long)a.hi * c.hi;
    mid -= (long long)a.hi * c.lo + (long long)a.lo * c.hi;
  }
  __device__ __forceinline__ I value() const { return I::from((hi << 2) + (mid >> 30)); }
};

__device__ __forceinline__ I operator*(I a, I c) {
  Acc r;
  r.add(split(a.v), split(c.v));
  return r.value();
}

// v (wr + i wi), found by regfft's twiddle product
__device__ __forceinline__ cx<I> mul_const(cx<I> v, I wr, I wi) {
  const Split a = split(v.re.v), b = split(v.im.v), r = split(wr.v), i = split(wi.v);
  Acc re, im;
  re.add(a, r);
  re.sub(b, i);
  im.add(a, i);
  im.add(b, r);
  return mk<I>(re.value(), im.value());
}

// biased exponent of an FP64 bit pattern
__device__ __forceinline__ int exponent(long long bits) { return (int)((unsigned long long)bits >> 52) & 0x7ff; }

// x 2^(61 - down - (E - 1022)) as an integer, for |x| < 2^(E - 1022)
__device__ __forceinline__ long long from_bits(long long bits, int E, int down) {
  const int e = exponent(bits), sh = E - e + down;
  const unsigned long long m = (((unsigned long long)bits & 0xfffffffffffffull) | (1ull << 52)) << 8;
  const long long f = e != 0 && sh < 64 ? (long long)(m >> sh) : 0;  // subnormals count as zero
  return bits < 0 ? -f : f;
}

// a factor x >= 0 as x 2^(63 - (E - 1022)), for x < 2^(E - 1023): all of the 62 bits
// a constant may have, because the product with a column's largest factor is all
// that the smallest momenta, which carry most of the result, are left with
__device__ __forceinline__ I factor(long long bits, int E) {
  const int e = exponent(bits), sh = E - e;
  const unsigned long long m = (((unsigned long long)bits & 0xfffffffffffffull) | (1ull << 52)) << 10;
  return I::from(e != 0 && sh < 64 ? (long long)(m >> sh) : 0);
}

// |x| 2^(18 - (E - 1022)), rounded up to an integer
__device__ __forceinline__ int size_of_bits(long long bits, int E) {
  const int hi = (int)(bits >> 32) & 0x7fffffff;
  const int sh = E - (hi >> 20);
  return sh < 32 ? (int)((((unsigned)hi & 0xfffffu) | 0x100000u) >> 3 >> sh) + 1 : 1;
}

// f 2^X as the nearest FP64 number (0 below its normal range, infinite above it)
__device__ __forceinline__ double to_double(long long f, int X) {
  unsigned long long u = f < 0 ? 0ull - (unsigned long long)f : (unsigned long long)f;
  const int n = __clzll((long long)u);
  const int e = 1023 + 63 - n + X;
  if (u == 0 || e < 1) return 0.0;
  if (e > 2046) return __longlong_as_double(f < 0 ? (long long)0xfff0000000000000ull : 0x7ff0000000000000ll);
  u <<= n;
  unsigned long long v = u >> 11;
  const unsigned r = (unsigned)u & 0x7ffu;
  v += (r > 0x400u || (r == 0x400u && (v & 1))) ? 1ull : 0ull;
  v += (unsigned long long)(e - 1) << 52;
  return __longlong_as_double((long long)(v | (f < 0 ? 1ull << 63 : 0ull)));
}

// |x| 2^-44, rounded up to an integer
__device__ __forceinline__ int size_of(I x) {
  const int h = (int)(x.v >> 32);
  return ((h ^ (h >> 31)) >> 12) + 1;
}
// sum of |re| + |im| of a line, in units of 2^44 (below 2^26 for 64 numbers below 2^62)
// the right shift that brings line sums of up to m 2^unit below 2^62
__device__ __forceinline__ int shift_for(int m, int unit) {
  const int s = 32 - __clz(m) + unit - 62;
  return s > 0 ? s : 0;
}

// a tile that holds an infinity or a NaN comes out as NaN (an FP64 transform
// would spread it over the tile's lines as well)
__device__ __forceinline__ double nan64() { return __longlong_as_double(0x7ff8000000000000ll); }

// a >> s, rounded (a floor's bias would gather in the modes of momentum 0 along
// the axis, which the acceleration amplifies)
__device__ __forceinline__ I shifted(I a, int s, long long half) { return I::from((a.v + half) >> s); }

__device__ __forceinline__ cx<double> out(cx<I> a, int X, bool bad) {
  return bad ? mk<double>(nan64(), nan64()) : mk<double>(to_double(a.re.v, X), to_double(a.im.v, X));
}

// A line in shared memory, shifted down by s and transformed in place.  A
// transform of 32 is 24 KB of straight-line code; a kernel with its conversions
// and both axes unrolled as well ran 158 KB once per warp and spent its time
// fetching instructions (7.2 cycles per issue, ncu).  So everything but the
// transforms runs in short loops over shared memory.
template <int L, bool INV>
__device__ __forceinline__ void line_inlined(cx<I>* base, int stride, int s) {
  const long long half = (1ll << s) >> 1;
  cx<I> v[L];
  cx<I>* p = base;
#pragma unroll
  for (int i = 0; i < L; ++i) {
    const longlong2 b = *reinterpret_cast<const longlong2*>(p);
    v[i] = mk<I>(shifted(I::from(b.x), s, half), shifted(I::from(b.y), s, half));
    p += stride;
  }
  if (INV)
    regfft::inverse<I, L>(v);
  else
    regfft::forward<I, L>(v);
  p = base;
#pragma unroll
  for (int i = 0; i < L; ++i) {
    *reinterpret_cast<longlong2*>(p) = make_longlong2(v[i].re.v, v[i].im.v);
    p += stride;
  }
}

template <int L, bool INV>
__device__ __noinline__ void line(cx<I>* base, int stride, int s) {
  line_inlined<L, INV>(base, stride, s);
}

// lines of up to 32: 64 integers of 64 bits, in 128 registers.  (Longer ones
// spilled, and took ptxas minutes.)
constexpr int kMaxLine = 32;

// N: the length, if the kernel is instantiated for it, or 0
template <int N, bool INV>
__device__ __forceinline__ void any_line(int L, cx<I>* base, int stride, int s) {
  if constexpr (N != 0)
    line_inlined<N, INV>(base, stride, s);
  else
    anyfft::with_length<kMaxLine>(L, [&](auto n) { line<decltype(n)::value, INV>(base, stride, s); });
}

__device__ __forceinline__ longlong2 bits_at(const cx<double>* p) { return *reinterpret_cast<const longlong2*>(p); }
__device__ __forceinline__ longlong2 bits_at(const cx<I>* p) { return *reinterpret_cast<const longlong2*>(p); }

// maximum over the CTA, gathered in *slot (zeroed before; valid after the next
// barrier).  Every thread calls it; the CTA is whole warps.
__device__ __forceinline__ void gather_max(int* slot, int m) {
  m = __reduce_max_sync(0xffffffffu, m);
  if ((threadIdx.x & 31) == 0) atomicMax(slot, m);
}

// FP64 bits of a line in shared memory: the sum of its |re| + |im| in units of
// 2^43 of the integers that from_bits gives for down = 0
__device__ __forceinline__ int bits_sum(const cx<I>* p, int L, int stride, int E) {
  int m = 0;
#pragma unroll 4
  for (int i = 0; i < L; ++i) {
    const longlong2 b = bits_at(p + i * stride);
    m += size_of_bits(b.x, E) + size_of_bits(b.y, E);
  }
  return m;
}
// the same for integers, in units of 2^44
__device__ __forceinline__ int line_sum(const cx<I>* p, int L, int stride) {
  int m = 0;
#pragma unroll 4
  for (int i = 0; i < L; ++i) {
    const longlong2 b = bits_at(p + i * stride);
    m += size_of(I::from(b.x)) + size_of(I::from(b.y));
  }
  return m;
}
__device__ __forceinline__ void to_integers(cx<I>* p, int L, int stride, int E, int down) {
#pragma unroll 4
  for (int i = 0; i < L; ++i) {
    const longlong2 b = bits_at(p + i * stride);
    *reinterpret_cast<longlong2*>(p + i * stride) =
        make_longlong2(from_bits(b.x, E, down), from_bits(b.y, E, down));
  }
}

// 32^4: x-y 229 us on the FP64 pipe, now 90; z-t 455, now 171.
//
// The x-y pass: tpc tiles (one field of one plane each, tile = 4 plane + field)
// per CTA, which share an exponent; a thread per y-line, then per x-line.  The
// row pitch is odd, so no phase has bank conflicts.
template <bool INV, int N = 0>  // N: Lx = Ly, or 0
__global__ void __launch_bounds__(kFxThreads, 3)
    k_fx_xy(cx<double>* __restrict__ D, const anyfft::XyGeom g, const DevState* __restrict__ st) {
  pdl_wait();
  if (st != nullptr && st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int slot[3];
  cx<I>* tiles = reinterpret_cast<cx<I>*>(smem_raw);  // [tile][y][x], row pitch P
  const int t0 = blockIdx.x * g.tpc;
  const int nt = g.ntiles - t0 < g.tpc ? g.ntiles - t0 : g.tpc;
  const int NT = blockDim.x, nx = nt * g.Lx, ny = nt * g.Ly;
  if (threadIdx.x < 3) slot[threadIdx.x] = 0;
  __syncthreads();
  // a thread's columns: for each y the threads of a tile read one contiguous row
  int E = 0;
  for (int l = threadIdx.x; l < nx; l += NT) {
    const int j = anyfft::quot(l, g.x), x = l - j * g.Lx, tile = t0 + j;
    const cx<double>* src = D + ((tile & 3) * g.V + (tile >> 2) * g.N + x);
    cx<I>* col = tiles + j * g.Ly * g.P + x;
#pragma unroll 8
    for (int i = 0; i < g.Ly; ++i) {
      const longlong2 b = bits_at(src + i * g.Lx);
      *reinterpret_cast<longlong2*>(col + i * g.P) = b;
      E = max(E, max(exponent(b.x), exponent(b.y)));
    }
  }
  gather_max(slot, E);
  __syncthreads();
  E = slot[0];
  int m = 0;
  for (int l = threadIdx.x; l < nx; l += NT) {
    const int j = anyfft::quot(l, g.x);
    m = max(m, bits_sum(tiles + j * g.Ly * g.P + (l - j * g.Lx), g.Ly, g.P, E));
  }
  gather_max(slot + 1, m);
  __syncthreads();
  const int s0 = shift_for(slot[1], 43);
  for (int l = threadIdx.x; l < nx; l += NT) {
    const int j = anyfft::quot(l, g.x);
    cx<I>* col = tiles + j * g.Ly * g.P + (l - j * g.Lx);
    to_integers(col, g.Ly, g.P, E, s0);
    any_line<N, INV>(g.Ly, col, g.P, 0);
  }
  __syncthreads();
  m = 0;
  for (int l = threadIdx.x; l < ny; l += NT) m = max(m, line_sum(tiles + l * g.P, g.Lx, 1));
  gather_max(slot + 2, m);
  __syncthreads();
  const int s1 = shift_for(slot[2], 44);
  for (int l = threadIdx.x; l < ny; l += NT) any_line<N, INV>(g.Lx, tiles + l * g.P, 1, s1);
  __syncthreads();
  const int X = E - 1022 - 61 + s0 + s1;
  for (int l = threadIdx.x; l < nx; l += NT) {
    const int j = anyfft::quot(l, g.x), x = l - j * g.Lx, tile = t0 + j;
    cx<double>* dst = D + ((tile & 3) * g.V + (tile >> 2) * g.N + x);
    const cx<I>* col = tiles + j * g.Ly * g.P + x;
#pragma unroll 4
    for (int i = 0; i < g.Ly; ++i) dst[i * g.Lx] = out(col[i * g.P], X, E == 0x7ff);
  }
}

// The z-t pass: one CTA per field and run of bx columns, as k_any_zt; its columns
// share an exponent and the scale of their factors, which is the largest factor
// of any of them, at frequency 0 of z and t (in the origin's tile the lattice's).
template <int NZ = 0, int NT = 0>  // Lz and Lt, or 0
__global__ void __launch_bounds__(kFxThreads, 3)
    k_fx_zt(cx<double>* __restrict__ D, const anyfft::ZtGeom g, const double* __restrict__ kfac, int kmax_exponent,
            const DevState* __restrict__ st) {
  pdl_wait();
  if (st != nullptr && st->done) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ int slot[5];
  cx<I>* tile = reinterpret_cast<cx<I>*>(smem_raw);  // [t][z][column], t pitch PT
  const int q0 = blockIdx.x * g.bx;
  const int xb = threadIdx.x & (g.bx - 1), row = threadIdx.x >> g.lbx;
  const int q = q0 + xb;
  const bool inside = q < g.S;
  const bool zline = inside && row < g.Lt, tline = inside && row < g.Lz;
  cx<double>* Dq = D + (blockIdx.y * g.V + q + g.S * g.Lz * row);
  cx<I>* const zl = tile + row * g.PT + xb;    // z line of t = row
  cx<I>* const tl = tile + row * g.bx + xb;    // t line of z = row
  if (threadIdx.x < 5) slot[threadIdx.x] = 0;
  __syncthreads();
  int E = 0;
  if (zline) {
#pragma unroll 8
    for (int i = 0; i < g.Lz; ++i) {
      const longlong2 b = bits_at(Dq + i * g.S);
      *reinterpret_cast<longlong2*>(zl + i * g.bx) = b;
      E = max(E, max(exponent(b.x), exponent(b.y)));
    }
  }
  gather_max(slot, E);
  __syncthreads();
  E = slot[0];
  gather_max(slot + 1, zline ? bits_sum(zl, g.Lz, g.bx, E) : 0);
  __syncthreads();
  const int s0 = shift_for(slot[1], 43);
  if (zline) {
    to_integers(zl, g.Lz, g.bx, E, s0);
    any_line<NZ, false>(g.Lz, zl, g.bx, 0);
  }
  __syncthreads();
  gather_max(slot + 2, tline ? line_sum(tl, g.Lt, g.PT) : 0);
  int EK = kmax_exponent;
  if (q0 != 0) {
    EK = 0;
    for (int k = 0; k < g.bx && q0 + k < g.S; ++k)
      EK = max(EK, exponent(__double_as_longlong(__ldg(kfac + q0 + k))));
  }
  EK += 1;
  __syncthreads();
  const int s1 = shift_for(slot[2], 44);
  int m = 0;
  if (tline) {
    any_line<NT, false>(g.Lt, tl, g.PT, s1);
    const double* kl = kfac + (q + g.S * row);
    const int step = g.S * g.Lz;
#pragma unroll 4
    for (int i = 0; i < g.Lt; ++i) {
      const longlong2 b = bits_at(tl + i * g.PT);
      const I k = factor(__double_as_longlong(__ldg(kl + i * step)), EK);
      const I re = I::from(b.x) * k, im = I::from(b.y) * k;
      *reinterpret_cast<longlong2*>(tl + i * g.PT) = make_longlong2(re.v, im.v);
      m += size_of(re) + size_of(im);
    }
  }
  gather_max(slot + 3, m);
  __syncthreads();
  const int s2 = shift_for(slot[3], 44);
  if (tline) any_line<NT, true>(g.Lt, tl, g.PT, s2);
  __syncthreads();
  gather_max(slot + 4, zline ? line_sum(zl, g.Lz, g.bx) : 0);
  __syncthreads();
  const int s3 = shift_for(slot[4], 44);
  if (zline) {
    any_line<NZ, true>(g.Lz, zl, g.bx, s3);
    // the factor is k 2^-63 2^(EK - 1022), used as k 2^-62
    const int X = E - 1022 - 61 + s0 + s1 + s2 + s3 + EK - 1022 - 1;
#pragma unroll 4
    for (int i = 0; i < g.Lz; ++i) Dq[i * g.S] = out(zl[i * g.bx], X, E == 0x7ff);
  }
}

}  // namespace fxfft
}  // namespace lgf
