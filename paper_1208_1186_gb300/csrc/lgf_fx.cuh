// Fixed-point pairs: the working form of the links and of g in the plain FP64
// iteration.
//
// FP64 runs at 1/62 of the FP32 rate on this GPU (about 2 multiply-adds per
// clock and SM), so the 864 multiply-adds of the link update alone took half of
// the FP64 iteration.  Every number the products multiply is an entry of a
// unitary matrix, at most 1 in magnitude, so it needs no exponent:
//
//   x = (h + l) 2^-30,  h a 32-bit integer, l an FP32 number with |l| <= 1/2,
//
// a resolution of 2^-55 (FP64 resolves 2^-53 of a number near 1).  A product
// is
//
//   x y 2^60 = h_x h_y + (h_x l_y + l_x h_y) + l_x l_y:
//
// the first term exact in a 64-bit integer accumulator (one 32 x 32 + 64
// multiply-add; 32 a clock and SM), the second in an FP32 accumulator (two
// FMAs; the rounding of a term below 2^29 is 2^5, i.e. 2^-55 of the result),
// the third, at most 1/4, dropped.  A dot product of six terms is off by about
// 2^-54, where six FP64 roundings leave about 2^-53.
//
// The resolution is absolute: an entry below 1/8 keeps fewer significant bits than
// FP64 would.  Against 80-bit arithmetic the links after 26 updates of 32^4 are off
// by 3.1e-16 rms (FP64 kernels 4.4e-16), 16^4 3.0 (4.2), 12 x 18 x 10 x 20 in 12-real
// storage 3.4 (4.9); their entries below 1/8 alone 3.0 (1.6).  theta comes to rest at
// 1e-31 to 2e-31, where FP64 links go on to 6e-33 and, near the identity, below
// 1e-40; fixes to such tolerances run on the FP64 links (lgf_api.cu, kFxTheta).
//
// Range: |h| < 2^31 holds |x| < 2; rows of norm at most 1 + 2^-7 times unitary
// matrices keep every entry below 1.75 and every accumulator below 2^62.
#pragma once

#include "lgf_common.cuh"

namespace lgf {

// one complex number
struct alignas(16) fx {
  int hr;
  float lr;
  int hi;
  float li;
};

__device__ __forceinline__ fx fx_ldg(const fx* p) {
  const int4 v = __ldg(reinterpret_cast<const int4*>(p));
  return {v.x, __int_as_float(v.y), v.z, __int_as_float(v.w)};
}

__device__ __forceinline__ fx fx_neg(fx a) { return {-a.hr, -a.lr, -a.hi, -a.li}; }

// a real operand with its integer part also in FP32
struct fxr {
  int h;
  float l, f;
};

__device__ __forceinline__ fxr fx_re(const fx& a) { return {a.hr, a.lr, (float)a.hr}; }
__device__ __forceinline__ fxr fx_im(const fx& a) { return {a.hi, a.li, (float)a.hi}; }
__device__ __forceinline__ fxr fx_neg(fxr a) { return {-a.h, -a.l, -a.f}; }

struct fxacc {
  long long h;
  float l;
};

// a += x y
__device__ __forceinline__ void fx_mac(fxacc& a, const fxr& x, const fxr& y) {
  a.h += (long long)x.h * (long long)y.h;
  a.l = __fmaf_rn(x.f, y.l, __fmaf_rn(x.l, y.f, a.l));
}

// an accumulated product sum, in units of 2^-60, as h and l
__device__ __forceinline__ void fx_round(const fxacc& a, int& h, float& l) {
  h = (int)((a.h + (1ll << 29)) >> 30);
  const int rem = (int)((unsigned)a.h - ((unsigned)h << 30));  // |rem| <= 2^29
  const float t = __fmul_rn(__fadd_rn((float)rem, a.l), 0x1p-30f);
  const float k = __fadd_rn(t, 12582912.f);  // 1.5 2^23: t rounded to an integer in the low bits
  h += __float_as_int(k) - 0x4B400000;
  l = __fsub_rn(t, __fsub_rn(k, 12582912.f));
}

__device__ __forceinline__ fx fx_round(const fxacc& re, const fxacc& im) {
  fx r;
  fx_round(re, r.hr, r.lr);
  fx_round(im, r.hi, r.li);
  return r;
}

// entry j of row 3 of an SU(3) matrix from rows 1 and 2: conj(r1 x r2)
__device__ __forceinline__ fx fx_row3(const fx* r1, const fx* r2, int j) {
  const int k = (j + 1) % 3, l = (j + 2) % 3;
  const fxr ukr = fx_re(r1[k]), uki = fx_im(r1[k]), ulr = fx_re(r1[l]), uli = fx_im(r1[l]);
  const fxr vkr = fx_re(r2[k]), vki = fx_im(r2[k]), vlr = fx_re(r2[l]), vli = fx_im(r2[l]);
  fxacc re = {0, 0.f}, im = {0, 0.f};
  fx_mac(re, ukr, vlr);
  fx_mac(re, fx_neg(uki), vli);
  fx_mac(re, fx_neg(ulr), vkr);
  fx_mac(re, uli, vki);
  fx_mac(im, fx_neg(ukr), vli);
  fx_mac(im, fx_neg(uki), vlr);
  fx_mac(im, ulr, vki);
  fx_mac(im, uli, vkr);
  return fx_round(re, im);
}

// FP64 -> (h, l) by bit manipulation (FP64 arithmetic and conversions run at
// the FP64 rate); false for |x| >= 2 and for non-finite x
__device__ __forceinline__ bool fx_from_double(double x, int& h, float& l) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ffull) - 1023;
  const unsigned long long m = ((b << 11) | (1ull << 63));  // |x| = m 2^(e - 63)
  const int sh = 1 - e;                                      // |x| = (m >> sh) 2^-62
  long long f = sh < 64 ? (long long)(m >> (sh & 63)) : 0;
  if ((long long)b < 0) f = -f;
  h = (int)((f + (1ll << 31)) >> 32);
  l = __fmul_rn((float)(int)(unsigned)f, 0x1p-32f);
  return e <= 0;
}

// The row of three complex numbers as pairs relative to a power of two: the
// largest exponent among the six numbers, or up to two more where the row's
// norm would pass 1.97.  The norm of the result is then between 0.98 and 1.97.
// False for a row that is not finite or not normal.
__device__ __forceinline__ bool fx_row_from_double(const cx<double>* x, fx* r) {
  unsigned long long b[6];
  int top = 0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    b[2 * j] = (unsigned long long)__double_as_longlong(x[j].re);
    b[2 * j + 1] = (unsigned long long)__double_as_longlong(x[j].im);
    top = max(top, max((int)(b[2 * j] >> 52) & 0x7ff, (int)(b[2 * j + 1] >> 52) & 0x7ff));
  }
  if (top == 0x7ff || top < 64) return false;
  for (;; ++top) {  // each turn quarters n, which starts below 24
    float n = 0.f;
    int h[6];
    float l[6];
#pragma unroll
    for (int j = 0; j < 6; ++j) {
      const int sh = 1 + top - (int)((b[j] >> 52) & 0x7ff);  // at least 64 where x is 0
      const unsigned long long m = (b[j] << 11) | (1ull << 63);
      long long f = sh < 64 ? (long long)(m >> (sh & 63)) : 0;
      if ((long long)b[j] < 0) f = -f;
      h[j] = (int)((long long)((unsigned long long)f + (1ull << 31)) >> 32);  // +-2^31 wraps: n is too large then
      l[j] = __fmul_rn((float)(int)(unsigned)f, 0x1p-32f);
      n = __fmaf_rn((float)h[j], (float)h[j], n);
    }
    if (n > 3.88f * 0x1p60f) continue;
#pragma unroll
    for (int j = 0; j < 3; ++j) r[j] = {h[2 * j], l[2 * j], h[2 * j + 1], l[2 * j + 1]};
    return true;
  }
}

// f 2^-kScale as the nearest FP64 number, by bit manipulation
template <int kScale>
__device__ __forceinline__ double fx_scaled_to_double(long long f) {
  unsigned long long u = f < 0 ? 0ull - (unsigned long long)f : (unsigned long long)f;
  if (u == 0) return 0.0;
  const int n = __clzll((long long)u);
  u <<= n;  // the leading bit at 63
  unsigned long long v = u >> 11;
  const unsigned r = (unsigned)u & 0x7ffu;
  v += (r > 0x400u || (r == 0x400u && (v & 1))) ? 1ull : 0ull;
  // the leading bit of v adds one to the exponent field (and a carry another)
  v += (unsigned long long)(1023 + 63 - n - kScale - 1) << 52;
  return __longlong_as_double((long long)(v | (f < 0 ? 1ull << 63 : 0ull)));
}

__device__ __forceinline__ double fx_to_double(int h, float l) {
  return fx_scaled_to_double<62>(((long long)h << 32) + (long long)__float2int_rn(__fmul_rn(l, 0x1p32f * 0.5f)) * 2);
}

// a sum of (h, l) pairs, in units of 2^-30 and at most 2^34 of them, as FP64
__device__ __forceinline__ double fx_sum_to_double(const fxacc& a) {
  return fx_scaled_to_double<58>((a.h << 28) + __float2int_rn(__fmul_rn(a.l, 0x1p28f)));
}

// the squared norm of a row, below 4, in units of 2^-60
__device__ __forceinline__ long long fx_norm2(const fx* r) {
  fxacc n = {0, 0.f};
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    fx_mac(n, fx_re(r[j]), fx_re(r[j]));
    fx_mac(n, fx_im(r[j]), fx_im(r[j]));
  }
  // |n.l| < 2^33: to a multiple of 2^4, i.e. 2^-56
  return n.h + ((long long)__float2int_rn(__fmul_rn(n.l, 0x1p-4f)) << 4);
}

// A row of squared norm n2 2^-60, above 1/4, to norm 1.  What the FP64 inverse
// root leaves, some 2^-53, is a common factor of the row, an error that the
// iterations add up: it is measured on the result and taken out to first order.
__device__ __forceinline__ bool fx_normalize(fx* r, long long n2) {
  fxr k;
  const bool ok = fx_from_double(rsqrt(fx_scaled_to_double<60>(n2)), k.h, k.l);
  k.f = (float)k.h;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    fxacc re = {0, 0.f}, im = {0, 0.f};
    fx_mac(re, fx_re(r[j]), k);
    fx_mac(im, fx_im(r[j]), k);
    r[j] = fx_round(re, im);
  }
  const float c = __fmul_rn((float)(int)((1ll << 60) - fx_norm2(r)), 0x1p-61f);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    r[j].lr = __fmaf_rn((float)r[j].hr, c, r[j].lr);
    r[j].li = __fmaf_rn((float)r[j].hi, c, r[j].li);
  }
  return ok;
}

// Rows 1 and 2 of a matrix to the orthonormal rows of its reunitarisation
// (Gram-Schmidt, as reunitarize()).  A row's length cancels in its
// normalisation, so each is taken relative to a power of two and the products
// run on pairs; the two inverse square roots are FP64.  Where row 2 is nearly
// parallel to row 1 its remainder is normalised in FP64.  False if the result
// is not finite.
__device__ __forceinline__ bool fx_reunitarize(const M3<double>& m, fx* r) {
  bool ok = fx_row_from_double(m.e[0], r);
  ok = ok && fx_row_from_double(m.e[1], r + 3);
  if (!ok) return false;
  ok = fx_normalize(r, fx_norm2(r));
  fxacc pr = {0, 0.f}, pi = {0, 0.f};  // sum conj(r1_j) r2_j, at most the norm of row 2
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const fxr ur = fx_re(r[j]), ui = fx_im(r[j]), vr = fx_re(r[3 + j]), vi = fx_im(r[3 + j]);
    fx_mac(pr, vr, ur);
    fx_mac(pr, vi, ui);
    fx_mac(pi, vi, ur);
    fx_mac(pi, fx_neg(vr), ui);
  }
  const fx p = fx_neg(fx_round(pr, pi));
  const fxr qr = fx_re(p), qi = fx_im(p);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    const fxr ur = fx_re(r[j]), ui = fx_im(r[j]);
    fxacc re = {(long long)r[3 + j].hr << 30, r[3 + j].lr * 0x1p30f};
    fxacc im = {(long long)r[3 + j].hi << 30, r[3 + j].li * 0x1p30f};
    fx_mac(re, qr, ur);
    fx_mac(re, fx_neg(qi), ui);
    fx_mac(im, qr, ui);
    fx_mac(im, qi, ur);
    r[3 + j] = fx_round(re, im);
  }
  const long long n2 = fx_norm2(r + 3);
  if (n2 > 0x428ll << 48) return fx_normalize(r + 3, n2) && ok;  // 0.26
  double w[6], n = 0.0;
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    w[2 * j] = fx_to_double(r[3 + j].hr, r[3 + j].lr);
    w[2 * j + 1] = fx_to_double(r[3 + j].hi, r[3 + j].li);
    n = fma(w[2 * j], w[2 * j], fma(w[2 * j + 1], w[2 * j + 1], n));
  }
  n = rsqrt(n);
#pragma unroll
  for (int j = 0; j < 3; ++j) {
    ok = fx_from_double(w[2 * j] * n, r[3 + j].hr, r[3 + j].lr) && ok;
    ok = fx_from_double(w[2 * j + 1] * n, r[3 + j].hi, r[3 + j].li) && ok;
  }
  return ok;
}

}  // namespace lgf
