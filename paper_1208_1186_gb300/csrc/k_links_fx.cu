// The plain FP64 iteration on links in fixed-point pairs (lgf_fx.cuh): the
// same method as k_links.cu's FP64 kernels, with the link arithmetic on the
// integer and FP32 pipes.
//
//   k_fx_load      FP64 links -> pairs, at the start of an iteration queue
//   k_gradient_fx  Delta (FP64, packed), F and theta from exact integer sums
//   k_build_g_fx   g = reunitarised (1 + alpha/2 Delta~), Gram-Schmidt on pairs
//   k_update_fx    U_mu(x) <- g(x) U_mu(x) g(x+mu)^dag
//   k_fx_store     pairs -> FP64 links, at the end of the queue
//
// Delta's Fourier acceleration takes and gives FP64 numbers (lines up to 32 run as
// 64-bit integers inside, fft_fx.cuh).  Links whose rows are not unit vectors
// within 2^-7 do not fit the pairs' range: k_fx_load then stops the queue with
// DevState::unfit and the host runs the FP64 kernels on the untouched FP64 links,
// as it does for tolerances below the pairs' floor and on handles without pairs.
//
// 32^4, us per launch, FP64 kernels -> these: update 1570 -> 281, gradient
// 395 -> 118, g 218 -> 54; load and store of the pairs, once per queue, 180
// each.
#include "lgf_fx.cuh"
#include "lgf_kernels.cuh"
#include "lgf_reduce.cuh"

namespace lgf {

namespace {

// one thread per (site, direction), a block 32 sites x 4 directions
template <int NC>
__global__ void __launch_bounds__(128) k_fx_load(const cx<double>* __restrict__ U, fx* __restrict__ F, int V,
                                                 DevState* __restrict__ st) {
  const int s = blockIdx.x * 32 + (threadIdx.x & 31);
  if (s >= V) return;
  const int base = (threadIdx.x >> 5) * NC * V + s;
  bool ok = true;
#pragma unroll
  for (int i = 0; i < NC / 3; ++i) {
    float n = 0.f;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const cx<double> u = ldg(U + base + (i * 3 + j) * V);
      fx x;
      ok = fx_from_double(u.re, x.hr, x.lr) && ok;
      ok = fx_from_double(u.im, x.hi, x.li) && ok;
      F[base + (i * 3 + j) * V] = x;
      const float a = (float)x.hr * 0x1p-30f, b = (float)x.hi * 0x1p-30f;
      n += a * a + b * b;
    }
    ok = ok && fabsf(n - 1.f) <= 0x1p-7f;
  }
  if (!ok) {
    st->unfit = 1;
    st->done = 1;
  }
}

template <int NC>
__global__ void __launch_bounds__(128) k_fx_store(const fx* __restrict__ F, cx<double>* __restrict__ U, int V,
                                                  const DevState* __restrict__ st) {
  if (st->unfit || st->iters == 0) return;  // the FP64 links are still the current ones
  const int s = blockIdx.x * 32 + (threadIdx.x & 31);
  if (s >= V) return;
  const int base = (threadIdx.x >> 5) * NC * V + s;
#pragma unroll
  for (int c = 0; c < NC; ++c) {
    const fx x = fx_ldg(F + base + c * V);
    U[base + c * V] = mk<double>(fx_to_double(x.hr, x.lr), fx_to_double(x.hi, x.li));
  }
}

// the 3x3 matrix of NC planes at s (row 3 rebuilt for NC = 6)
template <int NC>
__device__ __forceinline__ void fx_load_m3(const fx* __restrict__ base, int V, int s, fx (&m)[9]) {
#pragma unroll
  for (int c = 0; c < NC; ++c) m[c] = fx_ldg(base + c * V + s);
  if constexpr (NC == 6) {
#pragma unroll
    for (int j = 0; j < 3; ++j) m[6 + j] = fx_row3(m, m + 3, j);
  }
}

__device__ __forceinline__ void fx_add(fxacc& a, int h, float l) {
  a.h += h;
  a.l += l;
}

// Delta from integer sums of the pairs, exact up to the FP32 sums of the low
// parts; FP64 only from Delta on (theta, the traceless diagonal).  Grid-stride
// over sites, so that the FP64 warp and block sums run once per thread.
//
// Bound by the loads in flight: all eight link matrices of a site are needed
// for its sums.  Three CTAs of 128 an SM leave 168 registers a thread, which
// hold them, and a grid of exactly those CTAs sweeps one contiguous region, so
// that the links of x - mu are still in cache.  32^4: 118 us (671 MB of links
// and Delta, 5.7 TB/s); eight CTAs of 128 at the compiler's own register count
// 188, with two CTAs an SM 123, with five 187; 16^4 20.6 -> 18.5.
constexpr int kGradFxCtas = 3;
template <int NC>
__global__ void __launch_bounds__(128, kGradFxCtas) k_gradient_fx(const fx* __restrict__ U, cx<double>* __restrict__ D,
                                                     double2* __restrict__ partial, const Geom geo, DevState* st,
                                                     int mode, double normF, double normT) {
  pdl_wait();
  if (queue_stopped(st, mode)) return;
  const int V = (int)geo.V;
  fxacc F = {0, 0.f};
  double tsum = 0.0;
  const int step = gridDim.x * blockDim.x;
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < V; s += step) {
    int c[4];
    site_coords_r(geo, s, c);
    // A_ij - conj(A_ji) off the diagonal, Im A_ii on it
    fxacc r01 = {0, 0.f}, i01 = r01, r02 = r01, i02 = r01, r12 = r01, i12 = r01, a0 = r01, a1 = r01, a2 = r01;
#pragma unroll
    for (int mu = 0; mu < 4; ++mu) {
      const fx* base = U + mu * NC * V;
      const int st_mu = (int)geo.stride[mu];
      const int sb = c[mu] > 0 ? s - st_mu : s + (geo.L[mu] - 1) * st_mu;
      fx o[9], b[9];
      fx_load_m3<NC>(base, V, s, o);
      fx_load_m3<NC>(base, V, sb, b);
      fx_add(F, o[0].hr, o[0].lr);
      fx_add(F, o[4].hr, o[4].lr);
      fx_add(F, o[8].hr, o[8].lr);
      auto off = [&](fxacc& re, fxacc& im, int p, int q) {  // p = (i, j), q = (j, i)
        fx_add(re, b[p].hr, b[p].lr);
        fx_add(re, -b[q].hr, -b[q].lr);
        fx_add(re, -o[p].hr, -o[p].lr);
        fx_add(re, o[q].hr, o[q].lr);
        fx_add(im, b[p].hi, b[p].li);
        fx_add(im, b[q].hi, b[q].li);
        fx_add(im, -o[p].hi, -o[p].li);
        fx_add(im, -o[q].hi, -o[q].li);
      };
      off(r01, i01, 1, 3);
      off(r02, i02, 2, 6);
      off(r12, i12, 5, 7);
      fx_add(a0, b[0].hi, b[0].li);
      fx_add(a0, -o[0].hi, -o[0].li);
      fx_add(a1, b[4].hi, b[4].li);
      fx_add(a1, -o[4].hi, -o[4].li);
      fx_add(a2, b[8].hi, b[8].li);
      fx_add(a2, -o[8].hi, -o[8].li);
    }
    const cx<double> d01 = mk<double>(fx_sum_to_double(r01), fx_sum_to_double(i01));
    const cx<double> d02 = mk<double>(fx_sum_to_double(r02), fx_sum_to_double(i02));
    const cx<double> d12 = mk<double>(fx_sum_to_double(r12), fx_sum_to_double(i12));
    // the traceless diagonal 2 a_i - (2/3) sum a = (2/3) (2 a_i - a_j - a_k), at
    // most 2^35 units: halved into the range of the conversion
    const fxacc n0 = {2 * a0.h - a1.h - a2.h, 2 * a0.l - a1.l - a2.l};
    const fxacc n1 = {2 * a1.h - a0.h - a2.h, 2 * a1.l - a0.l - a2.l};
    const double i0 = fx_scaled_to_double<57>((n0.h << 27) + __float2int_rn(n0.l * 0x1p27f)) * (2.0 / 3.0);
    const double i1 = fx_scaled_to_double<57>((n1.h << 27) + __float2int_rn(n1.l * 0x1p27f)) * (2.0 / 3.0);
    D[s] = d01;
    D[V + s] = d02;
    D[2 * V + s] = d12;
    D[3 * V + s] = mk<double>(i0, i1);
    // i0^2 + i1^2 + (i0 + i1)^2 = 2 (i0^2 + i1^2 + i0 i1)
    double t = norm2(d01);
    t = fma(d02.re, d02.re, fma(d02.im, d02.im, t));
    t = fma(d12.re, d12.re, fma(d12.im, d12.im, t));
    t = fma(i0, i0 + i1, fma(i1, i1, t));
    tsum += t;
  }
  // a thread's F: its integer sum (a few thousand terms of 2^30 at most) is
  // exact in FP64
  const double fs = fma((double)F.h, 0x1p-30, (double)F.l * 0x1p-30);
  grid_reduce<double>(fs, 2.0 * tsum, partial, st, normF, normT, mode);
}

// g from the accelerated gradient: 1 + alpha/2 Delta~ (or its exponential) in
// FP64, the Gram-Schmidt on pairs (fx_reunitarize).  In FP64 throughout its 85
// multiply-adds a site bound the kernel; on pairs 25 are left: 32^4 154 -> 54
// us (4.0 TB/s), 16^4 16.9 -> 10.3; with the exponential, which stays FP64 and
// bounds it, 16^3 x 32 takes 75.  Against 80-bit arithmetic, 28 iterations
// of 8^4 leave links off by 3.2e-16 rms (FP64 kernels 4.7e-16; pairs with FP64
// Gram-Schmidt 4.4e-16).  A non-finite g has no pair: the queue stops and is
// reported as not finite.
template <int NC, bool EXACT>
__global__ void __launch_bounds__(128) k_build_g_fx(const cx<double>* __restrict__ D, fx* __restrict__ g, int V,
                                                    double h, DevState* __restrict__ st) {
  pdl_wait();
  if (st->done) return;
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= V) return;
  const cx<double> c0 = ldg(D + s), c1 = ldg(D + V + s), c2 = ldg(D + 2 * V + s), c3 = ldg(D + 3 * V + s);
  M3<double> m;
  if constexpr (EXACT) {
    m = expm_taylor(unpack_ah(c0, c1, c2, c3, h));
  } else {
    m.e[0][0] = mk<double>(1, h * c3.re);
    m.e[0][1] = scale(c0, h);
    m.e[0][2] = scale(c1, h);
    m.e[1][0] = mk<double>(-h * c0.re, h * c0.im);
    m.e[1][1] = mk<double>(1, h * c3.im);
    m.e[1][2] = scale(c2, h);
  }
  fx r[9];
  const bool ok = fx_reunitarize(m, r);
  if (!ok) {
    st->nonfinite = 1;
    st->done = 1;
  }
  if constexpr (NC == 9) {
#pragma unroll
    for (int j = 0; j < 3; ++j) r[6 + j] = fx_row3(r, r + 3, j);
  }
#pragma unroll
  for (int q = 0; q < NC; ++q) g[q * V + s] = r[q];
}

// G(x) <- reunitarised g(x) G(x) in FP64 (LGF_TRACK_G)
template <int NC>
__global__ void __launch_bounds__(128) k_accumulate_fx(cx<double>* G, const fx* __restrict__ g, int V,
                                                       const DevState* __restrict__ st) {
  pdl_wait();
  if (st->done) return;
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= V) return;
  M3<double> a, b, r;
#pragma unroll
  for (int q = 0; q < 6; ++q) {
    const fx x = fx_ldg(g + q * V + s);
    a.e[q / 3][q % 3] = mk<double>(fx_to_double(x.hr, x.lr), fx_to_double(x.hi, x.li));
  }
#pragma unroll
  for (int q = 0; q < NC; ++q) b.e[q / 3][q % 3] = G[q * V + s];
  if constexpr (NC == 6) complete_row3(b);
  mm<double, 2>(r, a, b);
  reunitarize(r);
#pragma unroll
  for (int q = 0; q < NC; ++q) G[q * V + s] = r.e[q / 3][q % 3];
}

// One thread per (site, direction): w = g U row by row, then the row of
// w g'^dag: 216 real multiply-adds per thread as 216 integer and 432 FP32 ones.
//
// Bound by the links' round trip with few threads in flight, so a CTA is 64
// sites of one direction: 1 KB runs in each of the planes, a direction that is
// the same for the whole CTA (its neighbour stride is no select), g from L2 for
// the four CTAs of the same sites that run side by side.  32^4 281 us (1.36 GB,
// 4.8 TB/s); 32 sites x 4 directions in a CTA 307, 128 sites of one direction
// 284, 256 377.  Six CTAs an SM hold all of NC = 9 in registers (eight: 299);
// 12-real storage has room for eight (24^4 81 -> 74 us).
template <int NC>
__global__ void __launch_bounds__(64, NC == 9 ? 6 : 8) k_update_fx(fx* U, const fx* __restrict__ g, const Geom geo,
                                                                   const DevState* __restrict__ st) {
  pdl_wait();
  if (st->done) return;
  const int V = (int)geo.V;
  const int mu = blockIdx.x & 3;
  const int s = (blockIdx.x >> 2) * 64 + threadIdx.x;
  if (s >= V) return;
  int c[4];
  site_coords_r(geo, s, c);
  // selects, not a runtime index: keeps c and the geometry in registers
  const int cm = mu == 0 ? c[0] : mu == 1 ? c[1] : mu == 2 ? c[2] : c[3];
  const int Lm = mu == 0 ? geo.L[0] : mu == 1 ? geo.L[1] : mu == 2 ? geo.L[2] : geo.L[3];
  const int st_mu = mu == 0 ? 1 : mu == 1 ? geo.L[0] : mu == 2 ? geo.L[0] * geo.L[1] : geo.L[0] * geo.L[1] * geo.L[2];
  const int sf = cm < Lm - 1 ? s + st_mu : s - (Lm - 1) * st_mu;
  fx* base = U + mu * NC * V;
  fx u[9], f[9];
#pragma unroll
  for (int q = 0; q < NC; ++q) {
    const int4 v = *reinterpret_cast<const int4*>(base + q * V + s);
    u[q] = {v.x, __int_as_float(v.y), v.z, __int_as_float(v.w)};
  }
  fx_load_m3<NC>(g, V, sf, f);
  if constexpr (NC == 6) {
#pragma unroll
    for (int j = 0; j < 3; ++j) u[6 + j] = fx_row3(u, u + 3, j);
  }
#pragma unroll
  for (int a = 0; a < NC / 3; ++a) {
    fxacc wr[3] = {}, wi[3] = {};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const fx x = fx_ldg(g + (a * 3 + k) * V + s);
      const fxr xr = fx_re(x), xi = fx_im(x), nxi = fx_neg(xi);
#pragma unroll
      for (int b = 0; b < 3; ++b) {
        const fxr yr = fx_re(u[k * 3 + b]), yi = fx_im(u[k * 3 + b]);
        fx_mac(wr[b], xr, yr);
        fx_mac(wr[b], nxi, yi);
        fx_mac(wi[b], xr, yi);
        fx_mac(wi[b], xi, yr);
      }
    }
    fxacc rr[3] = {}, ri[3] = {};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const fx w = fx_round(wr[k], wi[k]);
      const fxr xr = fx_re(w), xi = fx_im(w), nxr = fx_neg(xr);
#pragma unroll
      for (int b = 0; b < 3; ++b) {  // w_k conj(f_bk)
        const fxr yr = fx_re(f[b * 3 + k]), yi = fx_im(f[b * 3 + k]);
        fx_mac(rr[b], xr, yr);
        fx_mac(rr[b], xi, yi);
        fx_mac(ri[b], xi, yr);
        fx_mac(ri[b], nxr, yi);
      }
    }
#pragma unroll
    for (int b = 0; b < 3; ++b) {
      const fx r = fx_round(rr[b], ri[b]);
      *reinterpret_cast<int4*>(base + (a * 3 + b) * V + s) =
          make_int4(r.hr, __float_as_int(r.lr), r.hi, __float_as_int(r.li));
    }
  }
}

// threads per CTA of the one-site-per-thread kernels: as many CTAs as SMs
// before larger CTAs
int site_threads(int64_t V) { return V <= 152 * 32 ? 32 : V <= 152 * 64 ? 64 : 128; }

inline unsigned nblocks(int64_t n, int thr) { return (unsigned)((n + thr - 1) / thr); }

}  // namespace

cudaError_t launch_fx_load(int nc, const void* U64, void* Ufx, int64_t V, DevState* st, cudaStream_t s) {
  const auto u = static_cast<const cx<double>*>(U64);
  auto f = static_cast<fx*>(Ufx);
  if (nc == 9)
    k_fx_load<9><<<nblocks(V, 32), 128, 0, s>>>(u, f, (int)V, st);
  else
    k_fx_load<6><<<nblocks(V, 32), 128, 0, s>>>(u, f, (int)V, st);
  return cudaPeekAtLastError();
}

cudaError_t launch_fx_store(int nc, const void* Ufx, void* U64, int64_t V, const DevState* st, cudaStream_t s) {
  const auto f = static_cast<const fx*>(Ufx);
  auto u = static_cast<cx<double>*>(U64);
  if (nc == 9)
    k_fx_store<9><<<nblocks(V, 32), 128, 0, s>>>(f, u, (int)V, st);
  else
    k_fx_store<6><<<nblocks(V, 32), 128, 0, s>>>(f, u, (int)V, st);
  return cudaPeekAtLastError();
}

cudaError_t launch_gradient_fx(int nc, const void* Ufx, void* D, double2* partial, const Geom& geo, DevState* st,
                               int mode, cudaStream_t s) {
  const double nF = 1.0 / (12.0 * (double)geo.V), nT = 1.0 / (3.0 * (double)geo.V);
  const int thr = site_threads(geo.V);
  const unsigned cap = 152 * kGradFxCtas, full = nblocks(geo.V, thr), nb = full < cap ? full : cap;
  const auto u = static_cast<const fx*>(Ufx);
  auto d = static_cast<cx<double>*>(D);
  if (nc == 9) return launch_pdl(k_gradient_fx<9>, nb, thr, 0, s, u, d, partial, geo, st, mode, nF, nT);
  return launch_pdl(k_gradient_fx<6>, nb, thr, 0, s, u, d, partial, geo, st, mode, nF, nT);
}

cudaError_t launch_build_g_fx(int nc, const void* D, void* g, int64_t V, double half_alpha, bool exact, DevState* st,
                              cudaStream_t s) {
  const int thr = site_threads(V);
  const auto d = static_cast<const cx<double>*>(D);
  auto gp = static_cast<fx*>(g);
  const int v = (int)V;
  if (nc == 9) {
    if (exact) return launch_pdl(k_build_g_fx<9, true>, nblocks(V, thr), thr, 0, s, d, gp, v, half_alpha, st);
    return launch_pdl(k_build_g_fx<9, false>, nblocks(V, thr), thr, 0, s, d, gp, v, half_alpha, st);
  }
  if (exact) return launch_pdl(k_build_g_fx<6, true>, nblocks(V, thr), thr, 0, s, d, gp, v, half_alpha, st);
  return launch_pdl(k_build_g_fx<6, false>, nblocks(V, thr), thr, 0, s, d, gp, v, half_alpha, st);
}

cudaError_t launch_update_fx(int nc, void* Ufx, const void* g, const Geom& geo, const DevState* st, cudaStream_t s) {
  auto u = static_cast<fx*>(Ufx);
  const auto gp = static_cast<const fx*>(g);
  if (nc == 9) return launch_pdl(k_update_fx<9>, 4 * nblocks(geo.V, 64), 64, 0, s, u, gp, geo, st);
  return launch_pdl(k_update_fx<6>, 4 * nblocks(geo.V, 64), 64, 0, s, u, gp, geo, st);
}

cudaError_t launch_accumulate_fx(int nc, void* G, const void* g, int64_t V, const DevState* st, cudaStream_t s) {
  const int thr = site_threads(V);
  auto Gp = static_cast<cx<double>*>(G);
  const auto gp = static_cast<const fx*>(g);
  if (nc == 9) return launch_pdl(k_accumulate_fx<9>, nblocks(V, thr), thr, 0, s, Gp, gp, (int)V, st);
  return launch_pdl(k_accumulate_fx<6>, nblocks(V, thr), thr, 0, s, Gp, gp, (int)V, st);
}

}  // namespace lgf
