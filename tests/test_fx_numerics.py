"""The fixed-point pairs of the plain FP64 iteration (lgf_fx.cuh), emulated in
numpy operation by operation (64-bit integers exactly; an FP32 fused
multiply-add as an FP64 one rounded to FP32, its product being exact in FP64).
One link update g U g'^dagger is compared with extended precision: the pairs
must not be less exact than FP64 matrix products."""
import numpy as np
import pytest

import lgf_inputs as I

f32, f64, i64 = np.float32, np.float64, np.int64


def fma32(a, b, c):
    return (a.astype(f64) * b.astype(f64) + c.astype(f64)).astype(f32)


def from_double(x):
    """fx_from_double: |x| < 2 as h 2^-30 + l 2^-30 (62 fraction bits kept)."""
    F = np.trunc(np.abs(x).astype(np.longdouble) * np.longdouble(2) ** 62).astype(i64)
    F = np.where(x < 0, -F, F)
    h = (F + (1 << 31)) >> 32
    low = (F - (h << 32)).astype(f32)
    return h, (low * f32(2.0 ** -32)).astype(f32)


def fx_round(a, al):
    h = (a + (1 << 29)) >> 30
    rem = a - (h << 30)
    t = ((rem.astype(f32) + al).astype(f32) * f32(2.0 ** -30)).astype(f32)
    k = (t + f32(12582912.0)).astype(f32) - f32(12582912.0)
    return h + k.astype(i64), (t - k).astype(f32)


def value(h, l):
    return (h.astype(np.longdouble) + l.astype(np.longdouble)) * np.longdouble(2) ** -30


def fx_mm(a, b, dag):
    """a b or a b^dagger of (h_re, l_re, h_im, l_im) matrices (n, 3, 3)."""
    n = a[0].shape[0]
    out = [np.zeros((n, 3, 3), dtype=t) for t in (i64, f32, i64, f32)]
    for i in range(3):
        for j in range(3):
            acc = [np.zeros(n, i64), np.zeros(n, f32), np.zeros(n, i64), np.zeros(n, f32)]

            def mac(o, x, y, sign=1):
                (xh, xl), (yh, yl) = x, y
                xh, xl = sign * xh, f32(sign) * xl
                acc[o] = acc[o] + xh * yh
                acc[o + 1] = fma32(xh.astype(f32), yl, fma32(xl, yh.astype(f32), acc[o + 1]))
            for k in range(3):
                xr, xi = (a[0][:, i, k], a[1][:, i, k]), (a[2][:, i, k], a[3][:, i, k])
                p, q = (j, k) if dag else (k, j)
                yr, yi = (b[0][:, p, q], b[1][:, p, q]), (b[2][:, p, q], b[3][:, p, q])
                mac(0, xr, yr)
                mac(0, xi, yi, 1 if dag else -1)
                mac(2, xi, yr) if dag else mac(2, xr, yi)
                mac(2, xr, yi, -1) if dag else mac(2, xi, yr)
            out[0][:, i, j], out[1][:, i, j] = fx_round(acc[0], acc[1])
            out[2][:, i, j], out[3][:, i, j] = fx_round(acc[2], acc[3])
    return out


def pairs(m):
    return [*from_double(m.real), *from_double(m.imag)]


def mm64(a, b):
    """The FP64 kernels' products: fused multiply-adds in the same order."""
    out = np.zeros_like(a)
    for i in range(3):
        for j in range(3):
            re = im = np.zeros(a.shape[0], np.longdouble)
            for k in range(3):
                x, y = a[:, i, k], b[:, k, j]
                xr, xi = x.real.astype(np.longdouble), x.imag.astype(np.longdouble)
                yr, yi = y.real.astype(np.longdouble), y.imag.astype(np.longdouble)
                re = (xr * yr + re).astype(f64).astype(np.longdouble)
                re = (-xi * yi + re).astype(f64).astype(np.longdouble)
                im = (xr * yi + im).astype(f64).astype(np.longdouble)
                im = (xi * yr + im).astype(f64).astype(np.longdouble)
            out[:, i, j] = re.astype(f64) + 1j * im.astype(f64)
    return out


def exact(a, b, c):
    """a b c^dagger in extended precision: (re, im)."""
    def mul(x, y):
        r = np.einsum("nij,njk->nik", x[0], y[0]) - np.einsum("nij,njk->nik", x[1], y[1])
        return r, np.einsum("nij,njk->nik", x[0], y[1]) + np.einsum("nij,njk->nik", x[1], y[0])

    def ext(m):
        return m.real.astype(np.longdouble), m.imag.astype(np.longdouble)
    cr, ci = ext(c)
    return mul(mul(ext(a), ext(b)), (np.swapaxes(cr, 1, 2), -np.swapaxes(ci, 1, 2)))


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 60, reason="needs extended precision")
@pytest.mark.parametrize("scale", [0.01, 0.3, 1.0, 3.0])
def test_update_in_pairs_is_no_less_exact_than_fp64(scale):
    n = 1500
    rng = np.random.default_rng(7)
    U, g, gf = (I.su3_from_coefficients(rng.standard_normal((n, 8)), s) for s in (scale, 0.3, 0.3))
    er, ei = exact(g, U, gf)
    w = fx_mm(pairs(g), pairs(U), dag=False)
    r = fx_mm(w, pairs(gf), dag=True)
    assert np.max(np.abs(r[1])) <= 0.5 and np.max(np.abs(r[3])) <= 0.5
    d_fx = np.concatenate([(value(r[0], r[1]) - er).ravel(), (value(r[2], r[3]) - ei).ravel()]).astype(f64)
    r64 = mm64(mm64(g, U), np.conj(np.swapaxes(gf, 1, 2)))
    d_64 = np.concatenate([(r64.real - er).ravel(), (r64.imag - ei).ravel()]).astype(f64)
    rms = [float(np.sqrt(np.mean(d ** 2))) for d in (d_fx, d_64)]
    # six terms off by at most 2 x 2^5 each in units of 2^-60, twice, and the
    # roundings of the two results: below 2^-51 at the worst
    assert np.max(np.abs(d_fx)) <= 2.0 ** -51
    assert rms[0] <= rms[1], rms


def test_pairs_hold_fp64_numbers_to_2_to_the_minus_55():
    x = np.concatenate([np.random.default_rng(1).uniform(-1.7, 1.7, 20000), [0.0, 1.0, -1.0, 0.5, 2.0 ** -31, 1e-300]])
    h, l = from_double(x)
    assert np.max(np.abs(value(h, l) - x.astype(np.longdouble))) <= np.longdouble(2) ** -55
    assert np.max(np.abs(l)) <= 0.5


def row_from_double(x):
    """fx_row_from_double on (n, 6) real rows: pairs, the norm at most 1.97."""
    top = np.max(np.frexp(x)[1], axis=1) - 1
    while True:
        F = np.trunc(np.ldexp(np.abs(x).astype(np.longdouble), (62 - top)[:, None])).astype(np.longdouble)
        F = np.where(x < 0, -F, F)
        h = np.floor((F + 2 ** 31) / np.longdouble(2) ** 32)
        l = (F - h * np.longdouble(2) ** 32).astype(f32) * f32(2.0 ** -32)
        big = np.sum(h.astype(f64) ** 2, axis=1) > 3.88 * 2.0 ** 60
        if not big.any():
            return h.astype(i64), l
        top = top + big


def mac(a, x, y, sign=1):
    (xh, xl), (yh, yl) = x, y
    xh, xl = sign * xh, f32(sign) * xl
    return a[0] + xh * yh, fma32(xh.astype(f32), yl, fma32(xl, yh.astype(f32), a[1]))


def norm2(h, l):
    """fx_norm2: the squared norm in units of 2^-60."""
    a = (np.zeros(h.shape[0], i64), np.zeros(h.shape[0], f32))
    for j in range(6):
        a = mac(a, (h[:, j], l[:, j]), (h[:, j], l[:, j]))
    return a[0] + 16 * np.rint(a[1] * f32(2.0 ** -4)).astype(i64)


def rsqrt64(n):
    return (1 / np.sqrt(n.astype(np.longdouble))).astype(f64)


def normalize(h, l, n2):
    """fx_normalize."""
    k = from_double(rsqrt64((n2.astype(np.longdouble) * np.longdouble(2) ** -60).astype(f64)))
    z = (np.zeros(h.shape[0], i64), np.zeros(h.shape[0], f32))
    r = [fx_round(*mac(z, (h[:, j], l[:, j]), k)) for j in range(6)]
    h, l = np.stack([a for a, _ in r], 1), np.stack([b for _, b in r], 1)
    c = ((1 << 60) - norm2(h, l)).astype(f32) * f32(2.0 ** -61)
    return h, fma32(h.astype(f32), c[:, None], l)


def reunitarize(m):
    """fx_reunitarize on (n, 2, 6) rows of (re, im) triples: values (n, 2, 6)."""
    u, v = row_from_double(m[:, 0]), row_from_double(m[:, 1])
    u = normalize(*u, norm2(*u))

    def at(r, j):
        return r[0][:, j], r[1][:, j]
    n = m.shape[0]
    pr = pi = (np.zeros(n, i64), np.zeros(n, f32))
    for j in range(3):
        ur, ui, vr, vi = at(u, 2 * j), at(u, 2 * j + 1), at(v, 2 * j), at(v, 2 * j + 1)
        pr = mac(mac(pr, vr, ur), vi, ui)
        pi = mac(mac(pi, vi, ur), vr, ui, -1)
    pr, pi = fx_round(*pr), fx_round(*pi)
    w = []
    for j in range(3):
        ur, ui = at(u, 2 * j), at(u, 2 * j + 1)
        re, im = ((at(v, q)[0] << 30, at(v, q)[1] * f32(2.0 ** 30)) for q in (2 * j, 2 * j + 1))
        w.append(fx_round(*mac(mac(re, pr, ur, -1), pi, ui)))
        w.append(fx_round(*mac(mac(im, pr, ui, -1), pi, ur, -1)))
    w = np.stack([a for a, _ in w], 1), np.stack([b for _, b in w], 1)
    n2 = norm2(*w)
    small = n2 <= 0x428 << 48
    out = value(*normalize(*w, np.where(small, 1 << 60, n2)))
    x = value(*w).astype(f64)
    out[small] = (x * rsqrt64(np.sum(x * x, 1))[:, None])[small]
    return np.stack([value(*u), out], 1)


def gram_schmidt(m, T):
    u = m[:, 0].astype(T)
    u = (u * (1 / np.sqrt(np.sum(u * u, 1).astype(np.longdouble))).astype(T)[:, None]).astype(T)
    v = m[:, 1].astype(T)
    a, b, c, d = u[:, 0::2], u[:, 1::2], v[:, 0::2], v[:, 1::2]
    pr, pi = np.sum(c * a + d * b, 1)[:, None], np.sum(d * a - c * b, 1)[:, None]
    w = np.empty_like(v)
    w[:, 0::2], w[:, 1::2] = c - (pr * a - pi * b), d - (pr * b + pi * a)
    w = w * (1 / np.sqrt(np.sum(w * w, 1).astype(np.longdouble))).astype(T)[:, None]
    return np.stack([u, w], 1)


@pytest.mark.skipif(np.finfo(np.longdouble).nmant < 60, reason="needs extended precision")
@pytest.mark.parametrize("scale", [1e-9, 0.01, 0.3, 1.0, 3.0, 100.0, 1e30])
def test_reunitarisation_in_pairs_is_no_less_exact_than_fp64(scale):
    """Rows of 1 + scale X, X anti-Hermitian: every entry within 2^-50 of the
    exact one times the condition of row 2 (the sine of its angle to row 1),
    and no larger an rms error than Gram-Schmidt in FP64, stored as pairs."""
    n = 4000
    rng = np.random.default_rng(11)
    X = rng.standard_normal((n, 3, 3)) + 1j * rng.standard_normal((n, 3, 3))
    M = np.eye(3) + scale * (X - np.conj(np.swapaxes(X, 1, 2))) / 2
    m = np.empty((n, 2, 6))
    m[:, :, 0::2], m[:, :, 1::2] = M[:, :2].real, M[:, :2].imag
    ref = gram_schmidt(m, np.longdouble)
    d_fx = (reunitarize(m) - ref).astype(f64)
    # the FP64 rows as the kernel stores them
    d_64 = (value(*from_double(gram_schmidt(m, f64))) - ref).astype(f64)
    u, v = M[:, 0], M[:, 1]
    cos2 = np.abs(np.sum(np.conj(u) * v, 1)) ** 2 / (np.sum(np.abs(u) ** 2, 1) * np.sum(np.abs(v) ** 2, 1))
    sine = np.sqrt(np.maximum(1 - cos2, 1e-300))
    assert np.all(np.max(np.abs(d_fx), axis=(1, 2)) * sine <= 2.0 ** -50)
    well = sine > 0.1
    rms = [float(np.sqrt(np.mean(d[well] ** 2))) for d in (d_fx, d_64)]
    # or the rounding of a number to the pairs' resolution, 2^-55
    assert rms[0] <= max(rms[1], 2.0 ** -55 / 12 ** 0.5), rms
