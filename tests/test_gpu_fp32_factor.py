"""The FP32 acceleration factor p2_max / p2(k) of shapes without tuned z-t kernels
is rounded once.  Links that are one diagonal plane wave, a(x) = A cos(k x + phase)
in one direction, have a gradient of modes +-k (and odd harmonics), so the ratio of
the accelerated gradient to the gradient in mode k shows the factor.  The modes are
those where an FP32 sum, reciprocal and product would be worst, 1.5e-7 to 2e-7 off;
rounded once it is off by at most 2^-24 = 6e-8.  The mode's coefficient passes about
eight roundings of its own in the transforms (2^-25 rms each, 8.5e-8 together), which
change with phase and amplitude: over 64 waves their mean is 1.1e-8, four times which
is allowed for."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lgf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1208_1186_gb300 as P
    from paper_1208_1186_gb300.build import build
    build()
    return P


def momenta(dims):
    """4 sin^2 per axis, and p2 of every mode (kx, ky, kz, kt) in FP64"""
    s = [4 * np.sin(np.pi * np.arange(L) / L) ** 2 for L in dims]
    return s, s[0][:, None, None, None] + s[1][:, None, None] + s[2][:, None] + s[3]


def worst_modes(dims, n):
    f = np.float32
    s, p2 = momenta(dims)
    h = [x.astype(f) for x in s]
    p = ((h[0][:, None, None] + h[1][:, None]) + h[2])[..., None] + h[3]
    with np.errstate(divide="ignore", invalid="ignore"):
        k = (f(p2.max()) * (1 / p.astype(np.float64)).astype(f)).astype(np.float64)
        err = np.abs(k * p2 / p2.max() - 1)
    err[0, 0, 0, 0] = 0
    return [np.unravel_index(i, err.shape) for i in np.argsort(err.ravel())[::-1][:n]]


# run-time z-t planes (both classes), pairs of common extents
@pytest.mark.parametrize("dims", [(6, 10, 9, 5), (3, 10, 9, 45), (6, 10, 10, 12), (5, 6, 18, 20)])
def test_factor_is_rounded_once(lgf, dims):
    Lx, Ly, Lz, Lt = dims
    V = int(np.prod(dims))
    _, p2 = momenta(dims)
    site = np.indices((Lt, Lz, Ly, Lx))[::-1]  # x, y, z, t
    rng = np.random.default_rng(1)
    U = np.zeros((Lt, Lz, Ly, Lx, 4, 3, 3), dtype=np.complex128)
    with lgf.GaugeFixer(dims, "f32") as gf:
        for k in worst_modes(dims, 6):
            mu = max(range(4), key=lambda a: np.sin(np.pi * k[a] / dims[a]) ** 2)
            kx = 2 * np.pi * sum(k[i] * site[i] / dims[i] for i in range(4))
            wave = np.exp(-1j * kx)
            factor = []
            for _ in range(64):
                a = 0.01 * 2 ** rng.random() * np.cos(kx + 2 * np.pi * rng.random())
                U[...] = np.eye(3)
                U[..., mu, 0, 0], U[..., mu, 1, 1] = np.exp(1j * a), np.exp(-1j * a)
                gf.load_links(U)
                p = gf.probe()
                D, T = (np.sum(wave * p[q][..., 3].real) for q in ("delta", "delta_tilde"))  # Im Delta_00
                if abs(D) > 1e-4 * V:  # (a mode that is its own -k vanishes at some phases)
                    factor.append((T / D).real)
            assert len(factor) >= 32
            err = np.mean(factor) * p2[k] / p2.max() - 1
            assert abs(err) <= 2.0 ** -24 + 4 * 8.5e-8 / np.sqrt(len(factor)), (k, err)
