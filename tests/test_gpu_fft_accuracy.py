"""FP64 accelerated gradients against the same in extended precision, as an rms
relative to the result's.  Lines up to 32 (64-bit block floating point): three
stores to FP64 round by 2^-53 / sqrt(3) each at most, 1.1e-16 together, the factor
as much again at worst; everything between keeps more bits.  2e-16 is what that
leaves, 2.5e-16 where the longest line is four times the shortest.  With x-y lines
above 32 (FP64, some dozen roundings of a line) the bound is what the FP64 stages in
shared memory left that ran before, plus a tenth: the z-t pass beside them must
not add to it."""
import numpy as np
import pytest

import lgf_inputs as I

pytestmark = pytest.mark.gpu
CASES = [((8, 8, 8, 8), 2e-16), ((12, 18, 10, 20), 2e-16), ((16, 16, 16, 16), 2e-16), ((27, 27, 6, 9), 2.5e-16),
         ((32, 32, 8, 8), 2.5e-16), ((24, 24, 24, 12), 2e-16),
         ((36, 36, 8, 6), 6.6e-16), ((40, 40, 10, 10), 6.1e-16), ((48, 48, 8, 8), 7.2e-16), ((50, 10, 6, 9), 9.7e-16)]


@pytest.fixture(scope="module")
def lgf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1208_1186_gb300 as P
    from paper_1208_1186_gb300.build import build
    build()
    return P


@pytest.mark.parametrize("dims,bound", CASES)
def test_error_against_extended_precision(lgf, dims, bound):
    fft = pytest.importorskip("scipy.fft")
    p2 = 0
    for a, L in enumerate(dims):
        s = 4 * np.sin(4 * np.arctan(np.longdouble(1)) * np.arange(L) / np.longdouble(L)) ** 2
        p2 = p2 + s.reshape([L if i == 3 - a else 1 for i in range(4)])
    K = p2.max() / np.where(p2 > 0, p2, 1)
    K[0, 0, 0, 0] = 0
    err = []
    with lgf.GaugeFixer(dims, "f64") as gf:
        for seed in range(3):
            gf.load_links(I.synthetic_config(dims, seed=seed, link_scale=0.5))
            p = gf.probe()
            for f in range(4):
                want = fft.ifftn(K * fft.fftn(p["delta"][..., f].astype(np.clongdouble)))
                err.append(float(np.mean(np.abs(p["delta_tilde"][..., f] - want) ** 2) / np.mean(np.abs(want) ** 2)))
    assert np.sqrt(np.mean(err)) <= bound
