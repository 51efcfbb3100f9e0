"""The plane passes in two steps a line (k_fft_long.cu): every length above 32 on
every axis in FP64, planes of few long lines and long x-y lines in FP32, several
tiles a CTA with a partial last one, ragged last runs of columns, lines of one step
(16 and less) beside lines of two.  Against the oracle: FP64 at 1e-12 of the largest
entry, FP32 at 4e-6 of it (a forward and inverse FP32 FFT over V points has error of
order eps log2 V relative to its largest entry), the bounds of
tests/test_gpu_any_extents.py; and the links after three updates."""
import numpy as np
import pytest

import lgf_inputs as I
from oracle import lgf_oracle as O

pytestmark = pytest.mark.gpu
ALPHA = 0.08
DIMS = [
    (36, 5, 2, 2), (40, 3, 2, 4), (45, 2, 2, 3), (48, 3, 2, 2), (50, 2, 3, 2), (54, 2, 2, 2), (60, 2, 2, 2), (64, 3, 2, 2),
    (2, 36, 2, 3), (3, 40, 2, 2), (2, 45, 3, 2), (2, 54, 2, 2), (5, 64, 2, 2), (36, 40, 2, 2),
    (3, 3, 36, 2), (5, 3, 2, 40), (3, 3, 45, 4), (2, 3, 3, 48), (3, 5, 50, 2), (3, 3, 54, 3), (3, 5, 2, 60), (5, 5, 64, 2),
    (15, 9, 25, 3), (9, 25, 3, 20), (10, 10, 2, 45), (48, 10, 9, 10), (3, 64, 10, 12),
]


@pytest.fixture(scope="module")
def lgf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1208_1186_gb300 as P
    from paper_1208_1186_gb300.build import build
    build()
    return P


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_acceleration_and_updates_match_the_oracle(lgf, dims, dtype):
    U = I.synthetic_config(dims, seed=19, link_scale=0.5)
    want = O.pack_delta(O.step_parts(U, ALPHA)["Delta_tilde"])
    ref = O.iterate(U, 3, ALPHA)
    with lgf.GaugeFixer(dims, dtype) as gf:
        gf.load_links(U)
        got = gf.probe()["delta_tilde"]
        assert np.max(np.abs(got - want)) <= (1e-12 if dtype == "f64" else 4e-6) * np.max(np.abs(want))
        gf.iterate(3)
        assert np.max(np.abs(gf.store_links() - ref)) <= (3e-12 if dtype == "f64" else 2e-5)
