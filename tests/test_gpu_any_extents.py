"""The plane passes of any extents (pipeline 1) over every line length and every
way a pass is dispatched: x-y planes of equal extents with their own kernel
(one warp, two warps; several tiles per warp, idle lanes), run-time x-y planes
(several tiles per CTA, one tile, both register classes), z-t planes by pair
(8- and 4-column runs, a ragged last run, odd Lx), run-time z-t planes (both
classes), and the fused inverse x-y + G update behind them.

Against the oracle: FP64 at 1e-12 of the largest entry, FP32 at 4e-6 of it (a
forward and inverse FP32 FFT over V points has error of order eps log2 V
relative to its largest entry), and FP32 links after ten updates at 2e-5, the
bounds of tests/test_gpu_parity.py."""
import numpy as np
import pytest

import lgf_inputs as I
from oracle import lgf_oracle as O

pytestmark = pytest.mark.gpu

ALPHA = 0.08
DIMS = [
    (10, 10, 4, 18), (18, 18, 2, 30), (30, 30, 4, 4), (36, 36, 4, 2), (40, 40, 2, 4),  # x-y planes of equal extents
    (2, 27, 3, 25), (45, 2, 5, 9), (50, 4, 2, 54), (4, 60, 2, 2), (64, 64, 2, 2), (3, 3, 3, 3),
    (15, 20, 9, 5), (9, 2, 40, 36), (6, 4, 32, 64), (5, 3, 64, 10), (5, 5, 8, 6), (3, 2, 64, 64),
    (12, 30, 20, 16), (24, 18, 10, 12),
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
    U = I.synthetic_config(dims, seed=17, link_scale=0.5)
    want = O.pack_delta(O.step_parts(U, ALPHA)["Delta_tilde"])
    n = 10 if dtype == "f32" else 2
    ref = O.iterate(U, n, ALPHA)
    big = np.max(np.abs(want))
    with lgf.GaugeFixer(dims, dtype) as gf:
        for pipeline in (0, 1):
            gf.set_param(lgf._lib.LGF_FFT_PIPELINE, pipeline)
            gf.load_links(U)
            got = gf.probe()["delta_tilde"]
            assert np.max(np.abs(got - want)) <= (4e-6 if dtype == "f32" else 1e-12) * big
            gf.load_links(U)
            gf.iterate(n)
            assert np.max(np.abs(gf.store_links() - ref)) <= (2e-5 if dtype == "f32" else 1e-12 * n)
