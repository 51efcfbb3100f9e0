"""Tolerances that FP64 links reach and fixed-point pairs (absolute resolution
2^-55, theta no lower than 1e-31) do not: a plain FP64 fix still converges to
them, alone, in a batch and with profiling on.  On FP64 links theta falls by more
than ten per update on fields near the identity, whose small entries keep their
relative precision, and stops near 6e-33 at 8^4 on rough ones."""
import numpy as np
import pytest

import lgf_inputs as I

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


@pytest.mark.parametrize("dims,link,gauge,tol", [((8, 8, 8, 8), 1e-3, 1.0, 1e-33), ((4, 6, 4, 10), 1e-8, 1e-3, 1e-36),
                                                 ((8, 8, 8, 8), 0.3, 1.0, 2e-32)])
@pytest.mark.parametrize("dtype", ["f64", "f64_r12"])
def test_fix_reaches_tolerances_below_the_pairs_floor(lgf, dims, link, gauge, tol, dtype):
    if dtype == "f64_r12" and tol > 1e-33:
        pytest.skip("row 3 from rounded rows: the rough field's floor lies near the tolerance")
    U = I.synthetic_config(dims, seed=8, link_scale=link, gauge_scale=gauge)
    with lgf.GaugeFixer(dims, dtype) as gf, lgf.GaugeFixer(dims, dtype) as other:
        for profile in (False, True):
            gf.load_links(U)
            gf.profile(profile)
            it, conv = gf.fix(tol, 200)
            gf.profile(False)
            F, theta = gf.functional()
            assert conv and theta < 2 * tol
        single = gf.store_links()
        gf.load_links(U)
        other.load_links(U)
        with lgf.GaugeBatch([gf, other]) as batch:
            its, convs = batch.fix(tol, 200)
        assert all(convs) and its == [it, it]
        assert np.array_equal(gf.store_links(), single) and np.array_equal(other.store_links(), single)
