"""The plain FP64 iteration on links in fixed-point pairs (k_links_fx.cu), and
its way back to the FP64 links for inputs that do not fit the pairs."""
import numpy as np
import pytest

import lgf_inputs as I
from oracle import lgf_oracle as O

pytestmark = pytest.mark.gpu

ALPHA = 0.08


@pytest.fixture(scope="module")
def lgf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1208_1186_gb300 as P
    from paper_1208_1186_gb300.build import build
    build()
    return P


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (3, 5, 2, 9), (8, 8, 8, 10), (24, 24, 12, 24)])
@pytest.mark.parametrize("dtype", ["f64", "f64_r12"])
@pytest.mark.parametrize("track", [0, 1])
def test_iterations_match_the_oracle(lgf, dims, dtype, track):
    """Below one block, a ragged last block, 64- and 128-thread blocks; the
    parity bound of the FP64 path, 1e-12 per step for three steps."""
    U = I.synthetic_config(dims, seed=3, link_scale=0.4)
    ref = O.iterate(U, 3, ALPHA)
    with lgf.GaugeFixer(dims, dtype) as gf:
        gf.set_param(lgf._lib.LGF_TRACK_G, track)
        gf.load_links(U)
        loaded = gf.store_links()
        gf.iterate(0)
        assert np.array_equal(gf.store_links(), loaded)  # no update: the FP64 links stay
        gf.iterate(3)
        out = gf.store_links()
        assert np.max(np.abs(out - ref)) <= 3e-12
        if track:
            assert np.max(np.abs(I.apply_gauge(U, gf.store_gauge()) - out)) <= 1e-13


@pytest.mark.parametrize("scale", [1.5, 0.5, 4.0])
def test_links_that_do_not_fit_the_pairs_take_the_fp64_kernels(lgf, scale):
    """Rows that are not unit vectors were accepted before and still are; the
    iteration is the oracle's on the same matrices (1e-12 per unit of the
    links' size), alone, through a fix, and in a batch beside links that fit."""
    dims = (4, 6, 4, 5)
    U = I.synthetic_config(dims, seed=4, link_scale=0.3)
    W = U.copy()
    W[2, 1, 3, 0, 2] *= scale  # one link
    ref = O.iterate(W, 2, ALPHA)
    with lgf.GaugeFixer(dims, "f64") as a, lgf.GaugeFixer(dims, "f64") as b:
        a.load_links(W)
        a.iterate(2)
        assert np.max(np.abs(a.store_links() - ref)) <= 1e-12 * max(1.0, scale) ** 2
        a.load_links(W)
        a.fix(1e-30, 2)
        single = a.store_links()
        assert np.max(np.abs(single - ref)) <= 1e-12 * max(1.0, scale) ** 2
        b.load_links(U)
        b.fix(1e-30, 2)
        single_fit = b.store_links()
        a.load_links(W)
        b.load_links(U)
        with lgf.GaugeBatch([a, b]) as batch:
            it, _ = batch.fix(1e-30, 2)
        assert it == [2, 2]
        assert np.array_equal(a.store_links(), single) and np.array_equal(b.store_links(), single_fit)


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_non_finite_links_are_still_reported(lgf, bad):
    dims = (4, 4, 4, 4)
    U = I.synthetic_config(dims, seed=4, link_scale=0.3)
    U[0, 1, 2, 3, 0, 1, 1] = bad
    with lgf.GaugeFixer(dims, "f64") as gf:
        gf.load_links(U)
        with pytest.raises(lgf.LgfError) as e:
            gf.iterate(2)
        assert e.value.status == lgf._lib.LGF_ERR_NONFINITE
        with pytest.raises(lgf.LgfError) as e:
            gf.fix(1e-12, 10)
        assert e.value.status == lgf._lib.LGF_ERR_NONFINITE


@pytest.mark.parametrize("dims,alpha", [((4, 6, 2, 5), 0.125), ((4, 6, 2, 5), 1e-12), ((2, 2, 2, 60), 0.125)])
@pytest.mark.parametrize("dtype", ["f64", "f64_r12"])
def test_gauge_step_of_random_links(lgf, dims, alpha, dtype):
    """Rows of 1 + alpha/2 Delta~ of any length and angle (random links; a long
    axis, whose slow modes are accelerated by up to 10^3): taken relative to one
    or two powers of two more, row 2 close to row 1.  Delta~ is good to some
    1e-15 of its largest entry, and Gram-Schmidt divides by the sine of the
    rows' angle, which stays above 1e-3 on a few hundred sites."""
    U = I.synthetic_config(dims, seed=6, link_scale=3.0)
    ref = O.iterate(U, 1, alpha)
    with lgf.GaugeFixer(dims, dtype, alpha=alpha) as gf:
        gf.load_links(U)
        gf.iterate(1)
        assert np.max(np.abs(gf.store_links() - ref)) <= 3e-12
