"""lgf_store_gauge moves chunks of 64 matrices through shared memory: lattices
below one chunk, at a whole number of chunks and with a ragged last chunk, in
every storage form, into pinned memory (written directly) and pageable memory
(through the staging buffer).

G U_loaded G(x+mu)^dagger must be the stored links.  FP64 handles: both are
products of FP64 rounding, 1e-13.  Mixed handles before the tail: the links are
formed from FP32 G and U, entries |u| <= 1 with 2 x 3 complex products of FP32
rounding 6e-8 each, bounded by 3e-6; after the double-float tail 1e-11, the
tail's own link accuracy (1e-12) times the six products."""
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


def _links_of(G, U):
    return I.apply_gauge(U, G)


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 4, 2, 2), (4, 4, 4, 4), (3, 5, 2, 9)])
@pytest.mark.parametrize("dtype", ["f64", "f64_r12", "f32", "f32_r12"])
def test_store_gauge_chunks(lgf, dims, dtype):
    import torch
    U = I.synthetic_config(dims, seed=5, link_scale=0.3)
    with lgf.GaugeFixer(dims, dtype) as gf:
        if dtype.startswith("f64"):
            gf.set_param(lgf._lib.LGF_TRACK_G, 1)
        gf.load_links(U)
        gf.iterate(3)
        tol = 1e-13 if dtype.startswith("f64") else 3e-6
        for _ in range(2):
            G = gf.store_gauge()
            pinned = torch.empty(G.shape, dtype=torch.complex128, pin_memory=True)
            gf.store_gauge(pinned.numpy())
            assert np.array_equal(pinned.numpy(), G)
            assert np.max(np.abs(_links_of(G, U) - gf.store_links())) <= tol
            if dtype.startswith("f64"):
                break
            assert gf.fix(1e-15, 2000)[1]
            tol = 1e-11
