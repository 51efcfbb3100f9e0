"""lgf_batch_autotune times what the batch then runs: plain FP64 members on their
links in fixed-point pairs.  Its updates are applied, so the links after it are
those of the same queues of updates on a single handle, bit for bit (the FP64
kernels round differently); a member whose links do not fit the pairs is tuned
and updated on its FP64 links."""
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


@pytest.mark.parametrize("dtypes", [("f64", "f64"), ("f64_r12", "f64"), ("f64", "f32")])
def test_tuning_updates_are_those_of_the_iteration(lgf, dtypes):
    dims = [(4, 6, 4, 5), (8, 8, 6, 4), (4, 4, 4, 4)]
    dtypes = dtypes + ("f64",)
    reps = 3
    queues = 2 * len([c for c in (1, 2, 4, 8, 16, 0) if c <= len(dims)])
    U = [I.synthetic_config(d, seed=21 + i, link_scale=0.4) for i, d in enumerate(dims)]
    U[2][1, 2, 3, 0, 1] *= 1.5  # one link that does not fit the pairs
    want = []
    for d, t, u in zip(dims, dtypes, U):
        with lgf.GaugeFixer(d, t) as gf:
            gf.load_links(u)
            for _ in range(queues):
                gf.iterate(reps)
            want.append(gf.store_links())
    fixers = [lgf.GaugeFixer(d, t) for d, t in zip(dims, dtypes)]
    try:
        for gf, u in zip(fixers, U):
            gf.load_links(u)
        with lgf.GaugeBatch(fixers) as batch:
            batch.autotune(reps)
            for gf, w in zip(fixers, want):
                assert np.array_equal(gf.store_links(), w)
            # the batch still runs, and alone each member as well
            batch.iterate(reps)
        for gf, d, t, w in zip(fixers, dims, dtypes, want):
            with lgf.GaugeFixer(d, t) as one:
                one.load_links(w)
                one.iterate(reps)
                if t.startswith("f64"):
                    assert np.array_equal(gf.store_links(), one.store_links())
    finally:
        for gf in fixers:
            gf.close()
