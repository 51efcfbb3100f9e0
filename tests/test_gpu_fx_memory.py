"""The fixed-point pairs of plain FP64 handles are optional memory: on a device
with room for everything else only, every call works as it did without them (on
the FP64 kernels), because any allocation that finds no room takes the pairs of
an idle handle back.  The room is limited by allocator hooks that count."""
import threading

import numpy as np
import pytest

import lgf_inputs as I

pytestmark = pytest.mark.gpu
DIMS = (8, 8, 8, 8)
V = 8 ** 4


@pytest.fixture(scope="module")
def lgf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1208_1186_gb300 as P
    from paper_1208_1186_gb300.build import build
    build()
    return P


class Room:
    """Allocator hooks of the library that hand out at most cap bytes at a time."""

    def __init__(self, lgf):
        import torch
        self.lib = lgf._lib.load()
        lgf._lib.use_torch_allocator()
        self.plain = lgf._lib._torch_hooks
        self.cap, self.held, self.used, self.refused = None, {}, 0, 0

        def alloc(n, device, stream, user):
            if self.cap is not None and self.used + n > self.cap:
                self.refused += 1
                return None
            p = torch.cuda.caching_allocator_alloc(int(n), int(device), int(stream or 0))
            self.held[p] = n
            self.used += n
            return p

        def free(p, n, device, stream, user):
            assert self.held.pop(p) == n
            self.used -= n
            torch.cuda.caching_allocator_delete(int(p))

        self.hooks = (lgf._lib.ALLOC_FN(alloc), lgf._lib.FREE_FN(free))

    def __enter__(self):
        assert self.lib.lgf_set_allocator(*self.hooks, None) == 0
        return self

    def __exit__(self, *exc):
        assert self.lib.lgf_set_allocator(*self.plain, None) == 0
        assert self.used == 0 and not self.held


def everything(lgf, n, U, dtype="f64"):
    """n handles, each taken through the calls that allocate; their fixed links."""
    out = []
    fixers = []
    try:
        for _ in range(n):
            gf = lgf.GaugeFixer(DIMS, dtype)
            fixers.append(gf)
            gf.set_param(lgf._lib.LGF_TRACK_G, 1)
            gf.load_links(U)  # pageable: the staging buffer
        for gf in fixers:
            gf.fix(1e-12, 200)
            gf.iterate(1)
            out.append(gf.store_links())
        if n > 1:
            with lgf.GaugeBatch(fixers) as batch:
                batch.iterate(1)
    finally:
        for gf in fixers:
            gf.close()
    return out


@pytest.mark.parametrize("n", [1, 3])
@pytest.mark.parametrize("dtype", ["f64", "f64_r12"])
def test_what_fitted_without_the_pairs_still_fits(lgf, n, dtype):
    U = I.synthetic_config(DIMS, seed=2, link_scale=0.4)
    pairs = 4 * (6 if dtype == "f64_r12" else 9) * V * 16
    with Room(lgf) as room:
        peak = [0]
        inner = room.hooks[0]

        def counting(nb, d, s, u):
            p = inner(nb, d, s, u)
            peak[0] = max(peak[0], room.used)
            return p

        hook = lgf._lib.ALLOC_FN(counting)
        assert room.lib.lgf_set_allocator(hook, room.hooks[1], None) == 0
        ref = everything(lgf, n, U, dtype)
        assert room.used == 0
        room.cap = peak[0] - n * pairs  # all but the pairs
        got = everything(lgf, n, U, dtype)
        assert room.refused > 0
        for a, b in zip(got, ref):  # the FP64 kernels, about 26 updates at the parity bound of one
            assert np.max(np.abs(a - b)) <= 3e-11
        room.cap -= 1  # less than that is out of memory as ever
        with pytest.raises(lgf.LgfError) as e:
            everything(lgf, n, U, dtype)
        assert e.value.status == lgf._lib.LGF_ERR_OOM


def test_pairs_in_use_by_another_thread_are_waited_for(lgf):
    U = I.synthetic_config(DIMS, seed=2, link_scale=0.4)
    with Room(lgf) as room:
        with lgf.GaugeFixer(DIMS, "f64") as a:
            a.load_links(U)
            a.iterate(600)
            want = a.store_links()
            a.load_links(U)
            need = room.used
            room.cap = need  # the second handle fits only in the first one's pairs and no further
            t = threading.Thread(target=a.iterate, args=(600,))
            t.start()
            try:
                with lgf.GaugeFixer((4, 4, 4, 4), "f64") as b:
                    b.load_links(U[:4, :4, :4, :4].copy())
                    b.iterate(2)
            finally:
                t.join()
            got = a.store_links()
            # the call ran on the pairs throughout, or on FP64 links throughout if they were taken first
            assert np.array_equal(got, want) or np.max(np.abs(got - want)) <= 600 * 1e-12
            a.iterate(1)
