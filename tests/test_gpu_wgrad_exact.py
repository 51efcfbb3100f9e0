"""The weight-gradient kernel (k_wgrad_tc) on caller-held operands, element by
element.  x and gy are multiples of 1/4 in [-1, 1]: every product is a multiple
of 1/16, every sum over sites below 2^15, so FP32 sums are exact in any order and
a row that is dropped, doubled or misplaced anywhere shows.  The kernel walks the
rows of the lattice with a halo in x and y, (Lx + 2)(Ly + 2) Lz Lt, in stages of
64 that several CTAs share: whole stages and remainders of 1 and 63 rows, from
fewer stages than the pipeline holds to more CTAs than one per four stages.  The
padding channels 8..15 of layer 3's gradient hold numbers that must not count."""
import numpy as np
import pytest

from oracle import warm_start_oracle as WO
import lgf_inputs as I

from .test_gpu_warm import lgf  # noqa: F401

DIMS = [
    (2, 2, 2, 2),     # 64 rows: one full stage
    (2, 2, 2, 3),     # 96: two stages
    (2, 2, 2, 5),     # 160: three
    (2, 2, 4, 5),     # 320: five full ones
    (3, 3, 7, 15),    # 2625 = 41 x 64 + 1
    (3, 3, 3, 29),    # 2175 = 33 x 64 + 63
    (7, 5, 3, 3),     # odd extents, 567 rows
    (16, 16, 8, 9),   # 23328 = 364 x 64 + 32, as many CTAs as a layer takes
    (64, 2, 3, 2),    # the longest rows
]


def test_shapes_cover_the_stage_remainders():
    rows = [(d[0] + 2) * (d[1] + 2) * d[2] * d[3] for d in DIMS]
    assert {1, 63, 0, 32} <= {r % 64 for r in rows}
    assert {1, 2, 3, 5} <= {-(-r // 64) for r in rows}
    assert max(int(np.prod(d)) for d in DIMS) <= 1 << 15


def test_null_network_is_rejected():
    from paper_1208_1186_gb300 import _lib
    from paper_1208_1186_gb300.build import build
    build()
    assert _lib.load().lgf_net_conv_weight_grad(None, 1, None, None, None, 8, 8, 8, 8, None) == _lib.LGF_ERR_ARG


@pytest.mark.gpu
def test_bad_arguments_are_rejected(lgf):  # noqa: F811
    import torch
    net = lgf.WarmStartNet(seed=1)
    try:
        x = torch.zeros((16, 48), dtype=torch.bfloat16, device="cuda")
        out = torch.zeros(81 * 48 * 32, device="cuda")
        call = net.lib.lgf_net_conv_weight_grad
        p = x.data_ptr()
        for layer, a, b, c, dims in [(0, p, p, out.data_ptr(), (2, 2, 2, 2)), (4, p, p, out.data_ptr(), (2, 2, 2, 2)),
                                     (1, None, p, out.data_ptr(), (2, 2, 2, 2)), (1, p, p, None, (2, 2, 2, 2)),
                                     (1, p, p, out.data_ptr(), (1, 2, 2, 2)), (1, p, p, out.data_ptr(), (2, 2, 2, 65))]:
            assert call(net.n, layer, a, b, c, *dims, None) == lgf._lib.LGF_ERR_ARG
    finally:
        net.close()


@pytest.mark.gpu
@pytest.mark.parametrize("layer", [1, 2, 3])
@pytest.mark.parametrize("dims", DIMS)
def test_weight_gradient_is_exact_on_dyadic_operands(lgf, layer, dims):  # noqa: F811
    import torch
    nin, nout = {1: (48, 32), 2: (32, 32), 3: (32, 8)}[layer]
    shp = I.lattice_shape(dims)
    V = int(np.prod(dims))
    rng = np.random.default_rng(50 + layer)
    x = rng.integers(-4, 5, (V, nin)) / 4
    gy = rng.integers(-4, 5, (V, max(nout, 16))) / 4
    net = lgf.WarmStartNet(seed=1)
    try:
        xt, gt = (torch.tensor(a, dtype=torch.float32).to(torch.bfloat16).cuda() for a in (x, gy))
        got = net.conv_weight_grad(layer, xt, gt, dims).cpu().numpy()
    finally:
        net.close()
    _, ref, _ = WO.conv_backward(x.reshape(shp + (nin,)), np.zeros((81, nin, nout)),
                                 gy[:, :nout].reshape(shp + (nout,)))
    assert np.array_equal(got, ref)
