"""The weight gradients on the tensor cores (k_wgrad_tc) where their tiling can
go wrong: a single stage of 64 rows, a last stage that is nearly empty, fewer
stages than the pipeline holds, odd extents, extents of 2 (both neighbours the
same site), and a lattice whose rows are split over many CTAs.  Against the
oracle with BF16 storage emulated, at the tolerances of tests/test_gpu_warm.py:
5e-2 in norm and a cosine above 0.99 for each layer, biases within 1e-2 of the
magnitude that cancels.  A tap or a channel in the wrong place would leave the
cosine near zero."""
import numpy as np
import pytest

from oracle import warm_start_oracle as WO

from .test_gpu_warm import _setup, bf16, lgf, oracle_forward_bf16, relnorm, unpack  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims", [(2, 2, 2, 2), (4, 2, 2, 3 * 3 + 1 + 6), (3, 4, 4, 5), (16, 3, 5, 2), (6, 10, 4, 4),
                                  (8, 8, 8, 8)])
def test_weight_gradients_at_tile_edges(lgf, dims):  # noqa: F811
    U, U32, gf, net, p = _setup(lgf, dims, 31)
    try:
        c = net.forward(gf).astype(np.float64)
        _, grad = net.train_step(gf, 0.0, want_grad=True)
        _, gc = WO.loss_and_signal(U32, c)
        _, (x0, z1, a1, z2, a2), pb = oracle_forward_bf16(U32, unpack(p))
        gc16 = bf16(gc)
        ga2, gW3, gb3 = WO.conv_backward(a2, pb[2][0], gc16)
        gz2 = bf16(ga2 * (a2 > 0))
        ga1, gW2, gb2 = WO.conv_backward(a1, pb[1][0], gz2)
        gz1 = bf16(ga1 * (a1 > 0))
        _, gW1, gb1 = WO.conv_backward(x0, pb[0][0], gz1)
        for (gW, gb), rW, rb, up in zip(unpack(grad), (gW1, gW2, gW3), (gb1, gb2, gb3), (gz1, gz2, gc16)):
            assert relnorm(gW, rW) < 5e-2
            assert float(np.sum(gW * rW) / (np.linalg.norm(gW) * np.linalg.norm(rW))) > 0.99
            scale = np.abs(up).sum(axis=(0, 1, 2, 3))[: rb.size]
            assert np.all(np.abs(gb - rb) <= 1e-2 * scale + 1e-12)
    finally:
        net.close()
        gf.close()
