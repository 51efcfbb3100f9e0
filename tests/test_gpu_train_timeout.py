"""A training step whose convolutions give up a bounded wait (a stage-wait budget
of 0, as in tests/test_gpu_warm.py) leaves the network as it was: parameters bit
for bit, and the step after it is the network's first.  Adam's first step moves
a weight by lr g / (|g| + 1e-12); a second one whose moments hold only one
gradient would move it by 0.74 of that, and the gradient's last bits, which vary
from run to run, change the sign of the few weights whose gradient is rounding
alone."""
import numpy as np
import pytest

from .test_gpu_warm import _setup, lgf  # noqa: F401

pytestmark = pytest.mark.gpu
LR = 1e-5


def test_a_timed_out_step_changes_nothing(lgf):  # noqa: F811
    from paper_1208_1186_gb300._lib import LGF_ERR_TIMEOUT
    _, _, gf, net, p0 = _setup(lgf, (4, 6, 4, 8), 9)
    try:
        F0, _ = net.train_step(gf, 0.0)  # activations of a step before, then no change
        assert np.array_equal(net.get_params(), p0)
        net.set_wait_budget(0)
        for _ in range(2):
            with pytest.raises(lgf.LgfError) as e:
                net.train_step(gf, LR)
            assert e.value.status == LGF_ERR_TIMEOUT
            assert np.array_equal(net.get_params(), p0)
        net.set_wait_budget(-1)
        F1, _ = net.train_step(gf, LR)
        assert F1 == F0
        after = net.get_params()
        net.set_params(p0)
        net.train_step(gf, LR)
        first = net.get_params()
        assert np.mean(np.abs(after - p0) > 0.5 * LR) > 0.5
        assert np.mean(np.abs(after - first) > 0.1 * LR) < 0.01
    finally:
        net.close()
        gf.close()
