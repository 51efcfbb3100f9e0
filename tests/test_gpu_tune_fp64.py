"""The schedule tuner on FP64 handles: pipelines 1 and 3 and every tile width are
the same kernels there, so what it returns is the default of them or the per-axis
passes, never a choice among equals.  Saved FP64 schedules of other widths still
apply."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lgf():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1208_1186_gb300 as P
    from paper_1208_1186_gb300.build import build
    build()
    P._lib.load().lgf_tune_clear()
    yield P
    P._lib.load().lgf_tune_clear()


@pytest.mark.parametrize("dims,default", [((16, 16, 16, 16), 3), ((32, 32, 8, 8), 3), ((10, 6, 4, 18), 1)])
def test_no_choice_among_equal_schedules(lgf, dims, default):
    for _ in range(6):
        lgf._lib.load().lgf_tune_clear()
        with lgf.GaugeFixer(dims, "f64") as gf:
            chosen = gf.autotune(reps=2)
            assert gf.schedule() == (chosen, 0, 0) and chosen in (2, default)
    if default == 3:
        with lgf.GaugeFixer(dims, "f64") as gf:
            gf.set_schedule(3, 4, 0)
            assert gf.schedule() == (3, 4, 0)
