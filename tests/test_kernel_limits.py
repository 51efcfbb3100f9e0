"""Shared-memory limits of kernels belong to the device that is current when they
are set, and handles and networks may live on any device of a process: the
limits are raised at creation, never remembered in a variable of the process."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1208_1186_gb300", "csrc")


def _sources():
    return {os.path.basename(f): open(f).read()
            for f in glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cuh"))}


def test_no_cuda_result_is_kept_in_a_static():
    kept = [(name, m.group(0)) for name, text in _sources().items()
            for m in re.finditer(r"\bstatic\b[^;{}()]*=\s*cuda\w+", text)]
    assert not kept, kept


def test_limits_are_raised_by_init_functions_only():
    """Every cudaFuncSetAttribute call stands in a function named *init*, *attr* or *smem*
    (called at creation), none beside a launch."""
    calls = 0
    for name, text in _sources().items():
        for m in re.finditer(r"cudaFuncSetAttribute\(", text):
            heads = re.findall(r"^(?:cudaError_t|static cudaError_t|bool|int)\s+(?:[\w<>, ]+::)?(\w+)\(", text[:m.start()], re.M)
            assert heads and re.search(r"init|attr|smem", heads[-1]), (name, heads[-1:])
            calls += 1
    assert calls >= 15
