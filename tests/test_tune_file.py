"""The product tuner's text file (ruqlp_tune_file) and what its kernels may
use: CPU only, nothing is launched."""
import glob
import os

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def lib():
    import __graft_entry__ as g
    g.build()
    from paper_2209_12464_gb300 import ruqlp
    return ruqlp


@pytest.mark.parametrize("line,loaded", [
    ("tc_gemm 0 0 911 457 32 1 4 12.5", 1),
    ("tc_gemm 1 1 911 457 64 2 3 12.5", 1),
    ("tc_gemm 0 0 912 457 32 1 68 12.5", 0),   # a CTA-pair choice of an older library
    ("tc_gemm 1 0 912 457 224 1 69 12.5", 0),
    ("tc_gemm 0 0 912 457 32 3 4 12.5", 0),    # no such split
    ("tc_gemm 0 0 912 457 224 1 9 12.5", 0),   # a ring that does not fit
])
def test_lines_of_other_configurations_are_skipped(lib, tmp_path, line, loaded):
    f = tmp_path / "tune.txt"
    f.write_text(line + "\n")
    try:
        assert lib.ruqlp_tune_file(str(f)) == loaded
    finally:
        lib.ruqlp_tune_file(None)


def test_no_multicast_loads():
    """Every rank of a multi-GPU run uses this library, and multicast loads are
    for one-GPU programs only: each CTA fetches its tiles itself."""
    for p in glob.glob(os.path.join(ROOT, "paper_2209_12464_gb300", "csrc", "*")):
        assert ".multicast::cluster" not in open(p).read(), p
