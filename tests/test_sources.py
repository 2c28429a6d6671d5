"""Rules of the CUDA sources that no run can show to hold."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1709_04060_b200", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)


def test_kernels_resident_early_use_no_read_only_loads():
    """A kernel launched with programmatic dependent launch lives while the kernel ahead may still write its
    inputs; ld.global.nc is for data that nothing writes during the kernel's whole life."""
    early = [f for f in sorted(os.listdir(CSRC)) if f.endswith(".cuh") or
             (f.endswith(".cu") and re.search(r"launch_pdl\s*[<(]|programmaticStreamSerializationAllowed", _code(f)))]
    assert {"gemv_mma.cu", "pool.cu", "gemm_tc.cu", "conv_direct.cu", "tc_epilogue.cuh"} <= set(early)
    for f in early:
        assert not re.search(r"__ldg\s*\(|\.global(\.\w+)*\.nc\b|__restrict__", _code(f)), f
