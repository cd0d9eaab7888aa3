"""Properties of the CUDA sources that no single run shows: CUDA's FP64
reciprocal, division and roots are called, not rebuilt from the approximation
instructions under them, and a kernel's limit of dynamic shared memory, which all
host threads share, is never set to the size of one launch."""
import glob
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def _lines(what):
    found = []
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_1102_4666_gb300", "csrc", "*"))):
        with open(path) as f:
            found += [(os.path.basename(path), line.strip()) for line in f if what in line]
    return found


def test_no_fp64_approximation_instructions():
    assert _lines("approx.ftz.f64") == []


def test_shared_memory_limits_are_constants():
    """Set in one place only, where the size is a template argument."""
    assert _lines("cudaFuncAttributeMaxDynamicSharedMemorySize") == [
        ("common.cuh", "return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, BYTES);")]
