"""CUDA's FP64 reciprocal, division and roots are called, not rebuilt from the
approximation instructions under them."""
import glob
import os

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


def test_no_fp64_approximation_instructions():
    found = []
    for path in sorted(glob.glob(os.path.join(ROOT, "paper_1102_4666_gb300", "csrc", "*"))):
        with open(path) as f:
            found += [(os.path.basename(path), i) for i, line in enumerate(f, 1) if "approx.ftz.f64" in line]
    assert found == []
