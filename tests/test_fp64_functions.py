"""The FP64 functions of the kernels are CUDA's own: no source forms a square root,
reciprocal or quotient in FP64 from the hardware's approximate instructions."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2606_02930_gb300", "csrc")


def test_no_source_builds_fp64_functions_from_approximations():
    found = [(f, m.group(0)) for f in sorted(os.listdir(CSRC))
             for m in re.finditer(r"\b\w+\.approx\.(?:\w+\.)*f64\b",
                                  open(os.path.join(CSRC, f), encoding="utf-8").read())]
    assert not found
