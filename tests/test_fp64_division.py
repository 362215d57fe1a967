"""FP64 quotients and roots in the kernels are CUDA's own (correctly rounded, or within CUDA's
documented bound): no kernel refines a hardware approximation by itself."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2505_23429_gb300", "csrc")


def test_no_fp64_approximation_instructions():
    found = []
    for name in sorted(os.listdir(CSRC)):
        if name.endswith((".cu", ".cuh")):
            text = open(os.path.join(CSRC, name)).read()
            found += [(name, m) for m in re.findall(r"\b\w+\.approx(?:\.ftz)?\.f64\b", text)]
    assert not found, found
