"""What the kernel sources must not contain (no GPU needed)."""
import os
import re

import paper_2501_19392_b200

CSRC = os.path.join(os.path.dirname(paper_2501_19392_b200.__file__), "csrc")


def test_special_functions_are_called_not_rebuilt():
    """Reciprocals, roots, logarithms and powers are CUDA's functions, whose error bounds are documented; none is made of
    the machine's approximate instruction and a refinement of our own."""
    made = re.compile(r"\b(rcp|rsqrt|sqrt|lg2|ex2|div|sin|cos|tanh)\.approx")
    found = [(name, line.strip()) for name in sorted(os.listdir(CSRC))
             for line in open(os.path.join(CSRC, name)) if made.search(line)]
    assert found == []
