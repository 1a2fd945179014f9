"""What the CUDA sources may hold."""
import glob
import os
import re

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1205_1926_gb300", "csrc")


def test_roots_and_quotients_are_cuda_functions():
    """FP64 roots, reciprocals and quotients call CUDA's functions and operators: the approximate instructions that
    those are built on (a reciprocal or a reciprocal root of an FP64 value) appear in no inline assembly."""
    files = sorted(f for e in ("*.cu", "*.cuh", "*.h", "*.cpp") for f in glob.glob(os.path.join(SRC, e)))
    assert files
    for f in files:
        with open(f) as fh:
            found = re.findall(r"\b(?:rsqrt|rcp|sqrt|div)\.approx[.\w]*\.f64\b", fh.read())
        assert not found, (os.path.basename(f), found)
