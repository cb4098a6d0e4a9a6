"""What the CUDA sources leave to the compiler (CPU)."""
import glob
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2603_10741_gb300", "csrc")


def test_divisions_and_roots_are_cudas_own():
    """No approximate reciprocal, division, root or exponential in inline PTX: pivots, inverses and
    norms are rounded as the compiler's operators round them."""
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        with open(path) as f:
            found = re.findall(r"(?:rcp|div|sqrt|rsqrt|ex2|lg2)\.(?:approx|full)\S*", f.read())
        assert not found, (path, found)
