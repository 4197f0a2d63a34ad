"""What the CUDA sources leave to CUDA: reciprocals, quotients and square roots in
64 bits are CUDA's own, not built on the approximate instructions."""
import glob
import os
import re

from paper_2608_06291_gb300 import buildlib


def test_no_hand_made_reciprocal_or_square_root():
    for path in glob.glob(os.path.join(buildlib.CSRC, "*.cu*")):
        with open(path) as f:
            found = re.findall(r"\b(?:rcp|rsqrt|sqrt|div)\.approx[.\w]*", f.read())
        assert not found, (path, found)
