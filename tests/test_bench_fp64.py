"""bench.py's count of the FP64 instructions that the plain FP64 form needs."""
import os
import sys

import pytest
import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402


@pytest.mark.parametrize("lmax,w,want", [
    (0.0, 4, 0), (1e-18, 4, 0), (1e-3, 1, 0),
    (1e-16, 4, 7 + 1 * 7 + 11),   # one term
    (1e-16, 2, 3 + 1 * 2 + 3),
    (1e-8, 6, 11 + 2 * 13 + 19),  # two terms
    (2.0, 5, 9)])                 # Bateman form: the rates alone
def test_fp64_instructions(lmax, w, want):
    assert bench.fp64_instructions(torch.tensor([lmax]).double(), torch.tensor([w])).item() == want
