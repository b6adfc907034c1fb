"""bench.max_frame_nmse: the worst frame, not the mean, by hand."""
import os
import sys

import torch

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))

import bench  # noqa: E402


def test_worst_frame():
    b = torch.ones(40, 2, 2, dtype=torch.complex64)
    a = b.clone()
    a[3, 0, 0] = 3.0                    # |3 - 1|^2 / 4
    a[37, 1, :] = 1.0 + 1j              # 2 |1j|^2 / 4
    assert bench.max_frame_nmse(a, b) == 1.0
    assert bench.max_frame_nmse(a[10:], b[10:]) == 0.5
    assert bench.max_frame_nmse(b, b) == 0.0
