"""The FBP filter's sums keep FP32's accuracy under every window."""

from __future__ import annotations

import math

import numpy as np
import pytest

import oracle as O
from gpu_cases import rel_l2, to_dev, to_np
from paper_2009_14788_gb300 import Geometry, filter_sinogram


@pytest.mark.gpu
@pytest.mark.parametrize("det", [1024, 4000])
def test_every_window_sums_as_accurately(det):
    """A smooth projection cancels most of a high-pass sum, so the rounding of the sums shows in the result.  The
    kernels of these windows are of a size near their centre, where the sums are large, so their sums round
    alike; the cosine's differs in that its taps at odd offsets are close to zero.  A plain sum along the row
    leaves it 1.0 .. 1.1 times the error of the others; it stays within a quarter of it."""
    views = 8
    angles = np.arange(views) * (math.pi / views)
    g = Geometry("parallel", 8, angles, det_count=det)
    og = O.Geometry.from_args(dict(kind="parallel", n=8, angles=angles, det_count=det))
    s = np.arange(det) - (det - 1) / 2
    y = np.stack([np.sqrt(np.maximum((0.35 * det) ** 2 - (s - 0.1 * det * math.cos(t)) ** 2, 0.0)) for t in angles])
    y = y[None].astype(np.float32)
    err = {name: rel_l2(to_np(filter_sinogram(g, to_dev(y), name)), O.filter_sinogram(og, y, name))
           for name in ("cosine", "hamming", "hann")}
    assert err["cosine"] <= 1.25 * max(err["hamming"], err["hann"]), err
