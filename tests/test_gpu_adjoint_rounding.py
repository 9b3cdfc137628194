"""How far the parallel-beam adjoint may be off in FP32.  Random sinograms: sums that do not cancel the positions'
rounding as smooth data does."""

from __future__ import annotations

import math

import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import rel_l2, to_dev, to_np
from paper_2009_14788_gb300 import Geometry, backward_raw

pytestmark = pytest.mark.gpu

# A sample's offset from a pixel passes through FP32 terms of up to eleven pixels (half a tile's diagonal): their
# rounding and that of the step, taken up to eleven times, leave about 2e-7 px rms per axis.  Bilinear weights
# (rms 1/3) change by it times sqrt(2) of rms 0.58: 4.9e-7 of the result.  Placing every ray by itself
# from the split-precision table measured 4.0 .. 4.9e-7 on these sinograms.
GATE = 5.5e-7


def _make(n, angles, det, spacing, step):
    kw = dict(det_count=det, det_spacing=spacing, step=step)
    return Geometry("parallel", n, angles, **kw), O.Geometry.from_args(dict(kind="parallel", n=n, angles=angles, **kw))


@pytest.mark.parametrize("n,views,det,spacing,step", [(64, 64, 91, 1.0, 1.0), (256, 128, 363, 1.0, 1.0),
                                                      (243, 91, 367, 1.0, 1.0), (300, 50, 300, 1.4, 0.75),
                                                      (97, 60, 150, 0.83, 0.7), (768, 40, 1100, 1.0, 1.0)])
def test_rounding_of_the_rays_places(n, views, det, spacing, step):
    g, og = _make(n, np.arange(views) * (math.pi / views), det, spacing, step)
    y = np.random.default_rng(n + views).normal(size=(1, views, det)).astype(np.float32)
    ref = O.adjoint(og, y)
    for batch in (1, 3, 16, 32):
        got = to_np(backward_raw(g, to_dev(np.repeat(y, batch, 0))))
        assert (got == got[:1]).all()
        assert rel_l2(got[:1], ref) <= GATE, batch


@pytest.mark.parametrize("n", [1025, 1027])
def test_tiles_of_a_few_pixels_at_the_images_edge(n):
    """The window is as wide as the widest tile's, and beside a tile one to three pixels wide most of it lies
    outside the image, where rays keep only their line."""
    angles = np.array([0.0, 0.0005, 0.001, -0.0007, 0.002, math.pi / 2, math.pi / 2 + 0.0008, math.pi / 2 - 0.0011,
                       math.pi, math.pi + 0.0006])
    g, og = _make(n, angles, 1451, 1.0, 1.0)
    y = np.random.default_rng(n).normal(size=(1, len(angles), 1451)).astype(np.float32)
    ref = O.adjoint(og, y)[0]
    edge = n // 16 * 16
    for batch in (1, 3, 16, 32):
        got = to_np(backward_raw(g, to_dev(np.repeat(y, batch, 0))))[batch - 1]
        assert rel_l2(got[edge:], ref[edge:]) <= GATE, batch
        assert rel_l2(got[:, edge:], ref[:, edge:]) <= GATE, batch
