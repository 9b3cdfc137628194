"""Packed adjoint of parallel beams: one re-based ray per view and tile places every ray of its window.  Every
image-group size and storage type matches the FP64 oracle over rays denser and sparser than a pixel, windows
of three and six samples, detectors that end inside the image and tiles at the image's edge; the groups that
read the weight table (16 images, six samples) give the same bits."""

from __future__ import annotations

import math

import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import TOL_F32, rel_l2, to_dev, to_np, within_16
from paper_2009_14788_gb300 import Geometry, backward_raw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("batch", [2, 16, 32])
@pytest.mark.parametrize("n,det,spacing,step", [(1, 1, 1.0, 1.0), (15, 1, 2.5, 1.0), (33, 60, 0.31, 1.0),
                                                (33, 20, 0.7, 0.5), (48, 70, 1.0, 1.0), (50, 25, 3.1, 1.9),
                                                (64, 91, 1.3, 0.75)])
def test_parallel_adjoint_matches_the_oracle(n, det, spacing, step, batch, dtype):
    angles = np.concatenate([np.array([0.0, math.pi / 4, math.pi / 2, 3 * math.pi / 4]),
                             np.arange(31) * (2 * math.pi / 31) + 0.03])
    args = dict(kind="parallel", n=n, angles=angles, det_count=det, det_spacing=spacing, step=step)
    og = O.Geometry.from_args(args)
    g = Geometry("parallel", n, angles, det_count=det, det_spacing=spacing, step=step)
    y = to_dev(np.random.default_rng(n + batch).normal(size=(batch,) + og.sino_shape), dtype)
    got = backward_raw(g, y)
    ref = O.adjoint(og, to_np(y))
    if dtype == torch.float32:
        assert rel_l2(to_np(got), ref) <= TOL_F32
    else:
        assert within_16(to_np(got), ref, dtype)
    g.build_adjoint_table()
    assert torch.equal(backward_raw(g, y), got)
