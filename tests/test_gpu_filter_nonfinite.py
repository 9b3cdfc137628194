"""Infinities and NaN through the FBP filter.  Every bin of a row takes part in every output (the Ram-Lak's taps at
even offsets are zero, and zero times an infinity is NaN), so such a bin leaves none of its row finite -- and
no other row touched, also where several rows share a CTA."""

from __future__ import annotations

import numpy as np
import pytest
import torch

from gpu_cases import to_dev
from paper_2009_14788_gb300 import Geometry, filter_sinogram

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["ram-lak", "hann"])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("det,views,batch", [(2, 3, 1), (91, 5, 2), (128, 5, 2), (725, 3, 1), (33, 61, 40), (6001, 2, 1)])
def test_a_bin_that_is_not_finite(det, views, batch, value, name):
    g = Geometry("parallel", 4, np.arange(views) * (np.pi / views), det_count=det)
    y = to_dev(np.random.default_rng(det).normal(size=(batch, views, det)))
    clean = filter_sinogram(g, y, name)
    for bin_ in sorted({0, det // 2, det - 1}):
        z = y.clone()
        z[batch - 1, 1, bin_] = value
        q = filter_sinogram(g, z, name)
        row = q[batch - 1, 1].clone()
        assert not torch.isfinite(row).any()
        if name == "ram-lak":
            assert torch.isnan(row[bin_ % 2::2]).all()
        q[batch - 1, 1] = clean[batch - 1, 1]
        assert torch.equal(q, clean)
