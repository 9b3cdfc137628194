"""FBP filter rows that share a CTA.  Short rows take a fraction of a warp each, and many of them share a CTA's
taps: the same bits as the row by itself, where the last CTA is partly filled too."""

from __future__ import annotations

import numpy as np
import pytest
import torch

from gpu_cases import to_dev
from paper_2009_14788_gb300 import Geometry, filter_sinogram

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name", ["ram-lak", "shepp-logan"])
@pytest.mark.parametrize("det", [1, 5, 16, 17, 40, 64, 65, 128, 129, 200, 400])
@pytest.mark.parametrize("batch", [131, 2053])
def test_shared_rows(batch, det, name):
    g = Geometry("parallel", 4, np.arange(7) * (np.pi / 7), det_count=det)
    y = to_dev(np.random.default_rng(det).normal(size=(batch, 7, det)))
    q = filter_sinogram(g, y, name)
    for b in (0, 1, 2, batch // 2, batch - 1):
        assert torch.equal(filter_sinogram(g, y[b:b + 1], name)[0], q[b])
