"""The FBP filter kernels against the FP64 oracle where their row splits can go wrong: detectors at the edges of
the eight-output groups and the 64 near taps, odd and even (the Ram-Lak's two half-size sums), enough rows
for several to share a CTA, and rows too long for shared memory."""

from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import TOL_F32, rel_l2, to_dev, to_np, within_16
from paper_2009_14788_gb300 import Geometry, filter_sinogram

pytestmark = pytest.mark.gpu


def _check(det, views, batch, name, dtype):
    args = dict(kind="parallel", n=4, angles=np.arange(views) * (np.pi / views), det_count=det)
    og = O.Geometry.from_args(args)
    g = Geometry("parallel", 4, args["angles"], det_count=det)
    y = to_dev(np.random.default_rng(det).normal(size=(batch, views, det)), dtype)
    got, ref = to_np(filter_sinogram(g, y, name)), O.filter_sinogram(og, to_np(y), name)
    if dtype == torch.float32:
        assert rel_l2(got, ref) <= TOL_F32
    else:
        assert within_16(got, ref, dtype)


@pytest.mark.parametrize("name", ["ram-lak", "hann"])
@pytest.mark.parametrize("det", [1, 2, 3, 7, 8, 9, 15, 16, 17, 63, 64, 65, 126, 127, 128, 129, 130, 131, 255, 257, 1021])
def test_filter_rows(det, name):
    _check(det, 5, 2, name, torch.float32)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("det,views,batch", [(33, 61, 40), (90, 61, 61), (33, 83, 61), (9602, 2, 1), (9999, 3, 1)])
def test_filter_shared_and_long_rows(det, views, batch, dtype):
    for name in ("ram-lak", "cosine"):
        _check(det, views, batch, name, dtype)
