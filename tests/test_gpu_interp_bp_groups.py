"""The interpolating backprojector's group sizes (8, 16, and 32 images with one pixel per thread, on images of more and
fewer tiles than the rule's line): against the oracle, and the same bits whichever group an image is in."""

from __future__ import annotations

import math

import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import TOL_F32, rel_l2, to_dev, to_np, within_16
from paper_2009_14788_gb300 import Geometry, _lib as L, backproject_interpolating

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("kind", ["fan", "parallel"])
@pytest.mark.parametrize("n,batch", [(46, 32), (145, 17), (161, 32), (161, 64)])
def test_groups_of_every_size(n, batch, kind, dtype):
    args = dict(kind=kind, n=n, angles=np.arange(13) * (2 * math.pi / 13) + 0.1, det_count=n + 9)
    if kind == "fan":
        args.update(source_distance=2.0 * n, det_distance=1.0 * n, det_spacing=1.5)
    g, og = Geometry(**args), O.Geometry.from_args(args)
    y = to_dev(np.random.default_rng(n + batch).uniform(0.0, 1.0, size=(batch,) + og.sino_shape), dtype)
    x = backproject_interpolating(g, y)
    for size in (5, 16):
        assert torch.equal(backproject_interpolating(g, y[-size:]), x[-size:]), size
    some = [0, batch // 2, batch - 1]
    ref = O.backproject_interpolating(og, to_np(y[some]))
    assert rel_l2(to_np(x[some]), ref) <= TOL_F32 if dtype == torch.float32 else within_16(to_np(x[some]), ref, dtype)
    assert L.radon_get_device_error(torch.cuda.current_stream().cuda_stream) == L.RADON_OK
