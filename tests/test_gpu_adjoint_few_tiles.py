"""Batches of more than 16 images on few tiles take groups of 16 images, on more tiles groups of 32: the same bits either
way, against the oracle at the library's gates."""

from __future__ import annotations

import math

import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import TOL_F32, rel_l2, to_dev, to_np, within_16
from paper_2009_14788_gb300 import Geometry, backward_raw, launch_config

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("batch", [17, 32, 64])
@pytest.mark.parametrize("kind,n,step", [("fan", 16, 1.0), ("fan", 46, 0.6), ("fan", 128, 1.0), ("fan", 129, 1.0),
                                         ("fan", 150, 1.0), ("parallel", 33, 0.7), ("parallel", 128, 1.0)])
def test_groups_on_few_tiles(kind, n, step, batch, dtype):
    args = dict(kind=kind, n=n, angles=np.arange(13) * (2 * math.pi / 13) + 0.1, det_count=n + 9, step=step)
    if kind == "fan":
        args.update(source_distance=2.0 * n, det_distance=1.0 * n, det_spacing=1.5)
    g, og = Geometry(**args), O.Geometry.from_args(args)
    y = to_dev(np.random.default_rng(n + batch).normal(size=(batch,) + og.sino_shape), dtype)
    x = backward_raw(g, y)
    for images in (16, 32):
        ws = torch.empty(8 * y.numel() + (1 << 22), dtype=torch.uint8, device="cuda")
        assert torch.equal(backward_raw(g, y, launch_config(images_per_cta=images), workspace=ws), x), images
    some = [0, batch // 2, batch - 1]
    ref = O.adjoint(og, to_np(y[some]))
    assert rel_l2(to_np(x[some]), ref) <= TOL_F32 if dtype == torch.float32 else within_16(to_np(x[some]), ref, dtype)
