"""Packed adjoint: the producer warp prepares the windows of 32 views at a time and hands them out four to a
chunk.  View counts around those edges match the FP64 oracle, with and without the weight table."""

from __future__ import annotations

import math

import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import TOL_F32, rel_l2, to_dev, to_np
from paper_2009_14788_gb300 import Geometry, backward_raw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("views", [1, 4, 5, 31, 32, 33, 36, 37, 65])
@pytest.mark.parametrize("kind", ["parallel", "fan"])
def test_adjoint_matches_the_oracle_at_view_batch_edges(kind, views):
    args = dict(kind=kind, n=45, angles=np.arange(views) * (2 * math.pi / views) + 0.1, det_count=70)
    if kind == "fan":
        args.update(source_distance=90.0, det_distance=40.0)
    og = O.Geometry.from_args(args)
    g = Geometry(kind, **{k: v for k, v in args.items() if k != "kind"})
    y = to_dev(np.random.default_rng(views).normal(size=(3,) + og.sino_shape), torch.float32)
    ref = O.adjoint(og, to_np(y))
    plain = backward_raw(g, y)
    assert rel_l2(to_np(plain), ref) <= TOL_F32
    g.build_adjoint_table()
    assert torch.equal(backward_raw(g, y), plain)
