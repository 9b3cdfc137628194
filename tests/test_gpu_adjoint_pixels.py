"""Single-image and plan adjoints take one pixel per thread where few tiles would leave the GPU short of warps
and a pair elsewhere (parallel beams).  Both match the FP64 oracle at sizes that end inside a tile or a pair,
and an item gives the same bits in a plan of its own as among enough others to take pairs."""

from __future__ import annotations

import math

import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import TOL_F32, rel_l2, to_dev, to_np, within_16
from paper_2009_14788_gb300 import BatchPlan, Geometry, backward_raw

pytestmark = pytest.mark.gpu


def _make(kind, n, views, **kw):
    args = dict(kind=kind, n=n, angles=np.arange(views) * (2 * math.pi / views) + 0.05, det_count=int(1.5 * n) + 1, **kw)
    if kind == "fan":
        args.update(source_distance=2.0 * n + 2, det_distance=1.0 * n, det_spacing=1.4)
    return Geometry(kind, **{k: v for k, v in args.items() if k != "kind"}), O.Geometry.from_args(args)


def _plan(geoms, ys, dtype):
    outs = [torch.empty((1, g.n, g.n), device="cuda", dtype=dtype) for g in geoms]
    BatchPlan(list(zip(geoms, ys, outs)), "adjoint", autotune=False).launch()
    return outs


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("kind,n,kw", [("parallel", 1, {}), ("parallel", 15, {}), ("parallel", 33, {}),
                                       ("parallel", 34, {"step": 0.5}), ("parallel", 31, {"det_spacing": 0.4}),
                                       ("fan", 17, {}), ("fan", 30, {})])
def test_one_pixel_and_a_pair_give_the_same_bits(kind, n, kw, dtype):
    g, og = _make(kind, n, 35, **kw)
    y = to_dev(np.random.default_rng(n).normal(size=(1,) + og.sino_shape), dtype)
    alone = _plan([g], [y], dtype)[0]
    ref = O.adjoint(og, to_np(y))
    if dtype == torch.float32:
        assert rel_l2(to_np(alone), ref) <= TOL_F32
    else:
        assert within_16(to_np(alone), ref, dtype)
    assert torch.equal(backward_raw(g, y), alone)
    # 29 x 25 tiles of parallel beams with as many views: more than 4.5 tiles per SM
    other, _ = _make("parallel", 80, 35)
    yo = to_dev(np.random.default_rng(3).normal(size=(1,) + other.sino_shape), dtype)
    among = _plan([g] + [other] * 29, [y] + [yo] * 29, dtype)
    assert torch.equal(among[0], alone)
    assert all(torch.equal(o, among[1]) for o in among[2:])
    assert torch.equal(among[1], _plan([other], [yo], dtype)[0])
