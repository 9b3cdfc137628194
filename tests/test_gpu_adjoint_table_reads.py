"""The exact adjoint's weight table on the calls that read it -- fan beams in groups of 8 and 16 images, parallel beams
of short steps in groups of 16 -- and no table where no call would: the same bits as without one, under fused
epilogues, graph replay, autograd, rebuilding, and where dense rays leave weights to be computed."""

from __future__ import annotations

import math

import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import TOL_F32, make, rel_l2, to_dev, to_np, within_16
from paper_2009_14788_gb300 import Geometry, RadonFanbeam, _lib as L, backward_fused, backward_raw
from synth import uniform_angles

pytestmark = pytest.mark.gpu


def _clean():
    assert L.radon_get_device_error(torch.cuda.current_stream().cuda_stream) == L.RADON_OK


def _build(g):
    """Builds the table; the number of kernels that took."""
    n = L.radon_kernel_launch_count()
    g.build_adjoint_table()
    return L.radon_kernel_launch_count() - n


@pytest.mark.parametrize("case", ["parallel_n64_full", "parallel_n256_sub", "parallel_coarse"])
def test_no_table_is_built_that_no_call_reads(case):
    g, og = make(case)
    y = to_dev(np.random.default_rng(1).normal(size=(16,) + g.sino_shape))
    want = backward_raw(g, y)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    assert _build(g) == 0
    assert torch.cuda.mem_get_info()[0] == free
    assert g.adjoint_table_overflow() == 0.0
    assert torch.equal(backward_raw(g, y), want)
    g.free_adjoint_table()


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("case,batch", [("fan_ragged", 6), ("fan_ragged", 13), ("parallel_ragged", 16)])
def test_fused_epilogues_and_graphs(case, batch, dtype):
    g, _ = make(case)
    rng = np.random.default_rng(12)
    y = to_dev(rng.normal(size=(batch,) + g.sino_shape), dtype)
    add = to_dev(rng.normal(size=(batch, g.n, g.n)), dtype)
    s_dev = torch.tensor([0.37], device="cuda")

    def fused(out=None):
        return backward_fused(g, y, op_scale=-1.5, op_scale_dev=s_dev, add=add, add_scale=0.5, out=out)

    want = fused()
    assert _build(g) == 1
    try:
        assert torch.equal(fused(), want)
        out, graph, stream = torch.empty_like(want), torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.stream(stream):
            fused(out)
            torch.cuda.synchronize()
            with torch.cuda.graph(graph, stream=stream):
                fused(out)
        out.zero_()
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, want)
        _clean()
    finally:
        g.free_adjoint_table()


def test_the_forwards_gradient():
    radon = RadonFanbeam(64, uniform_angles(33, 2 * np.pi), 120.0, det_distance=60.0, det_count=91)
    x = torch.from_numpy(np.random.default_rng(4).uniform(0.0, 1.0, (6, 64, 64))).to("cuda", torch.float32)

    def grad():
        xg = x.clone().requires_grad_(True)
        (radon.forward(xg) ** 2).sum().backward()
        return xg.grad

    want = grad()
    assert _build(radon.geometry) == 1
    try:
        assert torch.equal(grad(), want)
    finally:
        radon.geometry.free_adjoint_table()


def _dense_fan():
    args = dict(kind="fan", n=40, angles=uniform_angles(9, 2 * math.pi) + 0.1, det_count=300, det_spacing=0.5,
                source_distance=80.0, det_distance=60.0)
    return Geometry(**args), O.Geometry.from_args(args)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16], ids=["f32", "f16"])
@pytest.mark.parametrize("which,batch", [("fan", 4), ("fan", 16), ("parallel", 16)])
def test_dense_rays_keep_computing_their_weights(which, batch, dtype):
    g, og = _dense_fan() if which == "fan" else make("parallel_fine")
    y = to_dev(np.random.default_rng(3).normal(size=(batch,) + g.sino_shape), dtype)
    want = backward_raw(g, y)
    assert _build(g) == 1
    try:
        assert g.adjoint_table_overflow() > 0.5
        assert torch.equal(backward_raw(g, y), want)
        ref = O.adjoint(og, to_np(y))
        assert rel_l2(to_np(want), ref) <= TOL_F32 if dtype == torch.float32 else within_16(to_np(want), ref, dtype)
        _clean()
    finally:
        g.free_adjoint_table()


@pytest.mark.parametrize("case,batch", [("fan_close", 5), ("parallel_ragged", 16)])
def test_rebuilding_replaces_the_table(case, batch):
    g, _ = make(case)
    y = to_dev(np.random.default_rng(2).normal(size=(batch,) + g.sino_shape))
    want = backward_raw(g, y)
    assert _build(g) == 1
    held = torch.cuda.mem_get_info()[0]
    assert _build(g) == 1
    try:
        assert torch.cuda.mem_get_info()[0] == held
        assert torch.equal(backward_raw(g, y), want)
    finally:
        g.free_adjoint_table()


@pytest.mark.parametrize("views", [1, 4, 5, 31, 32, 33, 36, 37, 65])
def test_short_steps_at_the_producers_view_batches(views):
    """Parallel beams of short steps: 16 images read the table at view counts around the producer warp's 32."""
    args = dict(kind="parallel", n=45, angles=np.arange(views) * (2 * math.pi / views) + 0.1, det_count=70, step=0.7)
    g, og = Geometry(**args), O.Geometry.from_args(args)
    y = to_dev(np.random.default_rng(views).normal(size=(16,) + g.sino_shape))
    plain = backward_raw(g, y)
    assert rel_l2(to_np(plain), O.adjoint(og, to_np(y))) <= TOL_F32
    assert _build(g) == 1
    assert torch.equal(backward_raw(g, y), plain)
