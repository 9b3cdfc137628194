"""One texel group on fewer CTAs than fill the GPU: the packed forward takes two lanes per ray over four
views per CTA.  Against the oracle at the library's gates, with the same bits from the static-scratch
call, and an explicit views per CTA keeps one lane."""

import math

import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import TOL_F32, rel_l2, to_dev, to_np, within_16
from paper_2009_14788_gb300 import Geometry, _lib as L, forward_images_per_cta, forward_raw, launch_config
from synth import uniform_angles

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("args", [
    dict(kind="parallel", n=128, angles=uniform_angles(30, math.pi), det_count=181),
    dict(kind="parallel", n=61, angles=uniform_angles(7, math.pi) + 0.1, det_count=33, det_spacing=1.7),
    dict(kind="fan", n=96, angles=uniform_angles(41, 2 * math.pi), det_count=150, source_distance=180.0,
         det_distance=120.0),
], ids=["parallel", "ragged", "fan"])
def test_thin_grids(args, dtype):
    a = dict(args)
    g, og = Geometry(a.pop("kind"), **a), O.Geometry.from_args(args)
    for batch in (2, 4 if dtype == torch.float32 else 8):
        assert forward_images_per_cta(g, dtype, batch) == (4 if dtype == torch.float32 else 8)
        x = to_dev(np.random.default_rng(batch).uniform(0.0, 1.0, (batch, g.n, g.n)), dtype)
        y = forward_raw(g, x)
        ref = O.forward(og, to_np(x))
        assert (rel_l2(to_np(y), ref) <= TOL_F32) if dtype == torch.float32 else within_16(to_np(y), ref, dtype)
        z = torch.empty_like(y)
        code = {torch.float32: L.RADON_F32, torch.float16: L.RADON_F16, torch.bfloat16: L.RADON_BF16}[dtype]
        stream = torch.cuda.current_stream().cuda_stream
        assert L.radon_forward_static_scratch(g.handle, x.data_ptr(), z.data_ptr(), code, batch, stream) == L.RADON_OK
        assert torch.equal(y, z)
        one = forward_raw(g, x, launch_config("tiled", views_per_cta=8))
        assert (rel_l2(to_np(one), ref) <= TOL_F32) if dtype == torch.float32 else within_16(to_np(one), ref, dtype)
        assert L.radon_get_device_error(stream) == L.RADON_OK


@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16], ids=["f16", "bf16"])
@pytest.mark.parametrize("args,images", [
    (dict(kind="parallel", n=64, angles=uniform_angles(64, math.pi), det_count=91), 8),        # fewer CTAs than SMs
    (dict(kind="parallel", n=300, angles=uniform_angles(48, math.pi), det_count=425), 8),      # wide bands
    (dict(kind="parallel", n=96, angles=uniform_angles(500, math.pi), det_count=137), 16),
], ids=["few", "wide", "pair"])
def test_pairs_of_groups(args, images, dtype):
    """16-bit batches of more than eight images pair their texel groups where two CTAs of pairs fit an SM and
    fill it; single groups give the same bits at the same rows."""
    a = dict(args)
    g, og = Geometry(a.pop("kind"), **a), O.Geometry.from_args(args)
    assert forward_images_per_cta(g, dtype, 13) == images
    x = to_dev(np.random.default_rng(13).uniform(0.0, 1.0, (13, g.n, g.n)), dtype)
    y = forward_raw(g, x)
    assert within_16(to_np(y[::4]), O.forward(og, to_np(x[::4])), dtype)
    single = launch_config(images_per_cta=8, rows_per_slab=16 if images == 8 else 14)
    assert torch.equal(forward_raw(g, x, single), y)
