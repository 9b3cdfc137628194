"""The packed forward over four texel groups per CTA (16-bit batches of more than 24 images, FP32 ones of
more than 16, where the grid fills the GPU), which takes a ray texel row by texel row where three samples and four columns cover a row
and sample by sample elsewhere: against the oracle at the library's gates, on geometries where every
ray, some rays and no ray goes by rows, at batches whose last CTA holds one to four groups, and within
the FP32 gate of the one-group launch (sample by sample)."""

import numpy as np
import pytest
import torch

import oracle as O
from gpu_cases import TOL_F32, make, rel_l2, to_dev, to_np, within_16
from paper_2009_14788_gb300 import _lib as L, forward_images_per_cta, forward_raw, launch_config

pytestmark = pytest.mark.gpu

# all rays by rows: parallel_*; steep rays of a fan sample by sample: fan_*; steps other than one pixel
# (none by rows): parallel_ragged, parallel_fine, parallel_coarse; degenerate: one_ray, one_pixel
CASES = ["parallel_n64_full", "parallel_axes", "parallel_three_rays", "fan_ragged", "fan_close", "fan_steep",
         "parallel_ragged", "parallel_fine", "parallel_coarse", "one_ray", "one_pixel"]


def _smallest_four(g, dtype):
    """The smallest batch of whole four-group CTAs that takes them (a thin grid does not)."""
    images = 16 if dtype == torch.float32 else 32
    return next((b for b in range(images, 400 * images, images) if forward_images_per_cta(g, dtype, b) == images), 32)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float16, torch.bfloat16], ids=["f32", "f16", "bf16"])
@pytest.mark.parametrize("case", CASES)
def test_four_groups_match_the_oracle(case, dtype):
    g, og = make(case)
    f32 = dtype == torch.float32
    bg = 4 if f32 else 8
    four = _smallest_four(g, dtype)
    for batch in (33, four, four + 3 * bg - 1):   # a thin grid, whole CTAs, a last CTA of three groups
        rng = np.random.default_rng(batch)
        x = to_dev(rng.uniform(0.0, 1.0, (batch, g.n, g.n)), dtype)
        y = forward_raw(g, x)
        some = sorted({0, 1, batch // 2, batch - bg, batch - 2, batch - 1})
        ref = O.forward(og, to_np(x[some]))
        assert L.radon_get_device_error(torch.cuda.current_stream().cuda_stream) == L.RADON_OK
        if f32:
            assert rel_l2(to_np(y[some]), ref) <= TOL_F32, batch
            one = forward_raw(g, x, launch_config(images_per_cta=4))
            assert rel_l2(to_np(y), to_np(one)) <= TOL_F32, batch
        else:
            assert within_16(to_np(y[some]), ref, dtype), (batch, rel_l2(to_np(y[some]), ref))


def test_the_query_reports_four_groups():
    """Four groups where their CTAs fill the GPU: at least 300 of them, here 27 per four groups of images."""
    g, _ = make("parallel_n64_full")
    for dtype, batch, images in ((torch.float16, 24, 8), (torch.float16, 32, 8), (torch.float16, 352, 16),
                                 (torch.float16, 353, 32), (torch.bfloat16, 384, 32), (torch.float32, 16, 4),
                                 (torch.float32, 32, 4), (torch.float32, 176, 4), (torch.float32, 177, 16),
                                 (torch.float32, 192, 16)):
        assert forward_images_per_cta(g, dtype, batch) == images, (dtype, batch)


def test_a_pixel_that_is_not_finite_stays_in_the_rays_that_sample_it():
    """Rays none of whose samples reach an infinite pixel keep finite sums (texels of weight zero beside a
    ray's columns are not read)."""
    g, og = make("parallel_three_rays")
    batch = _smallest_four(g, torch.float32)
    x = np.random.default_rng(8).uniform(0.0, 1.0, (batch, g.n, g.n))
    x[:, 20, 31] = 0.0
    clean = forward_raw(g, to_dev(x)).clone()
    touched = np.zeros_like(x[:1])
    touched[0, 20, 31] = 1.0
    far = torch.from_numpy(O.forward(og, touched)[0] == 0.0).cuda()
    x[:, 20, 31] = np.inf
    y = forward_raw(g, to_dev(x))
    assert torch.equal(y[:, far], clean[:, far])
