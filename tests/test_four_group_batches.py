"""The geometries on which the forward over four texel groups is compared with the oracle have batches that take
four groups, and the smallest is found below 400 CTAs of images.  No GPU needed."""

import pytest
import torch

from gpu_cases import CASES
from paper_2009_14788_gb300 import Geometry, forward_images_per_cta
from paper_2009_14788_gb300.build import build


@pytest.mark.parametrize("case", ["parallel_n64_full", "parallel_axes", "parallel_three_rays", "fan_ragged", "fan_close",
                                  "fan_steep", "parallel_ragged", "parallel_fine", "parallel_coarse", "one_ray",
                                  "one_pixel"])
def test_the_four_group_cases_take_four_groups(case):
    build()
    args = dict(CASES[case])
    g = Geometry(args.pop("kind"), host_only=True, **args)
    for dtype, images in ((torch.float32, 16), (torch.float16, 32), (torch.bfloat16, 32)):
        assert any(forward_images_per_cta(g, dtype, b) == images for b in range(images, 400 * images, images)), dtype
