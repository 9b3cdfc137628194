"""Which geometries the forward takes over four texel groups: those whose rays mostly go row by row.  No GPU needed."""

import math

import pytest
import torch

from gpu_cases import CASES
from paper_2009_14788_gb300 import Geometry, forward_images_per_cta
from paper_2009_14788_gb300.build import build
from synth import uniform_angles


def _takes_four(g):
    """Whether some batch of whole CTAs takes four groups, by storage type."""
    return [any(forward_images_per_cta(g, dtype, b) == images for b in range(images, 400 * images, images))
            for dtype, images in ((torch.float32, 16), (torch.float16, 32), (torch.bfloat16, 32))]


@pytest.mark.parametrize("case", ["parallel_n64_full", "parallel_axes", "parallel_three_rays", "fan_ragged", "fan_close",
                                  "fan_steep", "one_ray", "one_pixel"])
def test_steps_of_one_pixel_take_four_groups(case):
    build()
    args = dict(CASES[case])
    assert _takes_four(Geometry(args.pop("kind"), host_only=True, **args)) == [True, True, True]


@pytest.mark.parametrize("step,four", [(0.5, [False, False, False]), (0.66, [False, False, False]),
                                       (0.78, [True, False, False]), (0.9, [True, True, True]),
                                       (1.02, [True, False, False]), (1.3, [False, False, False])])
def test_other_steps_take_four_groups_where_most_rays_go_by_rows(step, four):
    build()
    g = Geometry("parallel", 96, uniform_angles(96, math.pi), det_count=137, step=step, host_only=True)
    assert _takes_four(g) == four
