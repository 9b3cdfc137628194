"""The ray table's entries for parallel rays that miss the image.  No GPU needed."""

import math

import numpy as np
import pytest

from paper_2009_14788_gb300 import Geometry
from paper_2009_14788_gb300.build import build


@pytest.mark.parametrize("n,step", [(40, 1.0), (243, 1.0), (1000, 1.0), (97, 0.7)])
def test_steps_from_the_foot_point_stay_exact_across_the_image(n, step):
    """Such a ray may place its neighbours' samples in a tile at the image's edge, up to half a diagonal from its
    foot point (sample 0) either way: there k times the step's high part is exact in FP32, like within the
    range of the rays that hit, and high and low part together are the step."""
    build()
    angles = np.array([0.0, 0.003, 0.4, math.pi / 4, 1.2, math.pi / 2 - 0.002, 2.0, 3.0])
    g = Geometry("parallel", n, angles, det_count=2 * n, step=step, host_only=True)
    rays, counts = g.rays()
    miss = counts == 0
    assert miss.any()
    k = np.arange(0, int(0.75 * (n + 1) / step) + 24 * math.ceil(1.0 / step) + 8, dtype=np.float64)
    for part, truth in ((4, -np.sin(angles)), (5, np.cos(angles))):
        hi = rays[..., part][miss]
        assert np.array_equal(np.float32(k)[None, :] * hi[:, None], (k[None, :] * hi[:, None].astype(np.float64)))
        whole = hi.astype(np.float64) + rays[..., part + 2][miss]
        want = step * np.abs(np.broadcast_to(truth[:, None], counts.shape)[miss])
        assert np.all(np.abs(np.abs(whole) - want) <= 2.0 ** -34)
