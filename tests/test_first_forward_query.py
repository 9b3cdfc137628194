"""What a geometry's first forward call costs the host before anything is launched.  No GPU needed."""

import math
import time

import torch

from paper_2009_14788_gb300 import Geometry, forward_images_per_cta
from paper_2009_14788_gb300.build import build
from synth import uniform_angles


def test_choosing_the_launch_shape_is_cheap_beside_the_geometry():
    """The first call chooses its launch shape from the widest bands at several slab heights.  On this fan,
    looking at every slab of every CTA takes a tenth of the geometry's creation for one height and a third for
    all of them; the choice may take an eighth.  Both are single-threaded host arithmetic on the same machine;
    the best of five of each."""
    build()
    create, query = [], []
    for _ in range(5):
        t0 = time.perf_counter()
        g = Geometry("fan", 512, uniform_angles(720, 2 * math.pi), det_count=1024, det_spacing=1.5,
                     source_distance=1000.0, det_distance=500.0, host_only=True)
        t1 = time.perf_counter()
        images = forward_images_per_cta(g, torch.float16, 32)
        t2 = time.perf_counter()
        create.append(t1 - t0)
        query.append(t2 - t1)
        assert images == 32
        g.close()
    assert min(query) <= 0.125 * min(create), (min(query), min(create))
