"""The workspace size queries take any number of images that converts to an integer.  No GPU needed."""

import math

import numpy as np
import pytest
import torch

from paper_2009_14788_gb300 import Geometry
from paper_2009_14788_gb300.build import build
from paper_2009_14788_gb300.radon import backward_workspace_bytes, forward_workspace_bytes
from synth import uniform_angles


@pytest.mark.parametrize("batch", [4.0, np.float64(4.0), np.int64(4), np.array(4)], ids=["float", "np_float", "np_int", "np_0d"])
def test_any_number_of_images_is_taken(batch):
    build()
    g = Geometry("parallel", 32, uniform_angles(6, math.pi), host_only=True)
    for query in (forward_workspace_bytes, backward_workspace_bytes):
        want = query(g, torch.float16, 4)
        assert want > 0
        assert query(g, torch.float16, batch) == want
