"""Equal images of one batch have equal projections, whichever CTA takes them: in launches of four texel groups the
last CTA may hold one, two or three."""

from __future__ import annotations

import numpy as np
import pytest
import torch

from gpu_cases import make, to_dev
from paper_2009_14788_gb300 import _lib as L, forward_images_per_cta, forward_raw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype,batch,groups", [(torch.float32, 177, 4), (torch.float32, 181, 4), (torch.float32, 186, 4),
                                                (torch.float16, 353, 4), (torch.float16, 369, 4), (torch.bfloat16, 361, 4),
                                                (torch.float16, 9, None), (torch.float32, 3, None)])
@pytest.mark.parametrize("case", ["parallel_n64_full", "fan_ragged", "parallel_ragged"])
def test_equal_images_have_equal_projections(case, dtype, batch, groups):
    g, _ = make(case)
    if groups is not None and case == "parallel_n64_full":
        assert forward_images_per_cta(g, dtype, batch) == groups * (4 if dtype == torch.float32 else 8)
    x = to_dev(np.random.default_rng(batch).uniform(0.0, 1.0, (1, g.n, g.n)), dtype).expand(batch, g.n, g.n).contiguous()
    y = forward_raw(g, x)
    assert L.radon_get_device_error(torch.cuda.current_stream().cuda_stream) == L.RADON_OK
    assert torch.equal(y, y[:1].expand_as(y))
