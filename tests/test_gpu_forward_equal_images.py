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


@pytest.mark.parametrize("dtype,batch", [(torch.float32, 181), (torch.float16, 361), (torch.bfloat16, 369)])
def test_what_follows_waits_for_every_group(dtype, batch):
    """The groups left over run beside the CTAs of four groups; the stream's next kernel and a replayed graph's find
    the whole projection."""
    g, _ = make("parallel_n64_full")
    rng = np.random.default_rng(batch)
    xs = [to_dev(rng.uniform(0.0, 1.0, (batch, g.n, g.n)), dtype) for _ in range(4)]
    want = []
    for x in xs:
        want.append(forward_raw(g, x))
        torch.cuda.synchronize()
    y, x = torch.empty_like(want[0]), torch.empty_like(xs[0])
    for k in range(40):
        y.zero_()
        forward_raw(g, xs[k % 4], out=y)
        assert torch.equal(y.clone(), want[k % 4])
    stream, graph = torch.cuda.Stream(), torch.cuda.CUDAGraph()
    copy = torch.empty_like(y)
    with torch.cuda.stream(stream):
        forward_raw(g, x, out=y)
        torch.cuda.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            y.zero_()
            forward_raw(g, x, out=y)
            copy.copy_(y)
    for k in range(40):
        x.copy_(xs[k % 4])
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(copy, want[k % 4])
    assert L.radon_get_device_error(torch.cuda.current_stream().cuda_stream) == L.RADON_OK
