"""Landweber's reverse mode leaves out what only serves a gradient that nobody asked for; the gradients
that are asked for keep their bits."""

import numpy as np
import pytest
import torch

from gpu_cases import make, phantoms, to_dev
from paper_2009_14788_gb300 import Landweber, forward_raw

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16], ids=["f32", "bf16"])
@pytest.mark.parametrize("iterations", [0, 1, 4])
def test_each_subset_of_gradients_has_the_bits_of_all(iterations, dtype):
    g, _ = make("parallel_ragged")
    y0 = forward_raw(g, to_dev(phantoms(g.n, 3, seed=5), dtype))
    x0 = to_dev(phantoms(g.n, 3, seed=9), dtype)
    up = to_dev(np.random.default_rng(3).normal(size=tuple(x0.shape)), dtype)

    def grads(needs):
        ts = [y0.clone(), torch.tensor([2e-3], device="cuda"), x0.clone()]
        for t, n in zip(ts, needs):
            t.requires_grad_(n)
        xk = Landweber(g).run(ts[2], ts[0], ts[1], iterations)
        out = torch.autograd.grad(xk, [t for t, n in zip(ts, needs) if n], up)
        it = iter(out)
        return [next(it) if n else None for n in needs]

    whole = grads((True, True, True))
    for m in range(1, 7):
        needs = tuple(bool(m >> i & 1) for i in range(3))
        for got, want in zip(grads(needs), whole):
            assert got is None or torch.equal(got, want), needs
