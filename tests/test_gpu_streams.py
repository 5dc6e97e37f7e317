"""Contexts on streams of their own, stepping at the same time: each gives what it gives alone."""
import numpy as np
import pytest

from paper_2401_07965_gb300 import pa

pytestmark = pytest.mark.gpu

# one-launch and general resampling, the 2D kernel, the walks, the general kernel
CASES = [(2, 16, 1000, "multinomial"), (2, 32, 4500, "systematic"), (2, 16, 40000, "residual"),
         (3, 6, 2000, "poisson"), (2, 58, 500, "nearest"), (2, 24, 4500, "systematic")]


def test_contexts_on_streams():
    import torch
    betas, thetas = np.linspace(0.0, 0.8, 25), np.full(24, 3, np.uint32)
    res = []
    for together in (False, True):
        ps = [pa.Population(d, L, R, betas, thetas, rule, 5, stream=torch.cuda.Stream())
              for d, L, R, rule in CASES]
        if together:
            for k in range(3):
                for p in ps:
                    p.step(8)
        else:
            for p in ps:
                p.step(24)
                pa.pa_sync(p.ctx)
        res.append([(p.energies(), p.families(), p.spins_words(), p.free_energy()) for p in ps])
        for p in ps:
            p.close()
    for a, b in zip(*res):
        for x, y in zip(a, b):
            assert np.array_equal(np.asarray(x), np.asarray(y))
