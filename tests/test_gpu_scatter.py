"""The ancestor scatter against the oracle where copy numbers are far apart: one huge
temperature step (a few parents take most slots, blocks of parents without any), then a
small one (at most a few copies each), over several scan blocks and every rule."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2401_07965_gb300 import pa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rule", ["multinomial", "systematic", "residual", "poisson", "nearest"])
@pytest.mark.parametrize("R", [5, 512, 513, 3000])
@pytest.mark.parametrize("graph", [False, True])
def test_uneven_copy_numbers(rule, R, graph):
    import torch
    d, L = 2, 16
    betas = np.array([0.0, 0.5, 0.51, 2.0])
    th = np.full(3, 1, np.uint32)
    cap = 4 * R + 200
    stream = torch.cuda.Stream() if graph else None
    g = pa.Population(d, L, R, betas, th, rule, 9, R_cap=cap, stream=stream)
    o = O.Run(d, L, O.ferro_couplings(d, L), R, betas, th, O.RESAMPLERS[rule], 9, R_cap=cap)
    for i in range(3):
        g.step(1)
        assert o.step() == 0
        assert np.array_equal(g.counts(), o.counts()), i
        assert np.array_equal(g.ancestors(), o.ancestors()), i
        assert np.array_equal(g.families(), o.families()), i
        assert np.array_equal(g.energies(), o.energies()), i
        go, oo = g.observables(), o.obs()
        assert go["R_i"] == oo["R_i"] and go["sumC2"] == oo["sumC2"], i
        assert abs(go["sv"] - oo["sv"]) <= 1e-9 * max(oo["sv"], 1e-30), i
        assert abs(go["entropy"] - oo["entropy"]) <= 1e-9 * max(abs(oo["entropy"]), 1.0), i
    g.close()
