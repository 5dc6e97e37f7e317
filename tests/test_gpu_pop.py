"""The one-launch resampling of small populations against the oracle, and so against the
general kernels, which other tests hold to the same oracle: both sides of a CTA's replicas and
of each cluster size, the largest population it takes and the first that it leaves; smooth
steps and one whose few parents take most slots; a batch of uneven runs; every rule."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2401_07965_gb300 import pa

pytestmark = pytest.mark.gpu

RULES = ["multinomial", "systematic", "residual", "poisson", "nearest"]


def _same(go, oo, where):
    for k in ("R_i", "sumE", "sumE2", "sumC2", "accepts"):
        assert go[k] == oo[k], (where, k)
    assert math.isclose(go["sum_lnQ"], oo["sum_lnQ"], rel_tol=1e-12, abs_tol=1e-13), where
    # order-dependent double sums, compared as in the other tests
    assert math.isclose(go["sv"], oo["sv"], rel_tol=1e-9, abs_tol=1e-12), where
    assert math.isclose(go["entropy"], oo["entropy"], rel_tol=1e-9, abs_tol=1e-12), where


@pytest.mark.parametrize("rule", RULES)
@pytest.mark.parametrize("R", [1, 2, 2047, 2048, 2049, 4097, 8193, 16385, 32767, 32768, 32769])
def test_sizes(rule, R):
    d, L = 2, 8
    betas = np.array([0.0, 0.1, 0.13, 0.7, 0.72])
    n = len(betas) - 1
    th = np.full(n, 1, np.uint32)
    cap = R if rule in ("multinomial", "systematic", "residual") else min(2 * R + 400, 32768)
    cap = max(cap, R) if R <= 32500 else pa.default_capacity(R, rule)
    g = pa.Population(d, L, R, betas, th, rule, 9, R_cap=cap)
    o = O.Run(d, L, O.ferro_couplings(d, L), R, betas, th, O.RESAMPLERS[rule], 9, R_cap=cap)
    for i in range(n):
        try:
            g.step(1)
            go = g.observables()
        except pa.PAError as e:
            assert e.status == pa.PA_ERR_CAPACITY and o.step() != 0, i
            break
        assert o.step() == 0
        assert np.array_equal(g.counts(), o.counts()), i
        assert np.array_equal(g.ancestors(), o.ancestors()), i
        assert np.array_equal(g.families(), o.families()), i
        assert np.array_equal(g.energies(), o.energies()), i
        _same(go, o.obs(), i)
    g.close()


@pytest.mark.parametrize("rule", RULES)
@pytest.mark.parametrize("graph", [False, True])
def test_uneven_batch(rule, graph):
    import torch
    sizes = [(4, 5), (4, 3000), (8, 700), (16, 9000)]   # 6145 levels in the last
    runs = [{"dim": 3, "L": L, "R": R, "R_cap": 2 * R + 100, "couplings": ("ea", 3, k)}
            for k, (L, R) in enumerate(sizes)]
    betas = np.array([0.0, 0.2, 1.2, 1.25])
    th = np.full(3, 1, np.uint32)
    stream = torch.cuda.Stream() if graph else None
    b = pa.Batch(runs, betas, th, rule, 8, stream=stream)
    orcs = [O.Run(3, L, O.disorder(3, L, 3, k), R, betas, th, O.RESAMPLERS[rule], 8,
                  R_cap=2 * R + 100, slot_base=base, run_id=k)
            for k, ((L, R), base) in enumerate(zip(sizes, b.slot_bases()))]
    for i in range(3):
        b.step(1)
        for m, o in enumerate(orcs):
            assert o.step() == 0
            _same(b.observables(m), o.obs(), (m, i))
            assert np.array_equal(b.array(m, pa.PA_ARRAY_FAMILY), o.families()), (m, i)
            assert np.array_equal(b.array(m, pa.PA_ARRAY_ENERGY), o.energies()), (m, i)
    b.close()


@pytest.mark.parametrize("rule,alpha", [("systematic", 0.6), ("poisson", 0.9), ("residual", 0.6),
                                        ("multinomial", 1.0), ("nearest", 0.3)])
@pytest.mark.parametrize("R", [1, 513, 2049, 4097, 9000, 16385, 20000, 33000])
def test_partial_sizes(rule, alpha, R):
    d, L = 2, 8
    betas = np.array([0.0, 0.05, 0.08, 0.5, 0.52, 0.56])
    n = len(betas) - 1
    th = np.full(n, 1, np.uint32)
    cap = pa.default_capacity(R, rule) + 200
    g = pa.Population(d, L, R, betas, th, rule, 5, R_cap=cap)
    g.set_partial_resampling(alpha)
    o = O.Run(d, L, O.ferro_couplings(d, L), R, betas, th, O.RESAMPLERS[rule], 5, R_cap=cap,
              alpha=alpha)
    for i in range(n):
        g.step(1)
        assert o.step() == 0
        go, oo = g.observables(), o.obs()
        _same(go, oo, i)
        assert go["ess"] == oo["ess"] and go["resampled"] == oo["resampled"], i
        assert np.array_equal(g.weights(), o.weights()), i
        assert np.array_equal(g.families(), o.families()), i
        assert np.array_equal(g.energies(), o.energies()), i
        assert math.isclose(go["e"], oo["wE"] / (oo["wsum"] * o.N), rel_tol=1e-12), i
    g.close()
