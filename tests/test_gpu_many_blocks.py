"""Populations whose scan blocks outnumber the threads of the block that gathers them (257 and
1025 blocks of 512 replicas), and pa_weights_static on both sides of one CTA and beyond all
SMs' first pass, against the oracle: bit for bit, floating-point sums to 1e-12 (entropy and sampling
variance from the families and counts, summed exactly)."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from paper_2401_07965_gb300 import pa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [256 * 512, 256 * 512 + 1, 1024 * 512 + 1])
@pytest.mark.parametrize("alpha", [None, 0.9])
@pytest.mark.parametrize("rule", ["systematic", "poisson"])
def test_blocks_beyond_one_pass(R, alpha, rule):
    d, L, n = 2, 4, 4
    betas = np.array([0.0, 0.02, 0.04, 0.3, 0.32])
    th = np.full(n, 1, np.uint32)
    cap = pa.default_capacity(R, rule)
    p = pa.Population(d, L, R, betas, th, rule, 4, R_cap=cap)
    if alpha is not None:
        p.set_partial_resampling(alpha)
    o = O.Run(d, L, O.ferro_couplings(d, L), R, betas, th, O.RESAMPLERS[rule], 4, R_cap=cap,
              alpha=alpha)
    for i in range(n):
        E = o.energies()
        p.step(1)
        assert o.step() == 0
        go, oo = p.observables(), o.obs()
        for k in ("R_i", "sumE", "sumC2", "accepts") + (("ess", "resampled") if alpha else ()):
            assert go[k] == oo[k], (i, k)
        assert math.isclose(go["sum_lnQ"], oo["sum_lnQ"], rel_tol=1e-12, abs_tol=1e-12), i
        assert np.array_equal(p.families(), o.families()), i
        # sums over replicas exactly: the oracle adds 10^5 terms one after another (to 1e-11)
        if alpha is None:
            f = O.resample(E, R, betas[i + 1] - betas[i], O.RESAMPLERS[rule], 4, i + 1)["f"]
            dlt = o.counts() - np.ldexp(f.astype(np.float64), -40)
            assert math.isclose(go["sv"], math.fsum(dlt * dlt) / len(E), rel_tol=1e-12), i
        nk = np.unique(o.families(), return_counts=True)[1] / oo["R_i"]
        assert math.isclose(go["entropy"], -math.fsum(nk * np.log(nk)), rel_tol=1e-12), i
        assert np.array_equal(p.energies(), o.energies()), i
    p.close()


@pytest.mark.parametrize("R", [1, 2, 511, 2048, 2049, 152 * 2048 + 1])
@pytest.mark.parametrize("L", [8, 180])  # 65 levels; 32401 levels, most of them empty
def test_weights_static_sizes(R, L):
    import torch
    rng = np.random.default_rng(R + L)
    N = L * L
    E = (-2 * N + 4 * rng.binomial(N, 0.4, R)).astype(np.int32)
    Ed = torch.from_numpy(E).cuda()
    lnQ = torch.zeros(1, dtype=torch.float64, device="cuda")
    f = torch.full((R,), 7, dtype=torch.int64, device="cuda")
    ref = O.resample(E, R, 0.01, O.RESAMPLERS["nearest"], 1, 1)

    def call(buf):
        pa.pa_weights_static(buf.data_ptr(), R, R, 2, L, 0, 0.01, lnQ.data_ptr(), f.data_ptr(),
                             torch.cuda.current_stream().cuda_stream)
        return lnQ.item(), f.cpu().numpy().view(np.uint64)

    bad = E.copy()
    bad[R // 2] += 2          # the last of them: no valid energy at all where R = 1
    v, got = call(torch.from_numpy(bad).cuda())
    assert math.isnan(v) and np.all(got == 7)
    v, _ = call(torch.full((R,), 2 * N + 4, dtype=torch.int32, device="cuda"))
    assert math.isnan(v)
    v, got = call(Ed)         # the failed calls left nothing behind
    assert np.array_equal(got, ref["f"])
    assert math.isclose(v, ref["lnQ"], rel_tol=1e-12, abs_tol=1e-15)
