"""Batches whose sides take different sweep kernels, among them the general kernel for one side
only, against the oracle run by run."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2401_07965_gb300 import pa

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dim,sides,R,ea", [(2, [58, 24, 46], 70, False), (2, [16, 58], 33, True),
                                            (2, [74], 40, True), (3, [2, 6, 10], 100, True),
                                            (3, [2], 333, False)])
@pytest.mark.parametrize("threads", [0, 64])
def test_sides_of_different_kernels(dim, sides, R, ea, threads):
    betas, thetas = np.linspace(0.0, 0.6, 4), np.full(3, 2, np.uint32)
    runs = [{"dim": dim, "L": L, "R": R + k, "couplings": ("ea", 3, k) if ea else ("ferro",)}
            for k, L in enumerate(sides + sides[:1])]
    b = pa.Batch(runs, betas, thetas, "systematic", 5)
    if threads:
        pa.pa_set_sweep_threads(b.ctx, threads)
    orcs = [O.Run(dim, r["L"], O.disorder(dim, r["L"], 3, k % len(runs)) if ea else
                  O.ferro_couplings(dim, r["L"]), r["R"], betas, thetas, O.RESAMPLERS["systematic"],
                  5, R_cap=r["R"], slot_base=base, run_id=k)
            for k, (r, base) in enumerate(zip(runs, b.slot_bases()))]
    for i in range(3):
        b.step(1)
        for m, o in enumerate(orcs):
            assert o.step() == 0
            assert np.array_equal(b.spins_words(m), O.pack_spins(o.spins())), (i, m)
            assert np.array_equal(b.array(m, pa.PA_ARRAY_ENERGY), o.energies()), (i, m)
            assert b.observables(m)["accepts"] == o.obs()["accepts"], (i, m)
    b.close()
