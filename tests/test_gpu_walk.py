"""The column-walk sweep kernels against the oracle at the shapes where they can go wrong:
every thread variant of the 2D kernel, chunked and unchunked 2D walks of other sides, 3D
walks whose columns leave lanes idle or share warps between groups, populations that end
inside a CTA, and every copy of the walk (number of leading zero threshold bits)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2401_07965_gb300 import pa

pytestmark = pytest.mark.gpu


def _run(d, L, R, betas, theta, cpl, threads=0, groups=1, rule="systematic"):
    th = np.full(len(betas) - 1, theta, np.uint32)
    J = O.ferro_couplings(d, L) if cpl[0] == "ferro" else O.disorder(d, L, cpl[1], cpl[2])
    g = pa.Population(d, L, R, betas, th, rule, 31, couplings=cpl)
    if threads:
        pa.pa_set_sweep_threads(g.ctx, threads)
    if groups > 1:
        pa.pa_set_sweep_groups(g.ctx, groups)
    o = O.Run(d, L, J, R, betas, th, O.RESAMPLERS[rule], 31)
    for i in range(len(betas) - 1):
        g.step(1)
        assert o.step() == 0
        assert np.array_equal(g.spins_words(), O.pack_spins(o.spins())), (i, betas[i + 1])
        assert np.array_equal(g.energies(), o.energies()), (i, betas[i + 1])
    go, oo = g.observables(), o.obs()
    for k in ("R_i", "sumE", "sumE2", "sumAbsM", "sumM2", "accepts"):
        assert go[k] == oo[k], k
    g.close()


# one step in each range of leading zero bits of the dE = 4 threshold (0, 1, 2, 3, 4, 6, 8)
BETAS = np.array([0.0, 0.1, 0.25, 0.45, 0.6, 0.8, 1.1, 1.6])


@pytest.mark.parametrize("L", [16, 32, 64, 128])
@pytest.mark.parametrize("threads", [0, 64, 128, 256, 384, 512])
def test_2d_thread_variants(L, threads):
    R = {16: 545, 32: 161, 64: 70, 128: 33}[L]
    _run(2, L, R, BETAS[::2], 1, ("ferro",), threads)
    _run(2, L, R, BETAS[1:] - BETAS[1], 1, ("ea", 3, 2), threads)


@pytest.mark.parametrize("L,R,threads", [(2, 70, 0), (4, 1100, 0), (6, 333, 64), (12, 333, 0),
                                         (20, 130, 512), (26, 100, 128), (48, 70, 0),
                                         (48, 70, 64), (100, 33, 0), (150, 33, 0)])
def test_2d_other_sides(L, R, threads):
    _run(2, L, R, BETAS[::3], 1, ("ferro",), threads)
    _run(2, L, R, BETAS[1:6:2] - BETAS[1], 2, ("ea", 5, 1), threads)


@pytest.mark.parametrize("L,R,groups", [(2, 100, 1), (4, 2100, 1), (4, 2100, 2), (6, 500, 1),
                                        (6, 500, 2), (8, 300, 1), (8, 300, 2), (16, 65, 2),
                                        (18, 70, 1), (22, 33, 1), (28, 33, 1)])
def test_3d_sides(L, R, groups):
    _run(3, L, R, BETAS[::3], 1, ("ferro",), 0, groups)
    _run(3, L, R, BETAS if L < 10 else BETAS[::4], 1, ("ea", 5, 1), 0, groups)
