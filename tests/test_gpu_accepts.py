"""Accepted flips of a step are counted in 64 bits: steps of so many sweeps that a thread's,
or a warp's, flips pass 2^32.

At beta = 1e-12 every Metropolis threshold is 2^32 - 1, so a proposal with dE > 0 is refused
with probability 2^-32 and all others are accepted: of P = theta N R proposals P - X are
accepted, X at most Poisson of mean P 2^-32 (below 30 in every case; more than 100 has
probability below 1e-20).  In every case a warp makes more than 2^32 flips."""
import numpy as np
import pytest

from paper_2401_07965_gb300 import pa

pytestmark = pytest.mark.gpu


# the 2D kernel with one warp's lanes on 16 rows each, the walk with 34 rows per thread, the
# 3D walk, the flat 3D kernel, the general kernel (batches of five sides)
@pytest.mark.parametrize("d,sides,R,theta,threads", [(2, [16], 512, 150000, 64),
                                                     (2, [34], 640, 150000, 64),
                                                     (3, [8], 512, 300000, 0),
                                                     (3, [10], 64, 300000, 0),
                                                     (2, [4, 6, 8, 10, 40], 32, 200000, 64)])
def test_accepts_past_32_bits(d, sides, R, theta, threads):
    b = pa.Batch([{"dim": d, "L": L, "R": R} for L in sides], np.array([0.0, 1e-12]),
                 np.array([theta], np.uint32), "systematic", 7)
    if threads:
        pa.pa_set_sweep_threads(b.ctx, threads)
    b.step(1)
    for m, L in enumerate(sides):
        P = theta * L ** d * R
        got = b.observables(m)["accepts"]
        assert P - 100 <= got <= P, (L, P, got, P - got)
    b.close()
