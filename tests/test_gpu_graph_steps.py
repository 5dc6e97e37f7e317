"""Calls of pa_step that take one captured step, several at once and a mix of both, against
the same steps launched directly."""
import numpy as np
import pytest

from paper_2401_07965_gb300 import pa

pytestmark = pytest.mark.gpu

BETAS = np.linspace(0.0, 1.0, 42)
THETAS = np.arange(41, dtype=np.uint32) % 3 + 1


def _run(calls, graph, partial, R, threads=None):
    import torch
    p = pa.Population(2, 16, R, BETAS, THETAS, "poisson" if partial is None else "systematic", 5,
                      stream=torch.cuda.Stream())
    pa.pa_set_graph(p.ctx, graph)
    if partial is not None:
        p.set_partial_resampling(partial)
    for k, n in enumerate(calls):
        if threads and k == 1:  # the captured steps are dropped and taken again
            pa.pa_set_sweep_threads(p.ctx, threads)
        p.step(n)
    pa.pa_sync(p.ctx)
    out = (p.trace(), p.energies(), p.families(), p.spins_words(), pa.pa_launch_count(p.ctx))
    p.close()
    return out


@pytest.mark.parametrize("calls", [[7, 8], [15, 1], [16], [17, 8], [41], [1, 40], [24, 17]])
@pytest.mark.parametrize("partial", [None, 0.7])
@pytest.mark.parametrize("R", [700, 33000])  # one-launch resampling, general kernels
def test_graph_steps(calls, partial, R):
    a = _run(calls, True, partial, R, threads=64)
    b = _run([1] * sum(calls), False, partial, R)
    for x, y in zip(a[0], b[0]):
        for k in x:
            assert np.array_equal(np.asarray(x[k]), np.asarray(y[k]), equal_nan=True), k
    for x, y in zip(a[1:4], b[1:4]):
        assert np.array_equal(x, y)
    assert a[4] == b[4]
