"""Calls whose launches are chained to each other, captured on the caller's stream: the
replay gives what the direct call gives."""
import numpy as np
import pytest

from paper_2401_07965_gb300 import pa

pytestmark = pytest.mark.gpu


def _capture(call):
    import torch
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        call(s.cuda_stream)  # the library's code is loaded before the capture
    s.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=s):
        call(torch.cuda.current_stream().cuda_stream)
    return g


@pytest.mark.parametrize("R", [2048, 2049, 300001])  # one launch, two
def test_weights_static(R):
    import torch
    gen = torch.Generator(device="cuda").manual_seed(R)
    E = (-torch.randint(0, 200, (R,), device="cuda", generator=gen, dtype=torch.int32) * 4)
    out = [(torch.zeros(1, dtype=torch.float64, device="cuda"),
            torch.zeros(R, dtype=torch.int64, device="cuda")) for _ in range(2)]

    def call(k):
        return lambda st: pa.pa_weights_static(E.data_ptr(), R, R, 2, 32, 0, 0.01,
                                               out[k][0].data_ptr(), out[k][1].data_ptr(), st)

    g = _capture(call(0))
    for t in out[0]:
        t.zero_()
    g.replay()
    call(1)(torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert int(out[1][1].min()) > 0


@pytest.mark.parametrize("B", [33, 12040])
def test_mlp_gradients(B):
    import torch
    n = pa.PA_MLP_NPARAM
    gen = torch.Generator(device="cuda").manual_seed(B)
    w = torch.randn(n, device="cuda", generator=gen) * 0.2
    X = torch.randn(B, 8, device="cuda", generator=gen)
    Y = torch.randn(B, 2, device="cuda", generator=gen)
    mask = torch.ones(B, 2, device="cuda")
    scratch = torch.empty(pa.pa_mlp_scratch_bytes(B), dtype=torch.uint8, device="cuda")
    out = [(torch.zeros(n, device="cuda"), torch.zeros(1, device="cuda")) for _ in range(2)]

    def call(k):
        return lambda st: pa.pa_mlp_gradients(w.data_ptr(), X.data_ptr(), Y.data_ptr(),
                                              mask.data_ptr(), B, out[k][0].data_ptr(),
                                              out[k][1].data_ptr(), scratch.data_ptr(),
                                              scratch.numel(), st)

    g = _capture(call(0))
    for t in out[0]:
        t.zero_()
    g.replay()
    torch.cuda.synchronize()
    call(1)(torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    assert torch.equal(out[0][0], out[1][0]) and torch.equal(out[0][1], out[1][1])
    assert float(out[1][1]) > 0


@pytest.mark.parametrize("dim,L,R", [(2, 16, 1000), (2, 24, 1000), (2, 16, 33000), (3, 6, 1000)])
def test_direct_steps(dim, L, R):
    import torch
    betas = np.linspace(0.0, 0.6, 7)
    thetas = np.full(6, 2, np.uint32)
    res = []
    for capture in (False, True):
        s = torch.cuda.Stream()
        p = pa.Population(dim, L, R, betas, thetas, "systematic", 3, stream=s)
        pa.pa_set_graph(p.ctx, False)
        p.step(2)
        s.synchronize()
        if capture:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=s):
                p.step(4)
            with torch.cuda.stream(s):
                g.replay()
            s.synchronize()
        else:
            p.step(4)
        pa.pa_sync(p.ctx)
        res.append((p.energies(), p.families(), p.spins_words(), p.free_energy()))
        p.close()
    for x, y in zip(*res):
        assert np.array_equal(np.asarray(x), np.asarray(y))
