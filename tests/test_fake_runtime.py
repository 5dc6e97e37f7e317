"""What the library's host code asks the CUDA runtime for, on a stand-in for it (no GPU)."""
import ctypes as C

import numpy as np
import pytest

from tests import fake_runtime


@pytest.fixture
def pa():
    return fake_runtime.load()


def _run(pa, L, R, rule="systematic", dim=2, priority=0, steps=40, graph=True):
    return pa.Batch([{"dim": dim, "L": L, "R": R}], np.linspace(0.0, 1.0, steps + 1),
                    np.full(steps, 2, np.uint32), rule, 1, graph=graph, use_torch_memory=False,
                    stream=fake_runtime.Stream(pa._lib, priority))


@pytest.mark.parametrize("small,large", [((16, 500), (64, 500)), ((16, 500), (16, 8000))])
def test_one_launch_resampling_beside_another_context(pa, small, large):
    """Two contexts on two host threads: a step of one comes between the other's attribute calls
    and its launch, at every one of them."""
    a, b = _run(pa, *large, rule="multinomial", graph=False), _run(pa, *small, rule="multinomial",
                                                                   graph=False)
    inside = []

    @C.CFUNCTYPE(None)
    def other_thread():
        if not inside:
            inside.append(1)
            b.step(1)
            inside.pop()

    pa._lib.fake_attr_hook(other_thread)
    a.step(1)
    pa._lib.fake_attr_hook(None)
    names = [x["name"] for x in fake_runtime.launches(pa._lib)]
    assert sum("k_pop" in n for n in names) > 1


def test_static_weights_beside_another_call(pa):
    buf = np.zeros(64, np.int64).ctypes.data
    inside = []

    @C.CFUNCTYPE(None)
    def other_thread():
        if not inside:
            inside.append(1)
            pa.pa_weights_static(buf, 10, 10, 2, 114, 0, 0.01, buf, buf, 0)
            inside.pop()

    pa._lib.fake_attr_hook(other_thread)
    pa.pa_weights_static(buf, 10, 10, 3, 32, 0, 0.01, buf, buf, 0)
    pa._lib.fake_attr_hook(None)


@pytest.mark.parametrize("dim,L,R,ea", [(2, 16, 1000, False), (2, 64, 3000, True),
                                        (2, 24, 1000, False), (3, 6, 1000, True),
                                        (3, 10, 1000, True), (2, [4, 6, 8, 10, 100], 100, True)])
def test_every_device_of_a_process(pa, dim, L, R, ea):
    """A run on a second device, after one of the same shape on the first: function attributes
    are a device's own."""
    pa._lib.fake_reset(2)
    sides = L if isinstance(L, list) else [L]
    for dev in (0, 1, 0):
        pa._lib.fake_set_device(dev)
        first = pa._lib.fake_launches()
        b = pa.Batch([{"dim": dim, "L": s, "R": R, "couplings": ("ea", 3, 1) if ea else ("ferro",)}
                      for s in sides], np.linspace(0.0, 1.0, 5), np.full(4, 2, np.uint32),
                     "systematic", 1, use_torch_memory=False, stream=fake_runtime.Stream(pa._lib))
        b.step(2)
        new = fake_runtime.launches(pa._lib, first)
        assert len(new) >= 4 and all(x["device"] == dev for x in new)
        b.close()


@pytest.mark.parametrize("n", [1, 16])
def test_steps_with_another_device_current(pa, n):
    """A captured step is launched whatever device is current; a longer call, which captures
    several steps, must not need the context's own one either."""
    pa._lib.fake_reset(2)
    pa._lib.fake_set_device(0)
    b = _run(pa, 16, 1000)
    b.step(1)
    pa._lib.fake_set_device(1)
    first = pa._lib.fake_launches()
    b.step(n)
    assert all(x["device"] == 0 for x in fake_runtime.launches(pa._lib, first))
    assert pa._lib.fake_device() == 1


@pytest.mark.parametrize("dim,L,threads", [(2, 16, 64), (2, 16, 128), (2, 16, 512), (2, 32, 256),
                                           (2, 64, 128), (2, 48, 128)])
def test_small_sweeps_leave_room_for_others(pa, dim, L, threads):
    """A sweep launch asks for the shared memory it needs whatever its number of CTAs, so that
    contexts on other streams share the SMs with it."""
    def sweep(R):
        b = _run(pa, L, R, dim=dim, graph=False)
        pa.pa_set_sweep_threads(b.ctx, threads)
        first = pa._lib.fake_launches()
        b.step(1)
        x = [y for y in fake_runtime.launches(pa._lib, first)
             if "k_sweep2d" in y["name"] or "k_walk" in y["name"]]
        b.close()
        assert len(x) == 1
        return x[0]

    many = sweep(500000)
    same = [x for x in map(sweep, (1000, 4800, 9000, 20000, 60000, 150000))
            if (x["name"], x["block"]) == (many["name"], many["block"])]
    assert len(same) >= 1 and all(x["smem"] == many["smem"] for x in same)


@pytest.mark.parametrize("L,R", [(16, 1000), (16, 4800), (32, 2000), (32, 4500), (32, 9500),
                                 (64, 10000), (48, 4800), (48, 10000), (16, 60000)])
def test_sweeps_chained_to_the_one_launch_resampling(pa, L, R):
    """A sweep is placed while the one-launch resampling holds its SMs only where the others hold
    it at an even share each."""
    b = _run(pa, L, R)
    first = pa._lib.fake_launches()
    b.step(1)
    new = fake_runtime.launches(pa._lib, first)
    x = [y for y in new if "k_sweep2d" in y["name"] or "k_walk" in y["name"]]
    pop = sum(y["grid"] for y in new if "k_pop" in y["name"])
    assert len(x) == 1
    share = -(-x[0]["grid"] // 152)
    assert x[0]["chained"] == (pop == 0 or x[0]["grid"] <= share * (152 - pop))


@pytest.mark.parametrize("priority", [0, -1, -5])
@pytest.mark.parametrize("R", [1000, 100000])  # one launch for the resampling, several
def test_the_callers_stream_priority(pa, priority, R):
    """Captured kernels have the priority of the caller's stream; the family branch is never above
    it."""
    b = _run(pa, 16, R, priority=priority)
    first = pa._lib.fake_launches()
    b.step(1)
    new = fake_runtime.launches(pa._lib, first)
    for x in new:
        want = min(priority + 1, 0) if "k_family" in x["name"] else priority
        assert x["priority"] == want, x
    assert any("k_sweep2d" in x["name"] and x["captured"] for x in new)


def _sweeps(pa, L, R, ea=False, dim=2):
    b = pa.Batch([{"dim": dim, "L": L, "R": R, "couplings": ("ea", 3, 1) if ea else ("ferro",)}],
                 np.linspace(0.0, 1.0, 5), np.full(4, 2, np.uint32), "systematic", 1, graph=False,
                 use_torch_memory=False, stream=fake_runtime.Stream(pa._lib))
    first = pa._lib.fake_launches()
    b.step(1)
    new = fake_runtime.launches(pa._lib, first)
    b.close()
    return [x for x in new if any(k in x["name"] for k in ("k_sweep", "k_walk", "k_group"))]


@pytest.mark.parametrize("ea", [False, True])
@pytest.mark.parametrize("L", [24, 26, 38, 44, 46, 50, 54, 58, 60, 66, 74, 82, 90, 96, 100, 106, 118,
                               120, 134, 140, 158])
def test_plans_of_2d_sides_fill_the_sms(pa, L, ea):
    """Whatever the divisors of a side: a small population has at least 64 threads per group of
    32 replicas, and a large one leaves room for at least 256 threads on an SM (registers,
    shared memory), or the general kernel takes it."""
    x, = _sweeps(pa, L, 1000, ea)
    if "k_group" not in x["name"]:
        assert x["block"] >= 64 * -(-32 // x["grid"]), x
    x, = _sweeps(pa, L, 40000, ea)
    if "k_group" not in x["name"]:
        ctas = min(65536 // (96 * x["block"]), 228 * 1024 // (x["smem"] + 2048))
        assert ctas * x["block"] >= 256, x


def test_general_kernel_for_small_populations_of_tiny_lattices(pa):
    assert "k_group" in _sweeps(pa, 2, 1000, dim=3)[0]["name"]
    assert "k_walk" in _sweeps(pa, 2, 90000, dim=3)[0]["name"]


@pytest.mark.parametrize("R", [1000, 8000, 30000])
@pytest.mark.parametrize("alpha", [None, 0.5])
def test_clusters_that_the_device_cannot_place(pa, R, alpha):
    """Where no cluster of more than eight CTAs finds its SMs (a partition of a GPU), larger
    populations take the general resampling kernels instead of failing."""
    pa._lib.fake_clusters_fit(0)
    b = _run(pa, 16, R)
    if alpha is not None:
        b.set_partial_resampling(alpha)
    first = pa._lib.fake_launches()
    b.step(1)
    names = [x["name"] for x in fake_runtime.launches(pa._lib, first)]
    assert any("k_pop" in n for n in names) == (R == 1000)
    assert any("k_resample" in n for n in names) == (R > 1000)


def test_sweep_threads_while_the_stream_is_captured(pa):
    """The call is taken while the caller captures the stream; the launch follows it from the
    first step after the capture on."""
    s = fake_runtime.Stream(pa._lib)
    b = pa.Batch([{"dim": 2, "L": 64, "R": 1000}], np.linspace(0.0, 1.0, 9),
                 np.full(8, 2, np.uint32), "systematic", 1, graph=False, use_torch_memory=False,
                 stream=s)
    pa.pa_set_sweep_threads(b.ctx, 64)
    pa._lib.fake_capture(s.cuda_stream, 1)
    pa.pa_set_sweep_threads(b.ctx, 512)
    b.step(1)
    pa._lib.fake_capture(s.cuda_stream, 0)
    b.step(1)
    x = [y["block"] for y in fake_runtime.launches(pa._lib) if "k_sweep2d" in y["name"]]
    assert x == [128, 512] and pa.pa_get_sweep_threads(b.ctx) == 512
