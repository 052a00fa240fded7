"""Which sweeps are replayed as CUDA graphs: every calling pattern runs the
same chain, and none captures a graph per call (needs a CUDA GPU)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def hsg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1006_2566_gb300 import build

    build.build()
    from paper_1006_2566_gb300 import hsg as h

    return h


def run(hsg, L, sched, calls, graphs=True):
    """The spins after `calls`, and what was captured and launched."""
    with hsg.Lattice(L, 17, stream=torch.cuda.Stream() if graphs else None) as lat:
        lat.generate_couplings()
        for n in calls:
            lat.sweep(sched, n)
        return lat.spins(), *hsg.hsg_test_graph_counts(lat.ctx)


# a direct sweep first wherever the call begins on the other buffer; the fours of the last two begin there once
@pytest.mark.parametrize("calls,replayed", [((5,) * 8, 8), ((3,) * 8, 8), ((4, 1, 4, 1, 4), 2), ((5, 4, 5), 2)])
def test_odd_calls_with_odd_buffer_swaps_keep_their_graph(hsg, calls, replayed):
    sched = hsg.schedule(kind=hsg.HSG_HEATBATH, T=0.5, n_or=1, kernel=hsg.HSG_KERNEL_WAVE)
    spins, captured, launched = run(hsg, 74, sched, calls)
    assert np.array_equal(spins, run(hsg, 74, sched, (sum(calls),), graphs=False)[0])
    assert captured == 1 and launched >= replayed


@pytest.mark.parametrize("L,n_or,n,captured,launched", [
    (40, 20, 5, 1, 5),    # 42 launches a sweep: one sweep in a graph
    (40, 20, 1, 0, 0),    # a graph that would run once is not captured
    (40, 2, 10, 0, 0),
    (40, 2, 20, 1, 2),    # 60 launches in a graph
    (40, 0, 64, 1, 4),    # 16 sweeps
    (34, 31, 3, 1, 3),    # 64 launches a sweep
    (40, 20, 128, 1, 8),  # an eighth of the call
    (74, 20, 1, 1, 1)])   # where the host is hidden
def test_a_new_schedule_captures_no_more_than_it_replays(hsg, L, n_or, n, captured, launched):
    sched = hsg.schedule(kind=hsg.HSG_HEATBATH, T=0.5, n_or=n_or)
    spins, *counts = run(hsg, L, sched, (n,))
    assert np.array_equal(spins, run(hsg, L, sched, (n,), graphs=False)[0])
    assert counts == [captured, launched]


def test_a_schedule_seen_twice_has_its_graph(hsg):
    sched = hsg.schedule(kind=hsg.HSG_HEATBATH, T=0.5, n_or=2)
    assert run(hsg, 40, sched, (5, 5, 5, 5))[1:] == (1, 3)
    cadence = hsg.schedule(kind=hsg.HSG_HEATBATH, T=0.5, n_or=2, renorm_every=5, energy_every=5)
    assert run(hsg, 40, cadence, (5, 5, 5, 5))[1:] == (1, 3)


# calls shorter than the first, remainders, lengths in turn: after two calls alike a
# graph of that length, in the end one that divides them
@pytest.mark.parametrize("n_or,calls,captured,launched", [
    (5, (50, 1, 1, 1, 1), 2, 10 + 3),
    (5, (50, 13, 13, 13), 2, 10 + 2 + 3 + 3),
    (3, (64, 5, 3, 5, 3, 3, 5, 3, 5, 3), 3, 8 + 0 + 0 + 0 + 0 + 1 + 1 + 1 + 2 + 1),
    (0, (64, 1, 1, 1), 2, 4 + 0 + 1 + 1)])
@pytest.mark.parametrize("kernel", ["AUTO", "WAVE"])
def test_short_calls_get_a_graph(hsg, n_or, calls, captured, launched, kernel):
    k = getattr(hsg, "HSG_KERNEL_" + kernel)
    sched = hsg.schedule(kind=hsg.HSG_METROPOLIS, hits=2, T=0.5, n_or=n_or, kernel=k)
    spins, *counts = run(hsg, 40, sched, calls)
    want = hsg.schedule(kind=hsg.HSG_METROPOLIS, hits=2, T=0.5, n_or=n_or, kernel=hsg.HSG_KERNEL_GLOBAL)
    assert np.array_equal(spins, run(hsg, 40, want, (sum(calls),), graphs=False)[0])
    if kernel == "AUTO":
        assert counts == [captured, launched]
    else:  # other launches a sweep, buffers that swap
        assert counts[0] <= 4


def test_short_calls_stay_launches_in_the_callers_capture(hsg):
    """What a long call leaves to direct launches can be captured by the caller,
    also where a call like it has its own graph; each replay is new sweeps."""
    kw = dict(kind=hsg.HSG_HEATBATH, T=0.5, n_or=5)
    stream = torch.cuda.Stream()
    with hsg.Lattice(40, 5, stream=stream) as lat, hsg.Lattice(40, 5) as ref:
        for x in (lat, ref):
            x.generate_couplings()
        sched = hsg.schedule(**kw)
        for n in (50, 2, 2, 2):
            lat.sweep(sched, n)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            for n in (2, 3, 3):
                lat.sweep(sched, n)
        for _ in range(2):
            with torch.cuda.stream(stream):
                g.replay()
        torch.cuda.synchronize()
        ref.sweep(sched, 56 + 2 * 8)
        assert np.array_equal(lat.spins(), ref.spins())
