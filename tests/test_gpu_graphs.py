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
    spins, captured, launched = run(hsg, 36, sched, calls)
    assert np.array_equal(spins, run(hsg, 36, sched, (sum(calls),), graphs=False)[0])
    assert captured == 1 and launched >= replayed
