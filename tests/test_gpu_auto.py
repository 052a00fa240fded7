"""HSG_KERNEL_AUTO between three quarters and 1.2 times L2, where a renormalisation after
every sweep decides between the temporally blocked launch and half-sweeps: the
same chain, bit for bit, as with the global kernel (needs a CUDA GPU)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

L = 160  # 115 MB of state, 126 MB of L2


@pytest.fixture(scope="module")
def hsg():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1006_2566_gb300 import build

    build.build()
    from paper_1006_2566_gb300 import hsg as h

    return h


# an odd and an even number of buffer swaps per graph; half-sweeps; no over-relaxation
@pytest.mark.parametrize("n_or,renorm_every,energy_every,calls", [(1, 1, 0, (3, 2)), (2, 1, 2, (5,)), (2, 2, 1, (4, 3)), (0, 1, 0, (2,))])
@pytest.mark.parametrize("use_stream", [True, False])
def test_auto_equals_global(hsg, n_or, renorm_every, energy_every, calls, use_stream):
    l2 = torch.cuda.get_device_properties(0).L2_cache_size
    assert 3 * l2 < 4 * 28 * L ** 3 and 5 * 28 * L ** 3 <= 6 * l2
    out = []
    for kernel in (hsg.HSG_KERNEL_AUTO, hsg.HSG_KERNEL_GLOBAL):
        with hsg.Lattice(L, 5, stream=torch.cuda.Stream() if use_stream else None) as lat:
            lat.generate_couplings()
            sched = hsg.schedule(kind=hsg.HSG_HEATBATH, T=0.4, n_or=n_or, renorm_every=renorm_every,
                                 energy_every=energy_every, kernel=kernel)
            if kernel == hsg.HSG_KERNEL_AUTO:
                assert hsg.hsg_kernel_for(lat.ctx, sched) == (
                    hsg.HSG_KERNEL_WAVE if renorm_every == 1 else hsg.HSG_KERNEL_GLOBAL)
            for n in calls:
                lat.sweep(sched, n)
            out.append((lat.spins(), lat.energy_log(), lat.energy()))
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1]) and out[0][2] == out[1][2]
