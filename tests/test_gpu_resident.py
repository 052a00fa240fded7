"""The resident kernel (whole sweeps of a lone small lattice in one launch)
against the half-sweep launches, bit for bit (needs a CUDA GPU)."""
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


def chain(hsg, L, kernel, layout, stream, **kw):
    """Calls that start and end between cadences, a counter that crosses 2^32
    and one set by hand, spins set from outside: spins, log, counter, E/N."""
    sched = hsg.schedule(kernel=kernel, T=0.6, renorm_every=3, energy_every=2, **kw)
    with hsg.Lattice(L, 29, 1, 1, stream=stream, layout=layout) as lat:
        lat.generate_couplings()
        lat.sweep(sched, 1)
        lat.sweep_count = 2 ** 32 - 4
        lat.sweep(sched, 7)
        mid = lat.spins()
        lat.set_spins(mid[::-1].reshape(-1, 3)[:, ::-1].reshape(-1).copy())
        lat.sweep(sched, 4)
        return lat.spins(), lat.energy_log(), lat.sweep_count, lat.energy(), mid


# 4, 6, 8: one CTA; 10, 12, 14: eight CTAs, one or two planes each; 16, 18,
# 22, 30: sixteen, ragged; 32: 1024 threads each; 34: past the rule
@pytest.mark.parametrize("L", [4, 6, 8, 10, 12, 14, 16, 18, 22, 30, 32, 34])
def test_resident_sweeps_equal_half_sweep_launches(hsg, L):
    kinds = [dict(kind=hsg.HSG_METROPOLIS, hits=1, proposal=hsg.HSG_PROP_SPHERE, n_or=0),
             dict(kind=hsg.HSG_METROPOLIS, hits=3, proposal=hsg.HSG_PROP_BALL, n_or=2),
             dict(kind=hsg.HSG_HEATBATH, n_or=1),
             dict(kind=hsg.HSG_METROPOLIS_OR, hits=2, proposal=hsg.HSG_PROP_SPHERE, n_or=0),
             dict(kind=hsg.HSG_METROPOLIS_OR, hits=2, proposal=hsg.HSG_PROP_BALL, n_or=1),
             dict(kind=hsg.HSG_NONE, n_or=2),
             # the most hits that the rule lets in, and one more
             dict(kind=hsg.HSG_METROPOLIS, hits=16 if L <= 16 else 5 if L <= 24 else 2, proposal=1, n_or=1),
             dict(kind=hsg.HSG_METROPOLIS, hits=17 if L <= 16 else 6 if L <= 24 else 3, proposal=0, n_or=1)]
    for i, kw in enumerate(kinds):
        layout = (hsg.HSG_LAYOUT_FLOAT4, hsg.HSG_LAYOUT_PACKED)[i % 2]
        stream = torch.cuda.Stream() if i % 3 else None
        want = chain(hsg, L, hsg.HSG_KERNEL_GLOBAL, layout, stream, **kw)
        got = chain(hsg, L, hsg.HSG_KERNEL_AUTO, layout, stream, **kw)
        for a, b in zip(got, want):
            assert np.array_equal(a, b), (L, kw)


def test_nothing_to_do_only_counts(hsg):
    with hsg.Lattice(16, 3) as lat:
        lat.generate_couplings()
        s0 = lat.spins()
        lat.sweep(hsg.schedule(kind=hsg.HSG_NONE, n_or=0, energy_every=2), 5)
        assert lat.sweep_count == 5 and len(lat.energy_log()) == 2
        assert np.array_equal(lat.spins(), s0)


def test_a_captured_sweep_replays_as_new_sweeps(hsg):
    """A caller's own stream capture takes the half-sweep launches, which
    read the sweep counter from the device: each replay is the next sweep."""
    L, kw = 16, dict(kind=hsg.HSG_METROPOLIS, hits=2, proposal=1, T=0.7, n_or=1, renorm_every=9)
    stream = torch.cuda.Stream()
    with hsg.Lattice(L, 5, stream=stream) as lat, hsg.Lattice(L, 5) as ref:
        for x in (lat, ref):
            x.generate_couplings()
        ref.sweep(hsg.schedule(**kw), 3)
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            lat.sweep(hsg.schedule(**kw), 1)
        for _ in range(3):
            with torch.cuda.stream(stream):
                g.replay()
        torch.cuda.synchronize()
        assert np.array_equal(lat.spins(), ref.spins())


# alone in their clusters, and too many for the GPU at once (smaller clusters)
@pytest.mark.parametrize("sides,n", [((4, 6, 8, 10, 12, 14, 16, 18, 20, 22, 24, 26, 28, 30), 14), ((16,), 130), ((8,), 70), ((4, 8), 400),
                                     ((12, 20), 60), ((24,), 40), ((26, 28, 30), 30)])
@pytest.mark.parametrize("use_stream", [True, False])
def test_pools_of_small_lattices_equal_lattices_alone(hsg, sides, n, use_stream):
    """All sweeps of a call in one launch per side; counters
    stay right for the calls that take the half-sweep kernels."""
    kw = dict(kind=hsg.HSG_METROPOLIS, hits=2, proposal=hsg.HSG_PROP_BALL, n_or=1, renorm_every=3)
    many = dict(kw, hits=18)  # too many hits for the resident kernel
    specs = [(sides[k % len(sides)], 3, k, k & 1, 0.3 + 0.01 * k) for k in range(n)]
    with hsg.Pool(1 << 26, n, torch.cuda.Stream() if use_stream else None) as pool:
        slots = [pool.admit(*s) for s in specs]
        pool.sweep(hsg.schedule(**kw), 4)
        pool.sweep(hsg.schedule(**many), 1)
        pool.sweep(hsg.schedule(**kw), 2)
        e = pool.energies()
        for slot, (L, seed, sample, replica, T) in list(zip(slots, specs))[:: max(1, n // 20)]:
            with hsg.Lattice(L, seed, sample, replica) as lat:
                lat.generate_couplings()
                for s, k in ((kw, 4), (many, 1), (kw, 2)):
                    lat.sweep(hsg.schedule(T=T, kernel=hsg.HSG_KERNEL_GLOBAL, **s), k)
                assert np.array_equal(pool.spins(slot), lat.spins()), L
                assert abs(e[slot] - lat.energy()) <= 2e-6
                assert pool.sweep_count(slot) == 7


@pytest.mark.parametrize("L", [8, 16, 32])
def test_a_device_without_room_for_the_cluster_takes_half_sweeps(hsg, L):
    kw = dict(kind=hsg.HSG_HEATBATH, n_or=1, renorm_every=2)
    out = []
    try:
        for on in (0, 1):
            hsg.hsg_test_no_clusters(on)
            with hsg.Lattice(L, 3, stream=torch.cuda.Stream()) as lat, hsg.Pool(1 << 22, 2, torch.cuda.Stream()) as pool:
                lat.generate_couplings()
                slot = pool.admit(L, 3)
                n, m = hsg.hsg_launch_count(lat.ctx), hsg.hsg_pool_launch_count(pool.pool)
                lat.sweep(hsg.schedule(**kw), 5)
                pool.sweep(hsg.schedule(**kw), 5)
                n, m = hsg.hsg_launch_count(lat.ctx) - n, hsg.hsg_pool_launch_count(pool.pool) - m
                out.append((lat.spins(), pool.spins(slot), n, m))
    finally:
        hsg.hsg_test_no_clusters(0)
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])
    assert out[0][2] == 1 and out[1][2] >= 20 and out[1][3] >= 20  # 5 x 4 half-sweeps and what goes with them


def test_long_calls_let_other_streams_in(hsg):
    """A pool's launch can hold every SM (here with one CTA a lattice, in more
    than one wave); a call of many sweeps is several launches, between which
    another stream's kernel runs.  The counters and the renormalisations go on
    from launch to launch."""
    kw = dict(kind=hsg.HSG_HEATBATH, n_or=2, renorm_every=100)
    L, lattices, n = 8, 1200, 2000
    with hsg.Pool(1 << 26, lattices, torch.cuda.Stream()) as pool, hsg.Lattice(L, 3, 700, stream=torch.cuda.Stream()) as lat:
        slots = [pool.admit(L, 3, k, 0, 0.5) for k in range(lattices)]
        lat.generate_couplings()
        x = torch.zeros(1 << 20, device="cuda")
        other = torch.cuda.Stream()
        with torch.cuda.stream(other):
            x += 1.0  # loads its kernel, which waits for the device
        pool.sweep(hsg.schedule(**kw), 1)
        pool.energies()
        lat.sweep(hsg.schedule(T=0.5, **kw), 1)
        torch.cuda.synchronize()
        t = [torch.cuda.Event(enable_timing=True) for _ in range(3)]
        t[0].record(other)
        pool.sweep(hsg.schedule(**kw), n)
        with torch.cuda.stream(other):
            x += 1.0
        t[1].record(other)
        pool.energies()
        t[2].record(other)
        torch.cuda.synchronize()
        # an eighth of the call is one launch, of which the first wave has to end
        assert t[0].elapsed_time(t[1]) < 0.2 * t[0].elapsed_time(t[2])
        launches = hsg.hsg_launch_count(lat.ctx)
        lat.sweep(hsg.schedule(T=0.5, **kw), n)
        assert hsg.hsg_launch_count(lat.ctx) - launches == 8  # 256 sweeps each
        assert np.array_equal(pool.spins(slots[700]), lat.spins())
        with hsg.Lattice(L, 3, 700, stream=torch.cuda.Stream()) as ref:
            ref.generate_couplings()
            ref.sweep(hsg.schedule(T=0.5, kernel=hsg.HSG_KERNEL_GLOBAL, **kw), 1 + n)
            assert np.array_equal(lat.spins(), ref.spins())
