"""Pools whose larger lattices are swept in batches: every lattice as alone,
bit for bit (needs a CUDA GPU)."""
import math

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


# around the rule's sides (30 | 32, 34), a lattice larger than a batch's bytes
# (108: 35 MB), small ones between them
SPECS = [(32, 7, 0, 0, 0.5), (16, 7, 1, 0, 0.9), (108, 7, 2, 1, 0.4), (34, 7, 3, 0, math.inf), (30, 7, 4, 0, 0.6),
         (66, 7, 5, 0, 1.0), (8, 7, 6, 1, 0.3), (96, 7, 7, 0, 0.7)]


def alone(hsg, spec, kw, n, first=0):
    L, seed, sample, replica, T = spec
    with hsg.Lattice(L, seed, sample, replica) as lat:
        lat.generate_couplings()
        lat.sweep(hsg.schedule(T=T, **kw), n)
        return lat.spins(), lat.energy()


def kinds(hsg):
    return [dict(kind=hsg.HSG_METROPOLIS, hits=2, proposal=hsg.HSG_PROP_SPHERE, n_or=1, renorm_every=2),
            dict(kind=hsg.HSG_METROPOLIS, hits=3, proposal=hsg.HSG_PROP_BALL, n_or=0),
            dict(kind=hsg.HSG_HEATBATH, n_or=2, renorm_every=3),
            dict(kind=hsg.HSG_METROPOLIS_OR, hits=3, proposal=hsg.HSG_PROP_SPHERE, n_or=0, renorm_every=1),
            dict(kind=hsg.HSG_METROPOLIS_OR, hits=2, proposal=hsg.HSG_PROP_BALL, n_or=1),
            dict(kind=hsg.HSG_NONE, n_or=2, renorm_every=2)]


@pytest.mark.parametrize("k", range(6))
@pytest.mark.parametrize("use_stream", [True, False])
def test_batched_lattices_equal_lattices_alone(hsg, k, use_stream):
    kw = kinds(hsg)[k]
    with hsg.Pool(1 << 28, 12, torch.cuda.Stream() if use_stream else None) as pool:
        slots = [pool.admit(*s) for s in SPECS]
        if k % 2:
            hsg.hsg_pool_config(pool.pool, 128, 256, 4, 1)  # one hit per pass
        pool.sweep(hsg.schedule(**kw), 3)
        pool.retire(slots[2])
        late = pool.admit(40, 7, 9, 0, 0.8)
        pool.sweep(hsg.schedule(**kw), 2)
        e = pool.energies()
        for slot, spec in [(s, x) for s, x in zip(slots, SPECS) if x[0] != 108]:
            want, we = alone(hsg, spec, kw, 5)
            assert np.array_equal(pool.spins(slot), want), spec
            assert abs(e[slot] - we) <= 2e-6
            assert pool.sweep_count(slot) == 5
        assert np.array_equal(pool.spins(late), alone(hsg, (40, 7, 9, 0, 0.8), kw, 2)[0])


def test_more_lattices_than_a_batch_holds_and_back_under_the_rule(hsg):
    """60 lattices of L = 32 (three batches by count, on three streams), all but
    three retired (fewer sites than batches are made for), then more again."""
    kw = kinds(hsg)[0]
    sched = hsg.schedule(**kw)
    with hsg.Pool(1 << 27, 64, torch.cuda.Stream()) as pool:
        slots = [pool.admit(32, 5, k, 0, 0.5) for k in range(60)]
        pool.sweep(sched, 2)
        for s in slots[3:]:
            pool.retire(s)
        pool.sweep(sched, 3)
        more = [pool.admit(32, 5, 100 + k, 0, 0.5) for k in range(8)]
        pool.sweep(sched, 2)
        for k, s in enumerate(slots[:3]):
            assert np.array_equal(pool.spins(s), alone(hsg, (32, 5, k, 0, 0.5), kw, 7)[0])
        for k, s in enumerate(more):
            assert np.array_equal(pool.spins(s), alone(hsg, (32, 5, 100 + k, 0, 0.5), kw, 2)[0])


def test_work_queued_around_batches_keeps_its_order(hsg):
    """Sweeps, energies into both buffers, retirements that hand the memory on,
    without a wait between: each energy is that of its lattice at that point."""
    kw = kinds(hsg)[2]
    sched = hsg.schedule(**kw)
    sides = (48, 64, 40, 56)
    nbytes = sum((28 * L ** 3 + 255) // 256 * 256 for L in sides)
    with hsg.Pool(nbytes, 4, torch.cuda.Stream()) as pool:
        got = {}
        for r in range(3):
            slots = [pool.admit(L, 3, 10 * r + i, 0, 0.6) for i, L in enumerate(sides)]
            pool.sweep(sched, 4)
            pool.energies_async(r & 1, slots)
            for s in slots:
                pool.retire(s)
            if r:
                got[r - 1] = pool.energies_read(1 - (r & 1))[:4]
        got[2] = pool.energies_read(0)[:4]
        for r in range(3):
            for i, L in enumerate(sides):
                assert abs(got[r][i] - alone(hsg, (L, 3, 10 * r + i, 0, 0.6), kw, 4)[1]) < 1e-12


def test_a_lattice_beyond_32_bit_offsets(hsg):
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB of device memory")
    L, kw = 814, dict(kind=hsg.HSG_HEATBATH, n_or=1)
    out = torch.empty(3 * L ** 3, device="cuda")
    with hsg.Pool(28 * L ** 3 + 256, 1, torch.cuda.Stream()) as pool:
        slot = pool.admit(L, 1, 0, 0, 0.5)
        pool.sweep(hsg.schedule(**kw), 1)
        hsg.hsg_pool_get_spins(pool.pool, slot, out)
        torch.cuda.synchronize()
    ref = torch.empty_like(out)
    with hsg.Lattice(L, 1) as lat:
        lat.generate_couplings()
        lat.sweep(hsg.schedule(T=0.5, kernel=hsg.HSG_KERNEL_GLOBAL, **kw), 1)
        hsg.hsg_get_spins(lat.ctx, ref)
        torch.cuda.synchronize()
    assert torch.equal(out, ref)


@pytest.mark.parametrize("priority", [0, -1])
def test_side_streams_have_the_pools_priority(hsg, priority):
    with hsg.Pool(1 << 27, 4, torch.cuda.Stream(priority=priority)) as pool:
        pool.admit(64, 7)
        pool.sweep(hsg.schedule(kind=hsg.HSG_HEATBATH), 1)
        own, side = hsg.hsg_test_pool_priorities(pool.pool)
        assert len(side) == 2 and side == [own, own]
        assert (own < 0) == (priority < 0)


@pytest.mark.parametrize("k", range(6))
@pytest.mark.parametrize("use_stream", [True, False])
def test_long_calls_equal_lattices_alone(hsg, k, use_stream):
    """Calls long enough for graphs, whose sweeps the device counts, among short
    ones and over-relaxation alone, which it does not; several batches a lane."""
    kw = kinds(hsg)[k]
    alone_or = dict(kind=hsg.HSG_NONE, n_or=1)
    specs = SPECS + [(96, 7, 10 + j, j & 1, 0.4 + 0.1 * j) for j in range(6)]
    first = [(kw, 9), (kw, 3), (alone_or, 8), (kw, 10)]
    then = [(kw, 8), (kw, 8)]
    with hsg.Pool(1 << 28, 20, torch.cuda.Stream() if use_stream else None) as pool:
        slots = [pool.admit(*s) for s in specs]
        if k % 2:
            hsg.hsg_pool_config(pool.pool, 128, 256, 4, 1)  # one hit per pass
        for s, n in first:
            pool.sweep(hsg.schedule(**s), n)
        pool.retire(slots[2])
        late = pool.admit(40, 7, 90, 0, 0.8)
        for s, n in then:
            pool.sweep(hsg.schedule(**s), n)
        for slot, spec, calls in [(s, x, first + then) for s, x in zip(slots, specs) if x[0] != 108] + [(late, (40, 7, 90, 0, 0.8), then)]:
            L, seed, sample, replica, T = spec
            with hsg.Lattice(L, seed, sample, replica) as lat:
                lat.generate_couplings()
                for s, n in calls:
                    lat.sweep(hsg.schedule(T=T, kernel=hsg.HSG_KERNEL_GLOBAL, **s), n)
                assert np.array_equal(pool.spins(slot), lat.spins()), (L, kw)
                assert pool.sweep_count(slot) == lat.sweep_count


def test_a_long_call_does_not_wait_for_its_sweeps(hsg):
    import time

    with hsg.Pool(1 << 26, 4, torch.cuda.Stream()) as pool:
        for k in range(4):
            pool.admit(64, 7, k)
        sched = hsg.schedule(kind=hsg.HSG_METROPOLIS, hits=4, proposal=hsg.HSG_PROP_BALL, n_or=2)
        pool.sweep(sched, 10)
        torch.cuda.synchronize()
        t0 = time.perf_counter()
        pool.sweep(sched, 1000)  # 6000 half-sweeps
        returned = time.perf_counter() - t0
        torch.cuda.synchronize()
        assert returned < 0.5 * (time.perf_counter() - t0)


@pytest.mark.parametrize("kind,proposal", [("HEATBATH", 0), ("METROPOLIS", 0), ("METROPOLIS_OR", 1)])
def test_a_lattice_beyond_32_bit_offsets_in_a_long_call(hsg, kind, proposal):
    if torch.cuda.mem_get_info()[0] < 60 << 30:
        pytest.skip("needs 60 GB of device memory")
    L, kw = 814, dict(kind=getattr(hsg, "HSG_" + kind), hits=1, proposal=proposal)
    out = torch.empty(3 * L ** 3, device="cuda")
    with hsg.Pool(28 * L ** 3 + 256, 1, torch.cuda.Stream()) as pool:
        slot = pool.admit(L, 1, 0, 0, 0.5)
        pool.sweep(hsg.schedule(**kw), 8)
        hsg.hsg_pool_get_spins(pool.pool, slot, out)
        torch.cuda.synchronize()
    ref = torch.empty_like(out)
    with hsg.Lattice(L, 1) as lat:
        lat.generate_couplings()
        lat.sweep(hsg.schedule(T=0.5, kernel=hsg.HSG_KERNEL_GLOBAL, **kw), 8)
        hsg.hsg_get_spins(lat.ctx, ref)
        torch.cuda.synchronize()
    assert torch.equal(out, ref)
