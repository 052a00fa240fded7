"""The global half-sweep kernels at the sizes where their launch rule changes
(needs a CUDA GPU): one, two or four rows per thread, the heat-bath's column
march, 32- and 64-bit byte offsets, both spin layouts.  The slab kernel, which
shares none of their index arithmetic, has to give the same bits."""
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


def updates(hsg):
    return [(hsg.HSG_OVERRELAX, 0, 1), (hsg.HSG_HEATBATH, 0, 1), (hsg.HSG_METROPOLIS, 0, 2), (hsg.HSG_METROPOLIS, 1, 3),
            (hsg.HSG_METROPOLIS_OR, 0, 2), (hsg.HSG_METROPOLIS_OR, 1, 2), (hsg.HSG_METROPOLIS, 1, 1),
            (hsg.HSG_METROPOLIS_OR, 0, 1)]


def sweep_halves(hsg, lat, kernel):
    for upd, prop, hits in updates(hsg):
        for colour in (0, 1):
            lat.half_sweep(hsg.schedule(T=0.7, hits=hits, proposal=prop, kernel=kernel), upd, colour)


# 4, 6: the smallest; 94 | 96: one | two rows; 142 | 144: colour 1 from the top down; 150 | 152, 154: the heat-bath's
# column march; 122 | 124 | 224: ball, many hits, one | two | four rows; 158 | 160: packed two rows
@pytest.mark.parametrize("L", [4, 6, 94, 96, 122, 124, 142, 144, 150, 152, 154, 158, 160, 224, 226])
def test_global_kernels_equal_the_slab_kernel(hsg, L):
    outs = []
    for layout, kernel in ((hsg.HSG_LAYOUT_FLOAT4, hsg.HSG_KERNEL_SLAB), (hsg.HSG_LAYOUT_FLOAT4, hsg.HSG_KERNEL_GLOBAL),
                           (hsg.HSG_LAYOUT_PACKED, hsg.HSG_KERNEL_GLOBAL)):
        with hsg.Lattice(L, 17, 2, 1, layout=layout) as lat:
            lat.generate_couplings()
            sweep_halves(hsg, lat, kernel)
            outs.append(lat.spins())
    assert np.array_equal(outs[0], outs[1])
    assert np.array_equal(outs[0], outs[2])


@pytest.mark.parametrize("L", [812, 814])
def test_either_side_of_the_32_bit_offsets(hsg, L):
    """16 L^3/2 passes 2^32 between L = 812 and 814: random sites, the
    corners and the last plane."""
    rng = np.random.default_rng(L)
    sites = np.concatenate([rng.integers(0, L ** 3, 4000), L ** 3 - 1 - rng.integers(0, L * L, 2000),
                            rng.integers(0, L * L, 2000), [0, L - 1, L * L - 1, L ** 3 - 1]]).astype(np.uint32)
    outs = []
    for layout, kernel in ((hsg.HSG_LAYOUT_FLOAT4, hsg.HSG_KERNEL_SLAB), (hsg.HSG_LAYOUT_FLOAT4, hsg.HSG_KERNEL_GLOBAL),
                           (hsg.HSG_LAYOUT_PACKED, hsg.HSG_KERNEL_GLOBAL)):
        with hsg.Lattice(L, 3, layout=layout) as lat:
            lat.generate_couplings()
            sweep_halves(hsg, lat, kernel)
            outs.append(hsg.hsg_get_sites(lat.ctx, sites, want_bonds=False)[0])
    assert np.array_equal(outs[0], outs[1])
    assert np.array_equal(outs[0], outs[2])


# either side of where launches overlap the next one, and how: over-relaxation
# up to 72, the other updates up to 90 and up to 126
@pytest.mark.parametrize("L", [34, 72, 74, 90, 92, 126, 128])
@pytest.mark.parametrize("use_stream", [True, False])
def test_overlapping_launches_equal_the_slab_kernel(hsg, L, use_stream):
    for kw in (dict(kind=hsg.HSG_HEATBATH, n_or=2), dict(kind=hsg.HSG_METROPOLIS, hits=2, proposal=1, n_or=1),
               dict(kind=hsg.HSG_METROPOLIS_OR, hits=1, n_or=0)):
        outs = []
        for layout, kernel in ((0, hsg.HSG_KERNEL_SLAB), (0, hsg.HSG_KERNEL_GLOBAL), (1, hsg.HSG_KERNEL_GLOBAL)):
            stream = torch.cuda.Stream() if use_stream else None
            with hsg.Lattice(L, 31, stream=stream, layout=layout) as lat:
                lat.generate_couplings()
                sched = hsg.schedule(T=0.7, kernel=kernel, renorm_every=3, energy_every=2, **kw)
                lat.sweep(sched, 1)
                lat.sweep_count = 6
                lat.sweep(sched, 13)
                lat.half_sweep(sched, hsg.HSG_HEATBATH, 1)
                outs.append((lat.spins(), lat.energy_log(), lat.energy()))
        for o in outs[1:]:
            assert all(np.array_equal(a, b) for a, b in zip(o, outs[0]))


@pytest.mark.parametrize("kernel,n_or", [(1, 2), (3, 1), (3, 2)])
def test_graphs_without_cadences_equal_direct_launches(hsg, kernel, n_or):
    """Without cadences a graph holds as many sweeps as one call's number
    allows: calls of other lengths, a change of schedule, new spins and a
    counter set by hand in between."""
    L = 40
    outs = []
    for stream in (torch.cuda.Stream(), None):
        with hsg.Lattice(L, 13, stream=stream) as lat:
            lat.generate_couplings()
            sched = hsg.schedule(kind=hsg.HSG_HEATBATH, T=0.6, n_or=n_or, kernel=kernel)
            other = hsg.schedule(kind=hsg.HSG_METROPOLIS, T=0.6, n_or=1, kernel=kernel)
            got = []
            for n, sc in ((1, sched), (5, sched), (5, sched), (3, sched), (50, sched), (20, other), (2, sched), (17, sched),
                          (33, sched), (7, other), (7, other)):
                lat.sweep(sc, n)
                got.append((lat.energy(), lat.sweep_count))
            lat.sweep_count = 2 ** 32 - 5
            lat.sweep(sched, 12)
            lat.set_spins(lat.spins()[::-1].copy())
            lat.sweep(sched, 12)
            outs.append((got, lat.sweep_count, lat.spins()))
    assert outs[0][0] == outs[1][0] and outs[0][1] == outs[1][1]
    assert np.array_equal(outs[0][2], outs[1][2])
