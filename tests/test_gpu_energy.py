"""hsg_energy (one launch, the last block's sum, result in pinned memory)
against the logged energy (two launches), bit for bit (needs a CUDA GPU)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 4: one block; 6, 8: one full and a ragged block; 70, 72: either side of 672
# blocks, 74: the cap of 760; 130: many sites per thread
@pytest.mark.parametrize("L", [4, 6, 8, 10, 70, 72, 74, 130])
@pytest.mark.parametrize("layout", [0, 1])
def test_energy_equals_the_logged_energy(L, layout):
    from paper_1006_2566_gb300 import build

    build.build()
    from paper_1006_2566_gb300 import hsg

    with hsg.Lattice(L, 9, stream=torch.cuda.Stream(), layout=layout) as lat:
        lat.generate_couplings()
        for k in range(3):  # the ticket is back at zero every time
            lat.sweep(hsg.schedule(kind=hsg.HSG_HEATBATH, T=0.8, energy_every=1), 1)
            assert lat.energy() == lat.energy() == lat.energy_log()[k]
