"""TMA-staged collide where its blocks walk several tiles each: both stages in
use, stages refilled during an update, ragged shares of tiles. It computes the
same update as the kernel that reads global memory directly, from the same
inputs, so every population agrees bit for bit."""
import pytest

from paper_1909_01092_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# Up to 16 blocks are launched per SM, 2432 on 152 SMs.
CASES = [
    dict(lx=64, ly=64, lz=152, radius=0.0, kT=1e-5),                                # 2432 tiles: one each
    dict(lx=64, ly=64, lz=153, radius=0.0, kT=0.0),                                 # one block has a second
    dict(lx=68, ly=60, lz=330, radius=4.0, kT=0.0, g=2e-4, tau_s=0.8),              # 7920 ragged tiles, up to four
    dict(lx=128, ly=128, lz=150, wall=(1, 1, 0), radius=6.0, kT=1e-5, g=1e-5),      # 9600 tiles
]


@pytest.mark.parametrize("case", range(len(CASES)))
def test_many_tiles_per_block_equal_the_direct_kernel(case):
    from paper_1909_01092_gb300 import binding

    binding.load(build_if_missing=True)
    p = W.params(**CASES[case])
    got = []
    for tma in (True, False):
        sim = binding.Sim(p)
        sim.use_tma(tma)
        sim.set_density_mode(0)
        sim.step(5)
        got.append((sim.particle()["X"].tolist(), sim.read_f()))
        sim.close()
    assert got[0][0] == got[1][0]
    assert (got[0][1] == got[1][1]).all()
