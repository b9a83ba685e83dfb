"""The ensemble's bulk collide over work lists: more replicas of one kernel
variant than a launch takes descriptors, persistent blocks that walk several
items of different replicas, every packing. Each is the same arithmetic, so
the populations equal those of one block per tile bit for bit."""
import numpy as np
import pytest

from paper_1909_01092_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _members():
    out = []
    for r in range(70):  # 54 with noise, 8 without, 8 with other relaxation times
        kw = dict(tau_s=0.8) if r % 9 == 4 else {}
        out.append(W.params(lx=9 + r % 13, ly=8 + r % 11, lz=12 + r % 7, radius=2.5 if r % 3 else 0.0, g=1e-5,
                            kT=0.0 if r % 9 == 7 else 1e-5, replica=r, **kw))
    return out


@pytest.fixture(scope="module")
def per_tile():
    from paper_1909_01092_gb300 import binding

    binding.load(build_if_missing=True)
    return _run(binding, 0, 0)


def _run(binding, packing, ctas):
    ens = binding.Ensemble(_members(), config=dict(packing=packing, ctas_per_sm=ctas, tile_policy=0))
    ens.step(5)
    got = [ens.read_f(r) for r in range(70)], [p["X"] for p in ens.particles()]
    ens.close()
    return got


@pytest.mark.parametrize("packing,ctas", [(0, 1), (1, 1), (2, 1), (1, 3), (0, 4), (1, 4), (2, 8)])
def test_lists_equal_one_block_per_tile(per_tile, packing, ctas):
    from paper_1909_01092_gb300 import binding

    f, X = _run(binding, packing, ctas)
    for r in range(70):
        assert np.array_equal(f[r], per_tile[0][r], equal_nan=True), r
        assert np.array_equal(X[r], per_tile[1][r]), r
