"""The packed node update (both components per operation) on small lattices:
rows that end inside a tile and inside a warp, tiles whose second half has no
rows, one-node axes, each with and without noise and with every relaxation
time 1 or not, against the FP64 oracle.

Tolerance, from the arithmetic: an update rounds each population some thirty
times (2**-24 each), and errors add over the steps as the densities they feed
do, at most linearly: 30 * 2**-24 * steps = 1.8e-6 * steps of the field's mean
magnitude, which the approximations of the noise (2**-21 of a normal of
amplitude sqrt(3 kT rho)) do not reach.
"""
import numpy as np
import pytest

from paper_1909_01092_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 5), (2, 300, 3), (31, 7, 4), (33, 9, 3), (64, 4, 3), (32, 12, 3), (16, 24, 4), (5, 17, 6)]
WALLS = [(1, 1, 0), (0, 0, 0), (0, 1, 1)]


@pytest.fixture(scope="module")
def flbm():
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA")
    from paper_1909_01092_gb300 import binding
    binding.load()
    return binding


@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("kT", [0.0, 1e-5])
@pytest.mark.parametrize("shape", SHAPES)
def test_update_matches_oracle(flbm, oracle_mod, shape, kT, tau):
    steps = 4
    lx, ly, lz = shape
    wall = WALLS[(lx + ly) % len(WALLS)]
    p = W.params(lx=lx, ly=ly, lz=lz, wall=wall, G=1.2, rho_b0=0.4, kT=kT, tau_s=tau, tau_d=(1 + tau) / 2,
                 tau_g=2 - tau, fluid_force=(1e-4, -2e-4, 3e-4))
    f0 = W.random_populations(p, 11).astype(np.float32)
    sim, orc = flbm.Sim(p), oracle_mod.Oracle(p)
    sim.write_f(f0)
    orc.set_f(f0.astype(np.float64))
    sim.step(steps)
    orc.step(steps)
    g, o = sim.read_f().astype(np.float64), orc.get_f()
    sim.close()
    scale = np.mean(np.abs(o), axis=(2, 3, 4), keepdims=True)
    assert np.max(np.abs(g - o) / scale) < 1.8e-6 * steps
