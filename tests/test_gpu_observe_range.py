"""Observables of finite states far from equilibrium, and their precision
against exact rational arithmetic.

Fields: populations of a node that nearly cancel (velocity 2e5), and component
densities of opposite sign that do (interdiffusion momentum 3e7). Every
population is a multiple of 2**-12 below 2**14, so the node sums are exact, no
value of these nodes is a small difference, and a value takes fewer than 60
roundings; the sum over N nodes adds at most N more: tolerance
(N + 64) 2**-53 of each value.

Precision: a single node whose components move together in float-rounded
equilibrium, so that rho_B j_A and rho_A j_B differ in their roundings only.
The sums rho and j of 19 floats of similar size are exact in FP64, so d rounds
two products, uniformly within 2**-53 of them: 0.58 sqrt(2) < 1 unit of 2**-53
of a product in the root mean square, 4 allowed.
"""
from fractions import Fraction

import numpy as np
import pytest

from paper_1909_01092_gb300 import workloads as W
from test_gpu_observe import C, _basis, w

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def flbm():
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA")
    from paper_1909_01092_gb300 import binding
    binding.load()
    return binding


def _field(kind, shape):
    lx, ly, lz = shape
    f = np.zeros((2, 19, lz, ly, lx), dtype=np.float32)
    f[:] = np.array([0.25] + [0.0625] * 6 + [0.03125] * 12, dtype=np.float32)[None, :, None, None, None]
    if kind == "populations":
        f[:, :, 3, 2, 5] = 0.0
        f[0, 1, 3, 2, 5] = 100.0
        f[0, 2, 3, 2, 5] = -(100.0 - 2.0 ** -10)
    else:
        f *= 8192.0
        f[:, :, 7, 9, 30] = 0.0
        f[0, 1, 7, 9, 30] = 64.0
        f[1, 2, 7, 9, 30] = -(64.0 - 2.0 ** -12)
    return f


def _expected(f):
    E = _basis()
    b = (E * E * w).sum(1)
    m = np.einsum("ki,lizyx->lkzyx", E, f.astype(np.float64))
    rho, j = m[:, 0], m[0, 1:4] + m[1, 1:4]
    rt = rho.sum(0)
    u = j / rt
    uu = (u * u).sum(0)
    eq = [uu, 3 * u[0] ** 2 - uu, u[1] ** 2 - u[2] ** 2, u[0] * u[1], u[1] * u[2], u[0] * u[2]]
    mt = np.zeros((2, 19))
    for l in range(2):
        for k in range(4, 19):
            n = m[l, k] - rho[l] * eq[k - 4] if k <= 9 else m[l, k]
            mt[l, k] = (n * n).sum() / (3 * b[k] * rho[l].sum())
    d = (rho[1] * m[0, 1:4] - rho[0] * m[1, 1:4]) / rt
    ab = (rho[0] * rho[1] / rt).sum()
    assert ab > 0 and (rho.sum((1, 2, 3)) > 0).all()
    return dict(mass=rho.sum((1, 2, 3)), momentum=j.sum((1, 2, 3)), kinetic=(j * j / (2 * rt)).sum(), mode_temp=mt,
                diff_temp=(d * d).sum((1, 2, 3)) / ab, mom_temp=(j * j).sum((1, 2, 3)) / rt.sum())


@pytest.mark.parametrize("kind", ["populations", "densities"])
def test_finite_states_give_finite_observables(flbm, kind):
    shape = (40, 16, 20)
    p = W.params(lx=40, ly=16, lz=20, wall=(1, 0, 0), rho_b0=0.3)
    f = _field(kind, shape)
    sim = flbm.Sim(p)
    sim.write_f(f)
    o = sim.observables()
    sim.close()
    n = 40 * 16 * 20
    assert o["nonfinite"] == 0 and o["nfluid"] == o["n_bulk"] == n
    for name, v in _expected(f).items():
        got = np.asarray(o[name])
        assert np.isfinite(got).all(), name
        assert np.all(np.abs(got - v) <= (n + 64) * 2.0 ** -53 * np.abs(v)), name


def test_small_differences_have_fp64_precision(flbm):
    rng = np.random.default_rng(3)
    E = _basis()
    p = W.params(lx=1, ly=1, lz=1, wall=(0, 0, 0), rho_b0=0.3)
    sim = flbm.Sim(p)
    off = []
    for _ in range(64):
        u = rng.uniform(-0.1, 0.1, 3)
        cu = C @ u
        rho = (rng.uniform(0.5, 2.0), rng.uniform(0.05, 0.5))
        f = np.array([r * w * (1 + 3 * cu + 4.5 * cu ** 2 - 1.5 * (u @ u)) for r in rho]).astype(np.float32)
        sim.write_f(f.reshape(2, 19, 1, 1, 1))
        got = np.asarray(sim.observables()["diff_temp"])
        m = [[sum((int(E[k][i]) * Fraction(float(f[l][i])) for i in range(19)), Fraction(0)) for k in range(4)]
             for l in range(2)]
        rt = m[0][0] + m[1][0]
        ab = float(m[0][0] * m[1][0] / rt)
        for a in range(3):
            d = float(abs(m[1][0] * m[0][1 + a] - m[0][0] * m[1][1 + a]) / rt)
            unit = 2.0 ** -53 * float(abs(m[1][0] * m[0][1 + a]) / rt)
            off.append((np.sqrt(got[a] * ab) - d) / unit)
    sim.close()
    assert np.sqrt(np.mean(np.square(off))) < 4.0
