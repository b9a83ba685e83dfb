"""The observables reduction (double-float pass, FP64 for marked blocks) on
small and ragged lattices against numpy in FP64.

Tolerance: a double-float keeps 48 bits and a node's values take at most some
thirty operations each, so a value v formed from terms whose magnitudes add up
to M is good to d = 30 * 2**-48 M < 2**-42 M (FP64 on both sides has less), a
sum of values to the sum of their d, and a sum of squares to the sum of
2 |v| d + d**2.
"""
import numpy as np
import pytest

from paper_1909_01092_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = 2.0 ** -42


@pytest.fixture(scope="module")
def flbm():
    import torch
    if not torch.cuda.is_available():
        raise RuntimeError("GPU tests need CUDA")
    from paper_1909_01092_gb300 import binding
    binding.load()
    return binding


C = np.array([(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
              (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1),
              (0, 1, -1), (0, -1, 1)], dtype=float)
w = np.array([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12)


def _basis():
    x, y, z = C.T
    q = (C * C).sum(1)
    d, e = 3 * x * x - q, y * y - z * z
    return np.array([np.ones(19), x, y, z, q - 1, d, e, x * y, y * z, x * z, (3 * q - 5) * x, (3 * q - 5) * y,
                     (3 * q - 5) * z, (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z,
                     3 * q * q - 6 * q + 1, (2 * q - 3) * d, (2 * q - 3) * e])


def _expected(f):
    """Each observable of a field without a particle, and its tolerance."""
    E = _basis()
    b = (E * E * w).sum(1)
    f = f.astype(np.float64)
    m, M = (np.einsum("ki,lizyx->lkzyx", e, v) for e, v in ((E, f), (np.abs(E), np.abs(f))))
    rho, j, J = m[:, 0], m[0, 1:4] + m[1, 1:4], M[0, 1:4] + M[1, 1:4]
    rt = rho.sum(0)
    u, U = j / rt, J / rt
    both = lambda v: (np.sum(v * v, 0), 3 * v[0] ** 2, v[1] ** 2 + v[2] ** 2, v[0] * v[1], v[1] * v[2],  # noqa: E731
                      v[0] * v[2])
    uu = (u * u).sum(0)
    eq = [uu, 3 * u[0] ** 2 - uu, u[1] ** 2 - u[2] ** 2, u[0] * u[1], u[1] * u[2], u[0] * u[2]]
    top = lambda M, k: M + sum(both(U)[:2]) * rho.max() if k <= 9 else M  # noqa: E731

    def squares(v, size, axes=None):
        d = TOL * size
        return (v * v).sum(axes), (2 * np.abs(v) * d + d * d).sum(axes)

    mt, mt_tol = np.zeros((2, 19)), np.zeros((2, 19))
    for l in range(2):
        if rho[l].sum() <= 0:
            continue
        for k in range(4, 19):
            n = m[l, k] - rho[l] * eq[k - 4] if k <= 9 else m[l, k]
            s, tol = squares(n, top(M[l, k], k))
            mt[l, k], mt_tol[l, k] = (v / (3 * b[k] * rho[l].sum()) for v in (s, tol))
    mt_tol += TOL * mt
    d, D = (rho[1] * m[0, 1:4] - rho[0] * m[1, 1:4]) / rt, (rho[1] * M[0, 1:4] + rho[0] * M[1, 1:4]) / rt
    ab = (rho[0] * rho[1] / rt).sum()
    dt, dt_tol = squares(d, D, (1, 2, 3))
    dt, dt_tol = (dt / ab, dt_tol / ab + TOL * dt / ab) if ab > 0 else (np.zeros(3), np.zeros(3))
    jt, jt_tol = squares(j, J, (1, 2, 3))
    ke, ke_tol = (j * j / (2 * rt)).sum(), (TOL * (2 * np.abs(j) * J + J * J * TOL) / rt).sum()
    return dict(mass=(rho.sum((1, 2, 3)), TOL * M[:, 0].sum((1, 2, 3))),
                momentum=(j.sum((1, 2, 3)), TOL * J.sum((1, 2, 3))), kinetic=(ke, ke_tol), mode_temp=(mt, mt_tol),
                diff_temp=(dt, dt_tol), mom_temp=(jt / rt.sum(), jt_tol / rt.sum() + TOL * jt / rt.sum()))


def _field(p, kind):
    f = W.random_populations(p, 5).astype(np.float32)
    if kind == "large":      # one node above the double-float pass's range
        f[0, 3, -1, -1, -1] = 5.0e4
    elif kind == "tiny":     # component B below it everywhere
        f[1] *= np.float32(1e-12)
    elif kind == "no_b":     # B absent: in range
        f[1] = 0.0
    return f


@pytest.mark.parametrize("kind", ["ordinary", "large", "tiny", "no_b"])
@pytest.mark.parametrize("shape", [(1, 1, 1), (1, 300, 3), (5, 17, 6), (33, 9, 40), (64, 12, 70)])
def test_sums_match_fp64(flbm, shape, kind):
    lx, ly, lz = shape
    p = W.params(lx=lx, ly=ly, lz=lz, wall=(1, 0, 0), rho_b0=0.3)
    f = _field(p, kind)
    sim = flbm.Sim(p)
    sim.write_f(f)
    o = sim.observables()
    sim.close()
    assert o["n_bulk"] == o["nfluid"] == lx * ly * lz and o["nonfinite"] == 0
    for name, (v, tol) in _expected(f).items():
        assert np.all(np.abs(o[name] - v) <= tol), name


def test_nonfinite_populations_are_counted(flbm):
    p = W.params(lx=20, ly=9, lz=33, wall=(1, 1, 0), rho_b0=0.3)
    f = W.random_populations(p, 6).astype(np.float32)
    f[0, 2, 30, 4, 7] = np.nan
    f[1, 0, 2, 8, 19] = np.inf
    f[1, 5, 2, 8, 19] = -np.inf
    sim = flbm.Sim(p)
    sim.write_f(f)
    o = sim.observables(allow_nonfinite=True)
    sim.close()
    assert o["nonfinite"] == 3
    assert np.isnan(o["mass"]).all()
