"""The FP64 backward step in 64-bit fixed point (grids of 98,304 cells and more)
against the oracle's discrete adjoint: sizes at the edges of its tiles (30 columns
x 2 rows, chunks of layers), side walls, zero-flux plates, averaging steps, and
adjoint fields that fall off by many decades within a tile."""
import numpy as np
import pytest

import oracle as O
from tests.gpu_common import Problem
from tests.test_gpu_adjoint import _gpu_grad, _oracle_grad, _weights, mr  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LARGE = {
    "walls_62x58x58": dict(nx=31, ny=29, nz=29, mx=2, my=2, mz=2, gamma=1.5, walls=1),
    "periodic_60x57x60": dict(nx=20, ny=19, nz=20, mx=3, my=3, mz=3, gamma=1.2),
    "narrow_27x128x60": dict(nx=9, ny=64, nz=20, mx=3, my=2, mz=3, lx=0.4),
    "adiabatic_91x40x56": dict(nx=91, ny=20, nz=14, mx=1, my=2, mz=4, adiabatic=1, ly=0.5),
    "tall_30x4x1700": dict(nx=10, ny=4, nz=425, mx=3, my=1, mz=4, ly=0.1),
}


def _loss(p, S, wnu, wvar):
    # the oracle adds the 200,000 squares of a variance one after the other in FP64,
    # which is 1.3e-12 off by itself, so its fields' sums are taken in extended precision
    vel = O.refine(p.cfg, p.U, p.V, p.W)
    zf, zc = (p.grid[k].astype(np.longdouble) for k in ("zf", "zc"))
    L = np.longdouble(0.0)
    for s in range(S + 1):
        if wnu[s] == 0.0 and wvar[s] == 0.0:
            continue
        t = (O.run(p.cfg, vel, p.T0, s)[1] if s else p.T0).astype(np.longdouble)
        w = np.diff(zf)[:, None, None] / (zf[-1] - zf[0]) / (t.shape[1] * t.shape[2]) * np.ones(t.shape)
        L += wnu[s] * (0.5 - t[0]).mean() / (zc[0] - zf[0]) + wvar[s] * ((t - (t * w).sum()) ** 2 * w).sum()
    return float(L)


def _compare(mr, p, S, ck, wnu, wvar):
    # every sum is a few hundred FP64 roundings of its largest term: 1e-12 in all
    L, g = _gpu_grad(mr, p, mr.MR_F64, S, ck, wnu, wvar)
    Lr = _loss(p, S, wnu, wvar)
    _, gr = _oracle_grad(p, S, wnu, wvar)
    assert abs(L - Lr) <= 1e-12 * abs(Lr)
    for a, b in zip(g, gr):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


@pytest.mark.parametrize("name", sorted(LARGE))
def test_backward_steps_match_the_oracle(mr, name):  # noqa: F811
    p = Problem(np_average=4, dt=2e-4, ra=1e7, **LARGE[name])
    assert p.T0.size >= 196608
    _compare(mr, p, 7, 3, *_weights(7))


@pytest.mark.parametrize("name", ["walls_62x58x58", "periodic_60x57x60"])
def test_adjoint_of_the_last_heat_flux_alone(mr, name):  # noqa: F811
    # the adjoint starts on one layer and falls off by decades per layer
    p = Problem(np_average=4, dt=2e-4, ra=1e7, **LARGE[name])
    wnu, wvar = np.zeros(6), np.zeros(6)
    wnu[-1] = 1.0
    _compare(mr, p, 5, 5, wnu, wvar)


@pytest.mark.parametrize("walls", [0, 1])
@pytest.mark.parametrize("ny", [23, 24])
def test_grids_on_both_sides_of_the_smallest_one(mr, ny, walls):  # noqa: F811
    # 94,208 cells (FP64 arithmetic) and 98,304
    p = Problem(32, ny, 16, 2, 2, 2, gamma=1.2, walls=walls, np_average=4, dt=2e-4, ra=1e7)
    _compare(mr, p, 7, 3, *_weights(7))
