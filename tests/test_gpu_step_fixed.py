"""The FP64 step in 64-bit fixed point (grids of 196,608 cells and more) against
the oracle: sizes at the edges of its tiles (30 columns x 3 rows, chunks of
layers), sides, plates, implicit vertical diffusion, values of very different
size, and values that are not finite."""
import numpy as np
import pytest

import oracle as O
from tests.gpu_common import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mr():
    import paper_1805_03426_gb300.mr as m
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    m.lib()
    return m


PROBS = {
    "walls_62x58x58": dict(nx=31, ny=29, nz=29, mx=2, my=2, mz=2, gamma=1.5, walls=1),
    "periodic_60x57x60": dict(nx=20, ny=19, nz=20, mx=3, my=3, mz=3, gamma=1.2),
    "narrow_27x128x60": dict(nx=9, ny=64, nz=20, mx=3, my=2, mz=3, lx=0.4),
    "walls_implicit_31x65x100": dict(nx=31, ny=65, nz=25, mx=1, my=1, mz=4, gamma=1.5, walls=1, implicit=1),
    "implicit_adiabatic_91x40x56": dict(nx=91, ny=20, nz=14, mx=1, my=2, mz=4, implicit=1, adiabatic=1, ly=0.5),
    "tall_30x4x1700": dict(nx=10, ny=4, nz=425, mx=3, my=1, mz=4, ly=0.1),
}


def _run(mr, p, T0, steps):
    h = mr.mr_create(p.mr_config(mr, mr.MR_F64))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    mr.mr_refine_velocity(h, dev(p.U), dev(p.V), dev(p.W))
    mr.mr_set_scalar(h, dev(T0))
    mr.mr_scalar_step(h, steps)
    T = torch.empty(T0.shape, dtype=torch.float64, device="cuda")
    mr.mr_get_scalar(h, T)
    out = T.cpu().numpy()
    h.close()
    return out


@pytest.mark.parametrize("name", sorted(PROBS))
def test_steps_match_the_oracle(mr, name):
    # seven steps: the Euler start, leapfrog and averaging steps; a step rounds by
    # a few 2^-53 of the largest value, so 1e-14 in all
    p = Problem(np_average=4, dt=1e-3 if PROBS[name].get("implicit") else 2e-4, ra=1e7, **PROBS[name])
    assert p.T0.size >= 196608
    _, ref = O.run(p.cfg, O.refine(p.cfg, p.U, p.V, p.W), p.T0, 7)
    got = _run(mr, p, p.T0, 7)
    assert np.abs(got - ref).max() <= 1e-14 * np.abs(ref).max()


def test_scaling_by_a_power_of_two_is_exact(mr):
    # zero-flux plates: the scheme is linear, and every scale is relative
    p = Problem(adiabatic=1, dt=2e-4, ra=1e7, **PROBS["periodic_60x57x60"])
    base = _run(mr, p, p.T0, 3)
    for k in (-200, 90):
        assert np.array_equal(_run(mr, p, np.ldexp(p.T0, k), 3), np.ldexp(base, k))


def test_a_wide_range_of_values_keeps_its_local_precision(mr):
    # a blob falling off by 40 decades: every cell is right to FP64 precision of
    # the values around it (a few ulp; the neighbourhood is the tile's share)
    p = Problem(adiabatic=1, dt=2e-4, ra=1e7, **PROBS["walls_62x58x58"])
    Nz, Ny, Nx = p.T0.shape
    z, y, x = np.meshgrid(np.arange(Nz) / Nz - 0.4, np.arange(Ny) / Ny - 0.5, np.arange(Nx) / Nx - 0.3, indexing="ij")
    T0 = np.exp(-250.0 * (x * x + y * y + z * z))
    _, ref = O.run(p.cfg, O.refine(p.cfg, p.U, p.V, p.W), T0, 1)
    got = _run(mr, p, T0, 1)
    pad = np.pad(T0, ((1, 1), (4, 4), (1, 1)))
    near = np.max([pad[1 + a:1 + a + Nz, 4 + b:4 + b + Ny, 1 + c:1 + c + Nx]
                   for a in (-1, 0, 1) for b in range(-4, 5) for c in (-1, 0, 1)], axis=0)
    assert near.min() < 1e-40
    assert (np.abs(got - ref) <= 1e-15 * near).all()


def test_values_that_are_not_finite_stay_where_the_oracle_has_them(mr):
    p = Problem(dt=2e-4, ra=1e7, **PROBS["walls_62x58x58"])
    T0 = p.T0.copy()
    T0[20, 30, 29], T0[21, 3, 61], T0[57, 57, 0] = np.nan, np.inf, -np.inf
    _, ref = O.run(p.cfg, O.refine(p.cfg, p.U, p.V, p.W), T0, 2)
    got = _run(mr, p, T0, 2)
    fine = np.isfinite(ref)
    assert np.array_equal(np.isfinite(got), fine) and not fine.all()
    assert np.abs(got[fine] - ref[fine]).max() <= 1e-14 * np.abs(ref[fine]).max()
