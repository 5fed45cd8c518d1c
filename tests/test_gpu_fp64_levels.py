"""FP64 runs whose velocity changes, on grids of the fixed-point step (196,608 cells and
more): temporal refinement, staged hand-overs and coupled steps against the oracle, with
velocities of very different size one after the other (the step's scales follow the
current one)."""
import numpy as np
import pytest

import oracle as O
from paper_1805_03426_gb300 import synth
from tests.gpu_common import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROBS = {
    "walls": dict(nx=31, ny=29, nz=29, mx=2, my=2, mz=2, gamma=1.5, walls=1),
    "periodic_implicit": dict(nx=20, ny=19, nz=20, mx=3, my=3, mz=3, gamma=1.2, implicit=1),
}
SIZES = (1.0, 1.0 / 64.0, 40.0, 1e-7, 1.0)     # of the velocities, one after the other


@pytest.fixture(scope="module")
def mr():
    import paper_1805_03426_gb300.mr as m
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    m.lib()
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _problem(name):
    # at 40 times the first velocity a step is still within its stability limit
    p = Problem(np_average=4, dt=1e-5, ra=1e7, **PROBS[name])
    assert p.T0.size >= 196608
    g = p.grid
    vels = [tuple(f * a for a in synth.coarse_velocity(5 + n, g["Xf"], g["Yf"], g["Zf"], rms=0.2, walls=bool(p.kw["walls"])))
            for n, f in enumerate(SIZES)]
    return p, vels


def _levels(mr, h, p):
    T = torch.empty(p.T0.shape, dtype=torch.float64, device="cuda")
    Tp = torch.empty_like(T)
    mr.mr_get_scalar(h, T, Tp)
    return T.cpu().numpy(), Tp.cpu().numpy()


def _agree(got, ref):
    # a handful of steps, each a few roundings of the largest value
    assert np.abs(got - ref).max() <= 2e-14 * np.abs(ref).max()


@pytest.mark.parametrize("name", sorted(PROBS))
def test_temporal_refinement(mr, name):
    p, vels = _problem(name)
    h = mr.mr_create(p.mr_config(mr, mr.MR_F64))
    mr.mr_refine_velocity(h, *(dev(a) for a in vels[0]))
    mr.mr_set_scalar(h, dev(p.T0))
    mr.mr_scalar_step(h, 1)
    dense = [O.refine(p.cfg, *v) for v in vels]
    Tm, T = O.run(p.cfg, dense[0], p.T0, 1)
    s = 1
    for n, mt in enumerate((2, 1, 3, 2)):
        mr.mr_scalar_coarse_step(h, *(dev(a) for a in vels[n + 1]), mt)
        Tm, T = O.coarse_step(p.cfg, dense[n], dense[n + 1], Tm, T, s, mt)
        s += mt
    mr.mr_scalar_step(h, 1)                      # with the last velocity alone
    Tm, T = O.coarse_step(p.cfg, dense[-1], dense[-1], Tm, T, s, 1)
    got, prev = _levels(mr, h, p)
    _agree(got, T)
    _agree(prev, Tm)
    h.close()


@pytest.mark.parametrize("staged", [False, True])
@pytest.mark.parametrize("name", sorted(PROBS))
def test_coupled_steps(mr, name, staged):
    p, vels = _problem(name)
    h = mr.mr_create(p.mr_config(mr, mr.MR_F64))
    mr.mr_set_scalar(h, dev(p.T0))
    nu = torch.zeros(2, dtype=torch.float64, device="cuda")
    Tc = torch.zeros((p.kw["nz"], p.kw["ny"], p.kw["nx"]), dtype=torch.float64, device="cuda")
    Tm = T = p.T0
    for s, v in enumerate(vels):
        if staged:
            mr.mr_stage_velocity(h, *(dev(a) for a in v))
            mr.mr_refine_velocity_staged(h)
        else:
            mr.mr_refine_velocity(h, *(dev(a) for a in v))
        mr.mr_scalar_step_coupled(h, nu, Tc)
        d = O.refine(p.cfg, *v)
        Tm, T = O.coarse_step(p.cfg, d, d, Tm, T, s, 1)
    got, prev = _levels(mr, h, p)
    _agree(got, T)
    _agree(prev, Tm)
    st = O.stats(p.cfg, T)
    for k, name_ in enumerate(("nu_bot", "nu_top")):
        assert abs(nu.cpu().numpy()[k] - st[name_]) <= 1e-11 * max(1.0, abs(st[name_]))
    w = np.diff(p.grid["zf"])[:, None, None]
    c = (T * w).reshape(p.kw["nz"], p.kw["mz"], p.kw["ny"], p.kw["my"], p.kw["nx"], p.kw["mx"]).sum((1, 3, 5))
    c /= w.reshape(p.kw["nz"], p.kw["mz"]).sum(1)[:, None, None] * p.kw["my"] * p.kw["mx"]
    _agree(Tc.cpu().numpy(), c)
    h.close()
