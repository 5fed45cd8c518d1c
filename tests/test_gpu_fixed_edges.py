"""The fixed-point FP64 steps where their scales and coefficients matter: a constant
scalar in a box at rest, zeros of either sign beside large values, the scalar's sign,
a face velocity far above all others."""
import numpy as np
import pytest

import oracle as O
from tests.gpu_common import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PERIODIC = dict(nx=20, ny=19, nz=20, mx=3, my=3, mz=3, gamma=1.2)     # 60 x 57 x 60 dense cells
WALLS = dict(nx=31, ny=29, nz=29, mx=2, my=2, mz=2, gamma=1.5, walls=1)


@pytest.fixture(scope="module")
def mr():
    import paper_1805_03426_gb300.mr as m
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    m.lib()
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _run(mr, p, T0, steps, vel=None):
    h = mr.mr_create(p.mr_config(mr, mr.MR_F64))
    mr.mr_refine_velocity(h, *(dev(a) for a in (vel or (p.U, p.V, p.W))))
    mr.mr_set_scalar(h, dev(T0))
    mr.mr_scalar_step(h, steps)
    T = torch.empty(T0.shape, dtype=torch.float64, device="cuda")
    mr.mr_get_scalar(h, T)
    out = T.cpu().numpy()
    h.close()
    return out


@pytest.mark.parametrize("zero", [0.0, -0.0])
@pytest.mark.parametrize("prob", [PERIODIC, WALLS])
def test_zeros_of_either_sign_stay_zero_beside_large_values(mr, prob, zero):
    p = Problem(adiabatic=1, dt=2e-4, ra=1e7, **prob)
    Nz, Ny, Nx = p.T0.shape
    T0 = np.where(np.arange(Nx) < Nx // 2, 1.0 + p.T0, zero)
    got = _run(mr, p, T0, 2)
    # two steps reach two cells
    assert not got[:, :, Nx // 2 + 2:Nx - 2].any() and got[:, :, Nx // 2].any()


@pytest.mark.parametrize("prob", [PERIODIC, WALLS])
@pytest.mark.parametrize("dt", [1e-3, 2e-3, 4e-3])
def test_a_constant_scalar_stays_constant(mr, prob, dt):
    # zero-flux plates, nothing moves: what leaves a cell is what its neighbours give
    p = Problem(adiabatic=1, dt=dt, ra=1e4, **prob)
    ones = np.ones(p.T0.shape)
    assert (_run(mr, p, ones, 4, vel=tuple(0.0 * a for a in (p.U, p.V, p.W))) == 1.0).all()


@pytest.mark.parametrize("prob", [PERIODIC, WALLS])
def test_the_negative_scalar_steps_to_the_negative(mr, prob):
    # to rounding: either result is within a unit in the last place of the largest value
    p = Problem(adiabatic=1, dt=2e-3, ra=1e7, **prob)
    a, b = _run(mr, p, p.T0, 1), _run(mr, p, -p.T0, 1)
    assert np.abs(a + b).max() <= 2 * np.spacing(np.abs(a).max())


def _one_large_face(p, comp, factor):
    """The coarse velocity with one face of one component `factor` times the largest one,
    and the dense cells more than four coarse cells away from it on some axis: three that
    its refinement reaches, if only by rounding, and one for the steps."""
    vel = [p.U.copy(), p.V.copy(), p.W.copy()]
    at = tuple(n // 2 for n in vel[comp].shape)
    vel[comp][at] = factor * max(np.abs(a).max() for a in vel)
    Nz, Ny, Nx = p.T0.shape
    far = np.zeros(p.T0.shape, bool)
    for axis, m, N in ((0, p.kw["mz"], Nz), (1, p.kw["my"], Ny), (2, p.kw["mx"], Nx)):
        shape = [1, 1, 1]
        shape[axis] = N
        far |= (np.abs(np.arange(N) // m - at[axis]) > 4).reshape(shape)
    return tuple(vel), far


@pytest.mark.parametrize("prob", [PERIODIC, WALLS])
@pytest.mark.parametrize("comp", [0, 1, 2])
@pytest.mark.parametrize("factor", [1e3, 1e9, 1e30])
def test_one_large_face_leaves_the_others_their_precision(mr, prob, comp, factor):
    # a time step that suits the other faces: around this one the scalar runs away, beyond
    # its reach (a dense cell per step) a step rounds by a few 2^-53 as it does without it
    p = Problem(dt=2e-4, ra=1e7, **prob)
    vel, far = _one_large_face(p, comp, factor)
    _, ref = O.run(p.cfg, O.refine(p.cfg, *vel), p.T0, 2)
    got = _run(mr, p, p.T0, 2, vel=vel)
    assert far.sum() > p.T0.size // 2 and np.abs(ref[far]).max() < 1.0
    assert np.abs(got - ref)[far].max() <= 1e-14


@pytest.mark.parametrize("prob", [PERIODIC, WALLS])
def test_one_large_face_leaves_the_adjoint_its_precision(mr, prob):
    from tests.test_gpu_adjoint import _gpu_grad, _oracle_grad, _weights

    p = Problem(dt=2e-4, ra=1e7, **prob)
    (p.U, p.V, p.W), far = _one_large_face(p, 0, 1e6)
    wnu, wvar = _weights(2)
    wvar[:] = 0.0            # heat fluxes: the loss weighs every cell alike
    _, g = _gpu_grad(mr, p, mr.MR_F64, 2, 2, wnu, wvar)
    _, gr = _oracle_grad(p, 2, wnu, wvar)
    a, b = np.asarray(g[0])[far], np.asarray(gr[0])[far]
    assert np.abs(b).max() > 0.0 and np.abs(a - b).max() <= 1e-12 * np.abs(b).max()
