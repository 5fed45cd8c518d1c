"""Steps on both sides of the rules that choose how a step is launched, against the
oracle: FP64 grids whose blocks fit the chip twice, once and more often, fourth-order
FP32 grids from 4 M cells (their own kernel) and below, coupled steps over plate sizes."""
import numpy as np
import pytest

import oracle as O
from tests.gpu_common import Problem
from tests.test_gpu_adjoint import _gpu_grad, _oracle_grad, _weights

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def mr():
    import paper_1805_03426_gb300.mr as m
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    m.lib()
    return m


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _run(mr, p, precision, steps):
    h = mr.mr_create(p.mr_config(mr, precision))
    mr.mr_refine_velocity(h, dev(p.U), dev(p.V), dev(p.W))
    mr.mr_set_scalar(h, dev(p.T0))
    mr.mr_scalar_step(h, steps)
    T = torch.empty(p.T0.shape, dtype=torch.float64, device="cuda")
    mr.mr_get_scalar(h, T)
    out = T.cpu().numpy()
    h.close()
    return out


# dense rows of 64, four rows a block: 440, 480 and 720 blocks
@pytest.mark.parametrize("n", [(24, 22, 20), (26, 24, 20), (32, 30, 24)])
@pytest.mark.parametrize("form", [dict(), dict(walls=1), dict(face_order=4), dict(implicit=1)])
def test_fp64_steps(mr, n, form):
    p = Problem(*n, gamma=1.2, dt=2e-4, ra=1e7, np_average=4, **form)
    assert p.T0.size < 196608
    _, ref = O.run(p.cfg, O.refine(p.cfg, p.U, p.V, p.W), p.T0, 9)
    assert np.abs(_run(mr, p, mr.MR_F64, 9) - ref).max() <= 2e-14 * np.abs(ref).max()


@pytest.mark.parametrize("n", [(20, 18, 16), (24, 22, 20)])
def test_fp64_backward_steps(mr, n):
    p = Problem(*n, gamma=1.2, dt=2e-4, ra=1e7, np_average=4)
    w = _weights(9)
    _, g = _gpu_grad(mr, p, mr.MR_F64, 9, 4, *w)
    _, gr = _oracle_grad(p, 9, *w)
    for a, b in zip(g, gr):
        assert np.abs(a - b).max() <= 1e-12 * np.abs(b).max()


# 160 x 160 x 160 cells and 160 x 166 x 160 (4.10 M, 4.25 M; the rule's 4 M is 4,194,304)
@pytest.mark.parametrize("ny", [80, 83])
@pytest.mark.parametrize("form", [dict(), dict(walls=1), dict(implicit=1)])
def test_fourth_order_fp32_steps(mr, ny, form):
    p = Problem(80, ny, 80, gamma=1.2, dt=2e-4, ra=1e7, np_average=4, face_order=4, **form)
    assert (p.T0.size >= 4 << 20) == (ny == 83)
    _, ref = O.run(p.cfg, O.refine(p.cfg, p.U, p.V, p.W), p.T0, 5)
    assert np.abs(_run(mr, p, mr.MR_F32, 5) - ref).max() <= 1e-5


@pytest.mark.parametrize("n", [(32, 16, 8), (64, 32, 8), (256, 256, 4)])
def test_coupled_steps_over_plate_sizes(mr, n):
    p = Problem(*n, gamma=1.2, dt=2e-4, ra=1e7)
    h = mr.mr_create(p.mr_config(mr, mr.MR_F32, mr.MR_VEL_FUSED))
    nu = torch.zeros(2, dtype=torch.float64, device="cuda")
    Tc = torch.zeros((n[2], n[1], n[0]), dtype=torch.float64, device="cuda")
    mr.mr_set_scalar(h, dev(p.T0))
    for _ in range(3):
        mr.mr_refine_velocity(h, dev(p.U), dev(p.V), dev(p.W))
        mr.mr_scalar_step_coupled(h, nu, Tc)
    st = mr.mr_scalar_stats(h)
    for k, name in enumerate(("nu_bot", "nu_top")):
        assert abs(float(nu[k]) - st[name]) <= 1e-12 * abs(st[name])
    h.close()
