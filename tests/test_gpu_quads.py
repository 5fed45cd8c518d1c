"""The FP32 stored step and its adjoint on rows of whole quads (Nx a multiple of
four) against the same kernels with a cell per thread: a problem that repeats after
half its length in x, stepped at its full length, has to give twice what it gives at
half of it, whose rows are no whole quads, to the last bit.  One, two and four layers
per thread with remainders of layers; blocks with idle threads; the scalar against
the oracle as well."""
import numpy as np
import pytest

import oracle as O
from tests.gpu_common import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# half problems: cells in x are 2 mod 4, refinement 1 in x (no R_x, whose rows at the
# periodic seam depend on the length of the domain in their last bits)
PROBS = {
    "6x10x7": dict(nx=6, ny=5, nz=7, mx=1, my=2, mz=1),            # one layer per thread
    "34x60x79": dict(nx=34, ny=30, nz=79, mx=1, my=2, mz=1),       # two
    "66x64x75": dict(nx=66, ny=32, nz=25, mx=1, my=2, mz=3),       # four
}
S = 4                                                       # Euler, leapfrog and averaging steps


def _gradient(mr, p, vel, T0, wnu, **size):
    cfg = p.mr_config(mr, mr.MR_F32)
    for k, v in size.items():
        setattr(cfg, k, v)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    h = mr.mr_create(cfg)
    mr.mr_refine_velocity(h, *[dev(v) for v in vel])
    mr.mr_set_scalar(h, dev(T0))
    mr.mr_adjoint_forward(h, S, 2, wnu)
    T = torch.empty(T0.shape, dtype=torch.float64, device="cuda")
    mr.mr_get_scalar(h, T)
    g = [torch.empty(h.shapes[k], dtype=torch.float64, device="cuda") for k in ("T", "U", "V", "W")]
    mr.mr_adjoint_backward(h, 1.0, *g)
    h.close()
    return T.cpu().numpy(), [x.cpu().numpy() for x in g]


@pytest.mark.parametrize("name", sorted(PROBS))
@pytest.mark.parametrize("adiabatic", [0, 1])
def test_quads_give_the_same_bits_as_single_cells(name, adiabatic):
    import paper_1805_03426_gb300.mr as mr
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    p = Problem(gamma=1.3, dt=3e-4, np_average=3, adiabatic=adiabatic, lx=0.5, **PROBS[name])
    wnu = np.array([0.0, 0.5, 0.0, 0.0, 1.0])
    half = _gradient(mr, p, (p.U, p.V, p.W), p.T0, wnu)
    twice = lambda a: np.concatenate([a, a], axis=2)
    # the Nusselt number averages over twice the cells: twice the weight
    full = _gradient(mr, p, [twice(v) for v in (p.U, p.V, p.W)], twice(p.T0), 2 * wnu, nx=2 * p.cfg.nx, lx=1.0)
    assert np.array_equal(full[0], twice(half[0]))
    assert np.array_equal(full[1][0], twice(half[1][0]))
    # the coarse gradients are FP64 sums of the same FP32 face gradients, in any order
    for a, b in zip(full[1][1:], half[1][1:]):
        assert np.abs(a - twice(b)).max() <= 1e-12 * np.abs(b).max()
    # the scalar against the oracle, to the repository's FP32 bar
    _, ref = O.run(p.cfg, O.refine(p.cfg, p.U, p.V, p.W), p.T0, S)
    assert np.abs(half[0] - ref).max() <= 1e-5 * np.abs(ref).max()
