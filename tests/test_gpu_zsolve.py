"""Implicit vertical diffusion against the oracle over column heights: two and
three layers, odd and even halves, batches of eight layers and their remainders,
columns kept in shared memory and not (448 and 896 layers), the two sizes of the
coefficient table (256, 1280 layers) and columns beyond it; planes that are no
multiple of the 16 columns a warp takes."""
import numpy as np
import pytest

import oracle as O
from tests.gpu_common import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

HEIGHTS = [(2, 1), (3, 1), (15, 1), (16, 1), (17, 1), (33, 1), (64, 4), (64, 7), (300, 3), (431, 3)]


@pytest.mark.parametrize("nz,mz", HEIGHTS)
@pytest.mark.parametrize("f64", [True, False])
def test_implicit_steps_match_the_oracle(nz, mz, f64):
    import paper_1805_03426_gb300.mr as mr
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    # a diffusion number of 10 and more per step on the finer columns
    p = Problem(nx=5, ny=3, nz=nz, mx=1, my=1, mz=mz, implicit=1, ra=1e4, pr=1.0, dt=2e-3, np_average=3)
    h = mr.mr_create(p.mr_config(mr, mr.MR_F64 if f64 else mr.MR_F32))
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    mr.mr_refine_velocity(h, dev(p.U), dev(p.V), dev(p.W))
    mr.mr_set_scalar(h, dev(p.T0))
    mr.mr_scalar_step(h, 5)
    T = torch.empty(p.T0.shape, dtype=torch.float64, device="cuda")
    mr.mr_get_scalar(h, T)
    h.close()
    _, ref = O.run(p.cfg, O.refine(p.cfg, p.U, p.V, p.W), p.T0, 5)
    # the repository's bars: 1e-12 of the largest value in FP64, 1e-5 in FP32
    assert np.abs(T.cpu().numpy() - ref).max() <= (1e-12 if f64 else 1e-5) * np.abs(ref).max()
