"""The plate Nusselt numbers of a fused coupled step for plates of one tile, a few
tiles and more cells than one round of its blocks takes (311,296), twice in a row
(the block count is reset), against sums of the same values in extended precision."""
import numpy as np
import pytest

from tests.gpu_common import Problem
from tests.test_gpu_coupled import dev, mr  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nz", [(16, 4, 4), (48, 12, 3), (160, 128, 3)])
def test_plate_nusselt_numbers_of_a_coupled_step(mr, nx, ny, nz):  # noqa: F811
    p = Problem(nx, ny, nz, 4, 4, 4, gamma=1.2, dt=1e-4)
    h = mr.mr_create(p.mr_config(mr, mr.MR_F32, mr.MR_VEL_FUSED))
    mr.mr_refine_velocity(h, dev(p.U), dev(p.V), dev(p.W))
    mr.mr_set_scalar(h, dev(p.T0))
    nu = torch.zeros(2, dtype=torch.float64, device="cuda")
    Tc = torch.zeros((nz, ny, nx), dtype=torch.float64, device="cuda")
    T = torch.empty(p.T0.shape, dtype=torch.float32, device="cuda")
    zf, zc = p.grid["zf"], p.grid["zc"]
    for _ in range(2):
        mr.mr_scalar_step_coupled(h, nu, Tc)
        mr.mr_get_scalar(h, T)
        t = T.cpu().numpy().astype(np.longdouble)
        ref = np.array([(0.5 - t[0]).mean() / (zc[0] - zf[0]), (t[-1] + 0.5).mean() / (zf[-1] - zc[-1])], dtype=np.float64)
        # FP64 sums in a tree of about 30 additions, of terms of one sign: 1e-13
        assert np.abs(nu.cpu().numpy() / ref - 1).max() <= 1e-13
    h.close()
