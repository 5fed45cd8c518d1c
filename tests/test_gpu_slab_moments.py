"""Volume moments of y-slab handles: each slab's against extended-precision sums of its
rows, and the slabs' combined ones against the whole domain's."""
import numpy as np
import pytest

from paper_1805_03426_gb300 import slabs
from tests.gpu_common import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_slab_moments():
    import paper_1805_03426_gb300.mr as mr
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    p = Problem(nx=32, ny=24, nz=7, mx=4, my=4, mz=4, gamma=1.5)
    T = np.ascontiguousarray(p.T0.astype(np.float32))
    w = np.diff(p.grid["zf"])[:, None, None].astype(np.longdouble)

    def stats(j0, rows):
        cfg = p.mr_config(mr, mr.MR_F32, mr.MR_VEL_FUSED)
        if rows:
            cfg.slab_j0, cfg.slab_ny = j0, rows
        h = mr.mr_create(cfg)
        part = T[:, 4 * j0:4 * (j0 + rows)] if rows else T
        mr.mr_set_scalar(h, torch.from_numpy(np.ascontiguousarray(part)).cuda())
        st = mr.mr_scalar_stats(h)
        _, zf = mr.mr_grid(h)
        vol, area = slabs.slab_geometry(h.cfg, zf)
        h.close()
        t = part.astype(np.longdouble)
        mean = (t * w).mean((1, 2)).sum()
        var = ((t - mean) ** 2 * w).mean((1, 2)).sum()
        # pairs of FP32 values, 2^-47 a term: 1e-13 of the largest value, 1e-12 of the variance
        assert abs(st["mean"] - float(mean)) <= 1e-13 * np.abs(T).max()
        assert abs(st["integral"] - float(mean) * vol) <= 1e-13 * np.abs(T).max() * vol
        assert abs(st["var"] - float(var)) <= 1e-12 * float(var)
        return slabs.slab_stats(st, vol, area), st

    _, whole = stats(0, 0)
    comb = slabs.combine_stats([stats(j0, rows)[0] for j0, rows in ((0, 4), (4, 12), (16, 8))])
    assert abs(comb["mean"] - whole["mean"]) <= 2e-13 * np.abs(T).max()
    assert abs(comb["integral"] - whole["integral"]) <= 2e-13 * np.abs(T).max()
    assert abs(comb["var"] - whole["var"]) <= 3e-12 * whole["var"]
