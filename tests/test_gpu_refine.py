"""The dense refinement against the oracle at the edges of its tiles (32 coarse
columns x 8 dense rows, chunks of layers, groups of coarse slabs), with and without
walls, every kind of refinement factor, and the second copy of the faces that a
caller takes."""
import numpy as np
import pytest

import oracle as O
from tests.gpu_common import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PROBS = {
    "periodic_m2_33": dict(nx=33, ny=5, nz=6, mx=2, my=2, mz=2, gamma=1.5),
    "periodic_m2_32": dict(nx=32, ny=8, nz=3, mx=2, my=2, mz=4, lx=2.0),
    "walls_m2_31": dict(nx=31, ny=7, nz=9, mx=2, my=2, mz=2, walls=1, gamma=1.2),
    "walls_m4_64": dict(nx=64, ny=4, nz=4, mx=4, my=4, mz=4, walls=1),
    "ragged_8_1_3": dict(nx=35, ny=17, nz=5, mx=8, my=1, mz=3, gamma=1.5),
    "ragged_1_5_1": dict(nx=65, ny=3, nz=17, mx=1, my=5, mz=1, walls=1),
    "several_groups": dict(nx=160, ny=160, nz=128, mx=2, my=2, mz=2, gamma=1.5),
}


@pytest.mark.parametrize("name", sorted(PROBS))
@pytest.mark.parametrize("f64", [True, False])
def test_dense_faces_match_the_oracle(name, f64):
    import paper_1805_03426_gb300.mr as mr
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    p = Problem(**PROBS[name])
    ref = O.refine(p.cfg, p.U, p.V, p.W)
    h = mr.mr_create(p.mr_config(mr, mr.MR_F64 if f64 else mr.MR_F32))
    dtype = torch.float64 if f64 else torch.float32
    vel = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (p.U, p.V, p.W)]
    out = [torch.full(h.shapes[k], float("nan"), dtype=dtype, device="cuda") for k in ("Us", "Vs", "Ws")]
    mr.mr_refine_velocity(h, *vel, *out)
    # the repository's bars: each component 1e-12 of its largest value in FP64, 1e-5 in FP32
    for got, want in zip(out, ref):
        assert np.abs(got.cpu().numpy() - want).max() <= (1e-12 if f64 else 1e-5) * np.abs(want).max()
    # what the handle keeps is what it gave out: to host memory from its own copy
    host = [np.empty(h.shapes[k], dtype=np.float64 if f64 else np.float32) for k in ("Us", "Vs", "Ws")]
    mr.mr_refine_velocity(h, *vel, *host)
    torch.cuda.synchronize()
    for got, kept in zip(out, host):
        assert np.array_equal(got.cpu().numpy(), kept)
    h.close()
