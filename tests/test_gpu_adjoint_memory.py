"""An adjoint run that is refused memory, wherever it runs out, leaves what the library
holds and an earlier run's gradients as they were."""
import numpy as np
import pytest

from tests.gpu_common import Problem

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def test_refusals_change_nothing():
    import paper_1805_03426_gb300.mr as mr
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    p = Problem(nx=8, ny=8, nz=6, gamma=1.5)
    h = mr.mr_create(p.mr_config(mr, mr.MR_F64))
    mr.mr_refine_velocity(h, dev(p.U), dev(p.V), dev(p.W))
    T0 = dev(p.T0)

    def forward(S, ck):
        mr.mr_set_scalar(h, T0)
        return mr.mr_adjoint_forward(h, S, ck, np.ones(S + 1), np.ones(S + 1))

    live0 = mr.mr_debug_alloc_cap(-2)
    try:
        # a first run of nine levels, refused at every size up to what it needs
        forward(8, 5)
        need = mr.mr_debug_alloc_cap(-2) - live0
        h.close()
        h = mr.mr_create(p.mr_config(mr, mr.MR_F64))
        mr.mr_refine_velocity(h, dev(p.U), dev(p.V), dev(p.W))
        live0 = mr.mr_debug_alloc_cap(-2)
        for room in (0, 100, 400, need // 2, need - 1):
            mr.mr_debug_alloc_cap(live0 + room)
            with pytest.raises(mr.MRError) as e:
                forward(8, 5)
            assert e.value.code == mr.MR_ERR_OOM and mr.mr_debug_alloc_cap(-2) == live0
        mr.mr_debug_alloc_cap(live0 + need)
        forward(8, 5)
        # the same store holds a run of ten steps, whose results need a little more
        live1 = mr.mr_debug_alloc_cap(-2)
        mr.mr_debug_alloc_cap(live1)
        with pytest.raises(mr.MRError) as e:
            forward(10, 5)
        assert e.value.code == mr.MR_ERR_OOM and mr.mr_debug_alloc_cap(-2) == live1
        mr.mr_debug_alloc_cap(-1)
        assert np.isfinite(forward(10, 5))
        torch.cuda.synchronize()
        h.close()
    finally:
        mr.mr_debug_alloc_cap(-1)
