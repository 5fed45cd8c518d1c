"""mr_create allocates what mr_refine_velocity needs: the refinement takes no memory of
its own (so it can be captured from the first call on), and a handle whose refinement
work does not fit whole is created with a smaller one and refines to the same faces."""
import numpy as np
import pytest

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


def dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _modes(mr):
    return {"f64": (mr.MR_F64, mr.MR_VEL_STORED), "f32": (mr.MR_F32, mr.MR_VEL_STORED),
            "xfused": (mr.MR_F32, mr.MR_VEL_XFUSED), "fused": (mr.MR_F32, mr.MR_VEL_FUSED)}


@pytest.mark.parametrize("mode", ["f64", "f32", "xfused", "fused"])
def test_refinement_allocates_nothing(mr, mode):
    p = Problem(nx=16, ny=8, nz=7, mx=4, my=4, mz=4, gamma=1.5)
    h = mr.mr_create(p.mr_config(mr, *_modes(mr)[mode]))
    live = mr.mr_debug_alloc_cap(-2)
    mr.mr_refine_velocity(h, dev(p.U), dev(p.V), dev(p.W))
    torch.cuda.synchronize()
    assert mr.mr_debug_alloc_cap(-2) == live
    h.close()


@pytest.mark.parametrize("mode", ["f64", "f32"])
def test_the_first_refinement_can_be_captured(mr, mode):
    p = Problem(nx=16, ny=8, nz=7, mx=4, my=4, mz=4, gamma=1.5)
    vel = [dev(a) for a in (p.U, p.V, p.W)]
    out = []
    for captured in (False, True):
        h = mr.mr_create(p.mr_config(mr, *_modes(mr)[mode]))
        dtype = torch.float64 if mode == "f64" else torch.float32
        dense = [torch.zeros(h.shapes[k], dtype=dtype, device="cuda") for k in ("Us", "Vs", "Ws")]
        torch.cuda.synchronize()
        if captured:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g):
                mr.mr_refine_velocity(h, *vel, *dense)
            assert not any(d.any() for d in dense)
            g.replay()
        else:
            mr.mr_refine_velocity(h, *vel, *dense)
        torch.cuda.synchronize()
        out.append([d.cpu().numpy() for d in dense])
        h.close()
    for a, b in zip(*out):
        assert np.array_equal(a, b) and a.any()


@pytest.mark.parametrize("walls", [0, 1])
def test_a_smaller_work_refines_to_the_same_faces(mr, walls):
    p = Problem(nx=11, ny=9, nz=13, mx=2, my=3, mz=4, gamma=1.5, walls=walls)

    def faces(h):
        d = [torch.empty(h.shapes[k], dtype=torch.float64, device="cuda") for k in ("Us", "Vs", "Ws")]
        mr.mr_refine_velocity(h, dev(p.U), dev(p.V), dev(p.W), *d)
        torch.cuda.synchronize()
        return [a.cpu().numpy() for a in d]

    live0 = mr.mr_debug_alloc_cap(-2)
    h = mr.mr_create(p.mr_config(mr, mr.MR_F64))
    whole = mr.mr_debug_alloc_cap(-2)
    ref = faces(h)
    h.close()
    # the intermediates of one coarse slab (four layers), of the whole column (52)
    w = walls
    values = lambda L: L * (9 * (11 + w) + (9 + w) * 11 + 27 * (11 + w) + (27 + w) * 11) + (L + 1) * (9 * 11 + 27 * 11)  # noqa: E731
    try:
        for part in (0.6, 0.3, 0.0):
            room = int(8 * (values(52) * part if part else values(4) + 6 * 32))
            cap = whole - 8 * values(52) + room
            mr.mr_debug_alloc_cap(cap)
            h = mr.mr_create(p.mr_config(mr, mr.MR_F64))
            assert mr.mr_debug_alloc_cap(-2) <= cap < whole
            mr.mr_debug_alloc_cap(mr.mr_debug_alloc_cap(-2))      # nothing more
            for a, b in zip(faces(h), ref):
                assert np.array_equal(a, b)
            h.close()
            mr.mr_debug_alloc_cap(-1)
        # less than one slab's: refused, and everything is returned
        mr.mr_debug_alloc_cap(whole - 8 * values(52) + 8 * values(4) // 2)
        with pytest.raises(mr.MRError) as e:
            mr.mr_create(p.mr_config(mr, mr.MR_F64))
        assert e.value.code == mr.MR_ERR_OOM and mr.mr_debug_alloc_cap(-2) == live0
    finally:
        mr.mr_debug_alloc_cap(-1)
