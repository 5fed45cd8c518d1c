"""The variance of scalars whose outliers lie where a block of the reduction begins,
against extended-precision sums: as accurate as about the mean, wherever they lie."""
import numpy as np
import pytest

from tests import test_gpu_diagnostics as diagnostics

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


# 1700 layers of a unit each: more units than blocks
diagnostics.SIZES.setdefault("tall", dict(nx=10, ny=4, nz=425, mx=3, my=1, mz=4, walls=0, gamma=1.1))


def _fill(T, where, rng):
    Nz, Ny, Nx = T.shape
    flat = T.reshape(Nz, -1)
    n = flat.shape[1]
    per = -(-n // -(-n // 16384))                # cells of a block's share of a plane
    if where == "first cells":
        flat[:, ::per] = 1e3
    elif where == "one column":
        T[:, 0, 0] = -1e3
    elif where == "eighths":
        for q in range(0, n, per):
            flat[:, q:q + per // 8] += 1e3
    elif where == "one layer":
        T[0] += 1e3
    elif where == "alternate layers":            # among them a block's units, 1216 apart
        T[(np.arange(Nz) // 1216) % 2 == 1] += 1e3
    return T


@pytest.mark.parametrize("where", ["first cells", "one column", "eighths", "one layer", "alternate layers"])
@pytest.mark.parametrize("size", ["wide", "walls_odd", "tall"])
@pytest.mark.parametrize("f64", [True, False])
def test_outliers_cost_no_precision(size, where, f64):
    mr, h, d, zf, walls, W = diagnostics._case(size, f64)
    rng = np.random.default_rng(11)
    T = _fill(1e-3 * rng.standard_normal(h.shapes["T"]), where, rng)
    T = T if f64 else T.astype(np.float32)
    mr.mr_set_scalar(h, torch.from_numpy(np.ascontiguousarray(T)).cuda())
    st = mr.mr_scalar_stats(h)
    h.close()
    t = T.astype(np.longdouble)
    w = (np.diff(zf)[:, None, None] * np.ones(T.shape) / (T.shape[1] * T.shape[2])).astype(np.longdouble)
    m = (t * w).sum()
    var = ((t - m) ** 2 * w).sum()
    # squares to 2^-52 (FP32 pairs: 2^-47) of themselves, a chain of at most 100 additions,
    # and the eightfold that the squares about a block's reference may be
    assert abs(st["var"] - float(var)) <= (8 * 100 * 2.0 ** -53 if f64 else 8 * 100 * 2.0 ** -48) * float(var)
    assert abs(st["mean"] - float(m)) <= 1e-13 * np.abs(T).max()
