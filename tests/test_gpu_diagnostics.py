"""Statistics, profiles and the upscaled scalar against plain FP64 sums of the same
values: FP32 scalars (whose sums are pairs of FP32 values) and FP64 ones, large and
tiny values, a large mean with a small spread, values that are not finite, sizes
that leave remainders in every block."""
import numpy as np
import pytest

from paper_1805_03426_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = {
    "walls_odd": dict(nx=11, ny=7, nz=5, mx=3, my=5, mz=2, walls=1, gamma=1.3),
    "periodic": dict(nx=16, ny=24, nz=9, mx=4, my=2, mz=3, walls=0, gamma=0.0),
    "wide": dict(nx=150, ny=130, nz=3, mx=2, my=2, mz=2, walls=0, gamma=1.0),
}
# mean, spread of the scalar
VALUES = {"ordinary": (0.0, 0.3), "large": (0.0, 1e15), "tiny": (0.0, 1e-18), "offset": (1000.0, 1e-2)}


def _case(size, f64, order=2, adiabatic=0):
    import paper_1805_03426_gb300.mr as mr
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    d = dict(SIZES[size])
    walls = d.pop("walls")
    gamma = d.pop("gamma")
    h = mr.mr_create(mr.mr_config_default(
        stretch_gamma=gamma, ra=1e5, pr_or_sc=1.0, precision=mr.MR_F64 if f64 else mr.MR_F32, face_order=order,
        bc_horizontal=mr.MR_WALLS if walls else mr.MR_PERIODIC,
        bc_plates=mr.MR_ADIABATIC if adiabatic else mr.MR_DIRICHLET, **d))
    (Nx, Ny, Nz), zf = mr.mr_grid(h)
    Xf, Yf = np.linspace(0, 1, d["nx"] + 1), np.linspace(0, 1, d["ny"] + 1)
    vel = synth.coarse_velocity(7, Xf, Yf, zf[:: d["mz"]], rms=0.2, walls=bool(walls), kmax=4)
    dtype = torch.float64 if f64 else torch.float32
    dense = [torch.empty(h.shapes[k], dtype=dtype, device="cuda") for k in ("Us", "Vs", "Ws")]
    mr.mr_refine_velocity(h, *[torch.from_numpy(v).cuda() for v in vel], *dense)
    return mr, h, d, zf, walls, dense[2].double().cpu().numpy()


@pytest.mark.parametrize("values", sorted(VALUES))
@pytest.mark.parametrize("size", sorted(SIZES))
@pytest.mark.parametrize("f64", [True, False])
def test_statistics_and_upscaled_scalar(size, values, f64):
    mr, h, d, zf, walls, W = _case(size, f64)
    dz = np.diff(zf)
    mean, spread = VALUES[values]
    T = mean + spread * np.random.default_rng(3).standard_normal(h.shapes["T"])
    T = T if f64 else T.astype(np.float32)
    mr.mr_set_scalar(h, torch.from_numpy(np.ascontiguousarray(T)).cuda())
    T = T.astype(np.longdouble)
    w = (dz[:, None, None] * np.ones(T.shape) / (T.shape[1] * T.shape[2])).astype(np.longdouble)
    st = mr.mr_scalar_stats(h)
    m = (T * w).sum()
    var = ((T - m) ** 2 * w).sum()
    size_T = np.abs(T).max()
    # sums of n terms in FP64 (and FP32 pairs of 48 bits): 1e-13 of the terms' size; the
    # variance relative to itself however large the mean is
    assert abs(st["mean"] - float(m)) <= 1e-13 * size_T
    assert abs(st["integral"] - float(m)) <= 1e-13 * size_T
    assert abs(st["var"] - float(var)) <= 1e-11 * float(var)
    Tc = mr.mr_upscale_scalar(h)
    c = (T * dz[:, None, None]).reshape(d["nz"], d["mz"], d["ny"], d["my"], d["nx"], d["mx"]).sum((1, 3, 5))
    c = c / (dz.reshape(d["nz"], d["mz"]).sum(1)[:, None, None] * d["my"] * d["mx"])
    # the layers of a coarse cell are summed in the handle's precision
    assert np.abs(Tc - c.astype(float)).max() <= (1e-14 if f64 else 1e-5) * float(size_T)
    h.close()


@pytest.mark.parametrize("values", ["ordinary", "large", "tiny"])
@pytest.mark.parametrize("size", sorted(SIZES))
@pytest.mark.parametrize("f64,order,adiabatic", [(True, 2, 0), (False, 2, 0), (True, 4, 1), (False, 4, 1)])
def test_profiles(size, values, f64, order, adiabatic):
    import oracle as O

    mr, h, d, zf, walls, W = _case(size, f64, order, adiabatic)
    T = VALUES[values][1] * np.random.default_rng(4).standard_normal(h.shapes["T"])
    T = (T if f64 else T.astype(np.float32).astype(np.float64))
    mr.mr_set_scalar(h, torch.from_numpy(T).cuda())
    nu_z, nu_T = mr.mr_scalar_profiles(h)
    h.close()
    cfg = O.Config(gamma=SIZES[size]["gamma"], kappa=1e5 ** -0.5, face_order=order, walls_xy=walls,
                   plates_dirichlet=0 if adiabatic else 1, **d)
    rz, _ = O.nusselt_profile(cfg, T, W)
    # the oracle adds the 78,000 equal terms of a plate one after the other in FP64,
    # which is 2e-12 off by itself, so the squares are added here in extended precision
    t = T.astype(np.longdouble)
    Nz, Ny, Nx = T.shape
    dx, dy, dz, zc = 1 / Nx, 1 / Ny, np.diff(zf)[:, None, None], 0.5 * (zf[1:] + zf[:-1])
    gx, gy = (np.diff(t, axis=a) if walls else t - np.roll(t, 1, a) for a in (2, 1))
    rT = (gx ** 2 * dz).sum() * dy / dx + (gy ** 2 * dz).sum() * dx / dy
    rT += (np.diff(t, axis=0) ** 2 / np.diff(zc)[:, None, None]).sum() * dx * dy
    if not adiabatic:
        half = np.longdouble(0.5)
        rT += dx * dy * (((t[0] - half) ** 2).sum() / (zc[0] - zf[0]) + ((t[-1] + half) ** 2).sum() / (zf[-1] - zc[-1]))
    rT = float(rT)
    # FP64 sums of the same values on both sides: the repository's 1e-12, of the
    # largest flux (whose terms cancel on most faces)
    scale = np.abs(T).max() / np.diff(zf).min()
    assert np.abs(nu_z - rz).max() <= 1e-12 * max(scale, np.abs(rz).max())
    assert abs(nu_T - rT) <= 1e-12 * abs(rT)


def test_fused_profile_forms_the_same_vertical_velocity():
    import paper_1805_03426_gb300.mr as mr
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    for m, mode in ((2, mr.MR_VEL_FUSED), (4, mr.MR_VEL_FUSED), (4, mr.MR_VEL_XFUSED)):
        n = (64 // m, 48 // m, 7)
        out = []
        for md in (mr.MR_VEL_STORED, mode):
            h = mr.mr_create(mr.mr_config_default(nx=n[0], ny=n[1], nz=n[2], mx=m, my=m, mz=m, stretch_gamma=1.5, ra=1e6,
                                                  precision=mr.MR_F32, velocity_mode=md))
            _, zf = mr.mr_grid(h)
            vel = synth.coarse_velocity(9, np.linspace(0, 1, n[0] + 1), np.linspace(0, 1, n[1] + 1), zf[::m], kmax=3)
            mr.mr_refine_velocity(h, *[torch.from_numpy(v).cuda() for v in vel])
            zc = 0.5 * (zf[1:] + zf[:-1])
            mr.mr_set_scalar(h, torch.from_numpy(synth.initial_scalar(1, zc, 48, 64)).cuda())
            out.append(mr.mr_scalar_profiles(h))
            h.close()
        # the same W in FP32, rounded along another way: FP32 accuracy of the flux
        assert np.abs(out[0][0] - out[1][0]).max() <= 1e-5 * np.abs(out[0][0]).max()
        assert abs(out[0][1] - out[1][1]) <= 1e-12 * abs(out[0][1])


def test_values_that_are_not_finite():
    mr, h, d, zf, walls, W = _case("periodic", False)
    T = np.random.default_rng(5).standard_normal(h.shapes["T"]).astype(np.float32)
    T[3, 5, 7], T[20, 0, 0] = np.nan, np.inf
    mr.mr_set_scalar(h, torch.from_numpy(T).cuda())
    st = mr.mr_scalar_stats(h, allow_nonfinite=True)
    assert st.get("nonfinite") and np.isnan(st["var"])
    w = np.diff(zf)[:, None, None] / (T.shape[1] * T.shape[2]) * np.ones(T.shape)
    fine = np.isfinite(T)
    assert abs(st["mean"] - float((T[fine].astype(float) * w[fine]).sum())) <= 1e-13
    nu_z, nu_T = mr.mr_scalar_profiles(h)
    assert not np.isfinite(nu_T) and not np.isfinite(nu_z[3]) and not np.isfinite(nu_z[20])
    assert np.isfinite(nu_z[[0, 1, 2, 5, 19, 22]]).all()
    h.close()
