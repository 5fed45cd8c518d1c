"""Performance cases: the calls a solver makes of this library, over the range of grids it makes them on.

A case names one kind of call and a problem.  ``prepare`` makes what a solver holds before the call
(coarse face velocities, the initial scalar, a handle); ``run`` makes the call; ``exact`` computes the
same outputs in FP64 with plain torch and numpy, without the library.

Kinds
  steps     set the scalar, advance it by a number of time steps, read both levels and the plate Nusselt numbers
  coupled   a coupled run: every step the coarse solver hands over new face velocities, the scalar takes one
            step, and the coarse solver gets the upscaled scalar and the plate Nusselt numbers back
  temporal  coarse steps with temporal refinement, several scalar steps in each
  refine    a new coarse velocity refined onto the dense faces, which are read
  diagnose  what a run writes out between its steps: time-step limit, statistics, Nusselt profiles, coarse scalar
  adjoint   a loss of the run and its gradients with respect to the initial scalar and the coarse velocity

Outputs come in the precision of the handle: what an FP32 run gives out in FP64 (the coarse scalar, statistics,
coarse gradients) has been computed from FP32 values and is good to FP32.  The plate Nusselt numbers of an evolved FP32
scalar are differences of nearly equal values, whose rounding they carry many times over: the FP64 cases return them.
"""
import math

import numpy as np
import torch

PERIODIC = dict(walls=0, implicit=0, adiabatic=0, order=2)


def _case(kind, n, m, **kw):
    m = m if isinstance(m, tuple) else (m, m, m)
    d = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], mx=m[0], my=m[1], mz=m[2], gamma=1.5, ra=1e8, pr=7.0,
             precision="f32", mode="stored", lx=1.0, ly=1.0)
    d.update(PERIODIC)
    d.update(kw)
    return d


def listed():
    return [
        # a small box, 32^3 dense cells in FP64: development runs and parameter scans, where launches and latency count
        _case("steps", (16, 16, 16), 2, name="steps_f64_32", gamma=0.0, ra=1e6, precision="f64", steps=100),
        # the FP64 production grid, 256 x 256 x 192 dense cells
        _case("steps", (128, 128, 96), 2, name="steps_f64_256", precision="f64", steps=20),
        # the precision form: FP32, refinement 4, nothing of the refined velocity stored, 512 x 512 x 384 dense cells
        _case("steps", (128, 128, 96), 4, name="steps_fused_512", mode="fused", ra=1e9, pr=100.0, steps=50),
        # the large form of the same, 1024 x 1024 x 512 dense cells
        _case("steps", (256, 256, 128), 4, name="steps_fused_1024", mode="fused", ra=1e10, pr=100.0, steps=25),
        # a coupled run at refinement 2 on a grid that is no power of two (320 x 144 x 102 dense cells, box 2 : 1)
        _case("coupled", (160, 72, 51), 2, name="coupled_fused_m2", mode="fused", lx=2.0, ra=1e8, steps=10),
        # fourth-order face values in the split-x form, 256 x 192 x 128 dense cells
        _case("steps", (64, 48, 32), 4, name="steps_order4", mode="xfused", order=4, ra=1e9, pr=100.0, steps=25),
        # a box with side walls, ragged refinement 3 x 2 x 4 and implicit vertical diffusion, FP64 (123 x 74 x 148)
        _case("steps", (41, 37, 37), (3, 2, 4), name="steps_walls_implicit", precision="f64", walls=1, implicit=1, ra=1e7,
              steps=20),
        # the refined velocity on its own, FP64, 256 x 256 x 192 dense cells
        _case("refine", (128, 128, 96), 2, name="refine_f64_256", precision="f64"),
        # temporal refinement: 4 scalar steps per coarse step, 256 x 256 x 192 dense cells
        _case("temporal", (64, 64, 48), 4, name="temporal_fused", mode="fused", ra=1e9, pr=100.0, steps=5, mt=4),
        # output of a run: time-step limit, statistics, profiles, coarse scalar, 256 x 256 x 192 dense cells
        _case("diagnose", (64, 64, 48), 4, name="diagnose_f32", mode="fused", ra=1e9, pr=100.0),
        # the differentiation form, 128 x 128 x 96 dense cells, in both precisions
        _case("adjoint", (64, 64, 48), 2, name="adjoint_f64", precision="f64", ra=1e7, steps=40, every=10),
        _case("adjoint", (64, 64, 48), 2, name="adjoint_f32", ra=1e7, steps=40, every=10),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["f64", "f64", "fused", "fused", "coupled", "order4", "walls", "refine", "temporal", "diagnose",
                       "adjoint"])
    gamma = rng.choice([0.0, 1.0, 1.5])
    ra = 10.0 ** rng.uniform(6, 10)

    def box(cells, m, tile=(1, 1)):
        # coarse sizes of about that many dense cells; dense x and y multiples of the tile
        edge = cells ** (1.0 / 3.0)
        out = []
        for a in range(3):
            q = max(1, (tile[a] if a < 2 else 1) // m[a])
            n = int(round(edge * rng.uniform(0.6, 1.5) / m[a] / q)) * q
            out.append(max(n, q, 4 + (-4) % q))
        return tuple(out)

    if kind in ("f64", "refine", "adjoint", "walls"):
        m = tuple(rng.choice([1, 2, 2, 3, 4]) for _ in range(3))
        m = m if max(m) > 1 else (2, 2, 2)
        n = box(_log(rng, 2e4, 6e6 if kind in ("f64", "refine") else 1.2e6), m)
        precision = rng.choice(["f64", "f32"]) if kind != "f64" else "f64"
        if kind == "f64":
            return _case("steps", n, m, gamma=gamma, ra=ra, precision=precision, steps=rng.choice([10, 20]),
                         adiabatic=rng.choice([0, 1]))
        if kind == "refine":
            return _case("refine", n, m, gamma=gamma, ra=ra, precision=precision, walls=rng.choice([0, 1]))
        if kind == "adjoint":
            return _case("adjoint", n, m, gamma=gamma, ra=ra, precision=precision, steps=rng.choice([20, 30]),
                         every=rng.choice([5, 10]), walls=rng.choice([0, 0, 1]))
        return _case("steps", n, m, gamma=gamma, ra=ra, precision=precision, walls=rng.choice([0, 1]), steps=20,
                     implicit=rng.choice([0, 1]), order=rng.choice([2, 4]))
    m = rng.choice([2, 4])
    n = box(_log(rng, 2e5, 3e8 if kind == "fused" else 3e7), (m, m, m), (64, 16))
    if kind == "fused":
        return _case("steps", n, m, gamma=gamma, ra=ra, mode=rng.choice(["fused", "fused", "xfused"]), steps=20, lx=2.0)
    if kind == "order4":
        return _case("steps", n, m, gamma=gamma, ra=ra, mode="xfused", order=4, steps=20)
    if kind == "coupled":
        return _case("coupled", n, m, gamma=gamma, ra=ra, mode=rng.choice(["fused", "fused", "xfused"]), steps=8)
    if kind == "temporal":
        return _case("temporal", n, m, gamma=gamma, ra=ra, mode=rng.choice(["fused", "fused", "xfused"]), steps=4,
                     mt=rng.choice([2, 3, 4]))
    return _case("diagnose", n, m, gamma=gamma, ra=ra, mode=rng.choice(["fused", "xfused", "stored"]))


# ---------------------------------------------------------------- inputs


def _zfaces(case):
    N = case["nz"] * case["mz"]
    e = np.arange(N + 1) / N
    g = case["gamma"]
    z = 0.5 * (1.0 + np.tanh(g * (2.0 * e - 1.0)) / math.tanh(g)) if g > 0 else e
    z[0], z[-1] = 0.0, 1.0
    return z


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _velocity(case, rs, dev):
    """Coarse face velocities: the discrete curl of a random vector potential of 24 Fourier modes with a
    k^-17/6 amplitude (kinetic energy ~ k^-5/3), discretely divergence-free and zero on the walls; rms 0.1."""
    nx, ny, nz, w = case["nx"], case["ny"], case["nz"], case["walls"]
    lx, ly = case["lx"], case["ly"]
    f64 = dict(dtype=torch.float64, device=dev)
    xf, yf = torch.linspace(0, lx, nx + 1, **f64), torch.linspace(0, ly, ny + 1, **f64)
    zf = torch.tensor(_zfaces(case)[:: case["mz"]], **f64)
    mid = lambda f: 0.5 * (f[1:] + f[:-1])  # noqa: E731
    wall = lambda x, L: (x / L * (1 - x / L)) ** 2  # noqa: E731

    def field(z, y, x, vz, vy, vx):
        out = torch.zeros((len(z), len(y), len(x)), **f64)
        kmax = max(2, min(nx, ny) // 6)
        for _ in range(24):
            k = [int(v) for v in rs.randint(0, min(kmax, 8) + 1, 3)]
            a = rs.standard_normal() * max(0.5, math.sqrt((k[0] / 2) ** 2 + k[1] ** 2 + k[2] ** 2)) ** (-17.0 / 6.0)
            p = rs.uniform(0, 2 * math.pi, 3)
            bz = torch.cos(math.pi * k[0] * z + p[0]) * vz
            by = torch.cos(2 * math.pi * k[1] * y / ly + p[1]) * vy
            bx = torch.cos(2 * math.pi * k[2] * x / lx + p[2]) * vx
            out += a * bz[:, None, None] * by[None, :, None] * bx[None, None, :]
        return out

    gz, one = wall(zf, 1.0), 1.0
    gx, gy = (wall(xf, lx), wall(yf, ly)) if w else (one, one)
    DX, DY, DZ = lx / nx, ly / ny, (zf[1:] - zf[:-1])[:, None, None]
    # circulations of the edges (the first and last edge of a periodic axis are the same one)
    Gx = field(zf, yf, mid(xf), gz, gy, one) * DX
    Gy = field(zf, mid(yf), xf, gz, one, gx) * DY
    Gz = field(mid(zf), yf, xf, one, gy, gx) * DZ
    if not w:
        Gx[:, -1], Gy[:, :, -1] = Gx[:, 0], Gy[:, :, 0]
        Gz[:, -1] = Gz[:, 0]
        Gz[:, :, -1] = Gz[:, :, 0]
    U = (Gz[:, 1:] - Gz[:, :-1] - Gy[1:] + Gy[:-1]) / (DY * DZ)
    V = (Gx[1:] - Gx[:-1] - Gz[:, :, 1:] + Gz[:, :, :-1]) / (DX * DZ)
    W = (Gy[:, :, 1:] - Gy[:, :, :-1] - Gx[:, 1:] + Gx[:, :-1]) / (DX * DY)
    if not w:
        U, V = U[:, :, :-1], V[:, :-1]
    s = 0.1 / torch.sqrt((U ** 2).mean() + (V ** 2).mean() + (W ** 2).mean())
    return tuple((a * s).contiguous() for a in (U, V, W))


def _dt(case, U, V, W):
    """A time step of about CFL 0.3, from the coarse faces on the dense spacing."""
    dz = torch.tensor(np.diff(_zfaces(case)[:: case["mz"]]) / case["mz"], dtype=torch.float64, device=U.device)
    wz = torch.maximum(W[1:].abs(), W[:-1].abs()).amax((1, 2)) / dz
    rate = U.abs().amax() * case["nx"] * case["mx"] / case["lx"] + V.abs().amax() * case["ny"] * case["my"] / case["ly"] + wz.amax()
    kappa = (case["ra"] * case["pr"]) ** -0.5
    d = np.diff(_zfaces(case)).min() if not case["implicit"] else 1.0
    h = min(d, case["lx"] / (case["nx"] * case["mx"]), case["ly"] / (case["ny"] * case["my"]))
    return min(0.25 / float(rate), 0.03 * h * h / kappa)


def _dtype(case):
    return torch.float64 if case["precision"] == "f64" else torch.float32


def _inputs(case, seed):
    """The coarse velocities (one, or the two a coupled or temporally refined run alternates between), the
    initial scalar (conduction profile and noise, as the handle's precision holds it) and the time step."""
    dev = _device()
    rs = np.random.RandomState(seed % (1 << 31))
    vel = [_velocity(case, rs, dev) for _ in range(2 if case["kind"] in ("coupled", "temporal") else 1)]
    zf = _zfaces(case)
    zc = torch.tensor(0.5 * (zf[1:] + zf[:-1]), device=dev)
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed + 1)
    dtype = _dtype(case)
    if case["kind"] == "adjoint":  # the parameters of an FP32 problem are FP32 values
        vel = [tuple(a.to(dtype).double() for a in v) for v in vel]
    Nx, Ny = case["nx"] * case["mx"], case["ny"] * case["my"]
    T0 = torch.randn((len(zc), Ny, Nx), generator=gen, device=dev, dtype=dtype)
    T0.mul_(1e-2).add_((0.5 - zc).to(dtype)[:, None, None])
    return vel, T0, min(_dt(case, *v) for v in vel)


def _loss_weights(case):
    """Bottom Nusselt number averaged over the last quarter, and the final variance."""
    S = case["steps"]
    wnu, wvar = np.zeros(S + 1), np.zeros(S + 1)
    wnu[-max(1, S // 4):] = 1.0 / max(1, S // 4)
    wvar[-1] = 1.0
    return wnu, wvar


# ---------------------------------------------------------------- the library's calls


def prepare(case, seed):
    import paper_1805_03426_gb300.mr as mr

    vel, T0, dt = _inputs(case, seed)
    h = mr.mr_create(mr.mr_config_default(
        nx=case["nx"], ny=case["ny"], nz=case["nz"], mx=case["mx"], my=case["my"], mz=case["mz"],
        lx=case["lx"], ly=case["ly"], stretch_gamma=case["gamma"], ra=case["ra"], pr_or_sc=case["pr"], dt=dt,
        precision=mr.MR_F64 if case["precision"] == "f64" else mr.MR_F32,
        velocity_mode={"stored": mr.MR_VEL_STORED, "fused": mr.MR_VEL_FUSED, "xfused": mr.MR_VEL_XFUSED}[case["mode"]],
        bc_plates=mr.MR_ADIABATIC if case["adiabatic"] else mr.MR_DIRICHLET,
        bc_horizontal=mr.MR_WALLS if case["walls"] else mr.MR_PERIODIC, diffz_implicit=case["implicit"],
        face_order=case["order"]))
    s = dict(case=case, mr=mr, h=h, vel=vel, T0=T0)
    f64 = dict(dtype=torch.float64, device=T0.device)
    kind = case["kind"]
    if kind == "adjoint":
        s["w"], s["par"] = _loss_weights(case), [v.to(T0.dtype) for v in vel[0]]
        return s
    mr.mr_refine_velocity(h, *vel[0])
    if kind in ("steps", "coupled", "temporal"):
        s["T"], s["Tprev"] = torch.empty_like(T0), torch.empty_like(T0)
        s["nu"] = torch.zeros((case["steps"] if kind == "coupled" else 1, 2), **f64)
    if kind == "coupled":
        s["Tc"] = torch.zeros((case["steps"], case["nz"], case["ny"], case["nx"]), **f64)
    if kind == "refine":
        s["dense"] = [torch.empty(h.shapes[k], dtype=T0.dtype, device=T0.device) for k in ("Us", "Vs", "Ws")]
    if kind == "diagnose":
        mr.mr_set_scalar(h, T0)
        s["Tc"] = torch.zeros((case["nz"], case["ny"], case["nx"]), **f64)
    return s


def _with_nu(s, out):
    return {**out, "nu": s["nu"]} if s["case"]["precision"] == "f64" else out


def run(s):
    case, mr, h, vel = s["case"], s["mr"], s["h"], s["vel"]
    kind = case["kind"]
    if kind == "steps":
        mr.mr_set_scalar(h, s["T0"])
        mr.mr_scalar_step(h, case["steps"])
        mr.mr_plate_nu(h, s["nu"])
        mr.mr_get_scalar(h, s["T"], s["Tprev"])
        return _with_nu(s, {"T": s["T"], "Tprev": s["Tprev"]})
    if kind == "coupled":
        mr.mr_set_scalar(h, s["T0"])
        for i in range(case["steps"]):
            mr.mr_refine_velocity(h, *vel[i % 2])
            mr.mr_scalar_step_coupled(h, s["nu"][i], s["Tc"][i])
        mr.mr_get_scalar(h, s["T"], s["Tprev"])
        return _with_nu(s, {"T": s["T"], "Tprev": s["Tprev"], "Tc": s["Tc"].to(s["T"].dtype)})
    if kind == "temporal":
        mr.mr_refine_velocity(h, *vel[0])
        mr.mr_set_scalar(h, s["T0"])
        for i in range(case["steps"]):
            mr.mr_scalar_coarse_step(h, *vel[(i + 1) % 2], case["mt"])
        mr.mr_plate_nu(h, s["nu"])
        mr.mr_get_scalar(h, s["T"], s["Tprev"])
        return _with_nu(s, {"T": s["T"], "Tprev": s["Tprev"]})
    if kind == "refine":
        mr.mr_refine_velocity(h, *vel[0], *s["dense"])
        return s["dense"]
    if kind == "diagnose":
        mr.mr_refine_velocity(h, *vel[0])
        dt = mr.mr_cfl_dt(h, 0.3)
        stats = mr.mr_scalar_stats(h)
        # max_div is the rounding error of a sum that is zero: computed with the rest, but no number to compare
        stats.pop("max_div")
        nu_z, nu_T = mr.mr_scalar_profiles(h)
        mr.mr_upscale_scalar(h, s["Tc"])
        p = np.float64 if case["precision"] == "f64" else np.float32
        return {"dt": np.array([dt], p), "stats": np.array([stats[k] for k in sorted(stats)], p), "nu_z": nu_z.astype(p),
                "nu_T": np.array([nu_T], p), "Tc": s["Tc"].to(s["T0"].dtype)}
    from paper_1805_03426_gb300.autograd import scalar_loss

    leaves = [t.detach().requires_grad_(True) for t in (s["T0"], *s["par"])]
    loss = scalar_loss(h, leaves[0], *(p.double() for p in leaves[1:]), case["steps"], case["every"], *s["w"])
    loss.backward()
    return {"loss": loss.detach().to(s["T0"].dtype), "gT0": leaves[0].grad, "gU": leaves[1].grad, "gV": leaves[2].grad, "gW": leaves[3].grad}


def work(case):
    e = 8 if case["precision"] == "f64" else 4
    w, m3 = case["walls"], case["mx"] * case["my"] * case["mz"]
    Nx, Ny, Nz = case["nx"] * case["mx"], case["ny"] * case["my"], case["nz"] * case["mz"]
    cells, coarse = Nx * Ny * Nz, case["nx"] * case["ny"] * case["nz"]
    dense = Nz * Ny * (Nx + w) + Nz * (Ny + w) * Nx + (Nz + 1) * Ny * Nx
    # a step reads two scalar levels and the velocity (its dense faces where they are kept, else the coarse ones) and
    # writes one level; the operations are the six face fluxes and the time integration (and, where the velocity is
    # refined in the step, the split and balance of three faces)
    stored = case["mode"] == "stored"
    step_b = 3 * e * cells + (dense * e if stored else 3 * e * cells // m3)
    step_f = (38 if case["order"] == 2 else 80) * cells + (0 if stored else 30 * cells) + (6 * cells if case["implicit"] else 0)
    kind = case["kind"]
    if kind == "steps":
        return {"bytes": case["steps"] * step_b + 3 * e * cells, "flops": case["steps"] * step_f}
    if kind == "coupled":
        return {"bytes": case["steps"] * (step_b + 4 * 8 * coarse) + 3 * e * cells, "flops": case["steps"] * step_f}
    if kind == "temporal":
        return {"bytes": case["steps"] * (case["mt"] * step_b + 3 * 8 * coarse) + 3 * e * cells,
                "flops": case["steps"] * case["mt"] * step_f}
    if kind == "refine":
        return {"bytes": 3 * 8 * coarse + dense * e, "flops": 30 * cells}
    if kind == "diagnose":
        return {"bytes": e * cells + 4 * 8 * coarse + (dense * e if stored else 0), "flops": 60 * cells}
    # forward, recomputation and the adjoint sweep, which reads the level, the velocity and three adjoint levels and
    # accumulates three face gradients
    return {"bytes": case["steps"] * (2 * step_b + 5 * e * cells + 3 * dense * e), "flops": case["steps"] * 140 * cells}


# ---------------------------------------------------------------- the same in 64 bits


class _Axis:
    """One axis: dense faces, the R rows of every dense cell and the coarse cells they weigh (Section 3.2)."""

    def __init__(self, n, m, faces, periodic, dev):
        L = faces[-1] - faces[0]
        self.n, self.m, self.N, self.periodic = n, m, n * m, periodic
        R, win = np.zeros((n * m, 3)), np.zeros((n * m, 3), dtype=np.int64)

        def mean(a, b):
            return [1.0, 0.5 * (a + b), (a * a + a * b + b * b) / 3.0]

        for i in range(n):
            if m == 1:
                R[i], win[i] = [0, 1, 0], [i, i, i]
                continue
            first = i - 1 if periodic else min(max(i - 1, 0), n - 3)
            c, h = 0.5 * (faces[i * m] + faces[(i + 1) * m]), faces[(i + 1) * m] - faces[i * m]
            A, cells = [], []
            for q in range(first, first + 3):
                off = L * (q // n) if periodic else 0.0
                A.append(mean((faces[q % n * m] + off - c) / h, (faces[(q % n + 1) * m] + off - c) / h))
                cells.append(q % n)
            inv = np.linalg.inv(np.array(A))
            for b in range(m):
                R[i * m + b] = np.array(mean((faces[i * m + b] - c) / h, (faces[i * m + b + 1] - c) / h)) @ inv
                win[i * m + b] = cells
        self.R, self.win = torch.tensor(R, device=dev), torch.tensor(win, device=dev)

    def split(self, a, dim):
        """Coarse values along dim to dense ones."""
        if self.m == 1:
            return a
        shape = [1] * a.dim()
        shape[dim] = self.N
        return sum(a.index_select(dim, self.win[:, p]) * self.R[:, p].reshape(shape) for p in range(3))


class _Exact:
    def __init__(self, case, dt, dev):
        self.case, self.dt, self.dev = case, dt, dev
        self.w = case["walls"]
        nx, ny, nz, mx, my, mz = (case[k] for k in ("nx", "ny", "nz", "mx", "my", "mz"))
        self.Nx, self.Ny, self.Nz = nx * mx, ny * my, nz * mz
        zf = _zfaces(case)
        self.ax = _Axis(nx, mx, np.linspace(0, case["lx"], self.Nx + 1), not self.w, dev)
        self.ay = _Axis(ny, my, np.linspace(0, case["ly"], self.Ny + 1), not self.w, dev)
        self.az = _Axis(nz, mz, zf, False, dev)
        self.dx, self.dy = case["lx"] / self.Nx, case["ly"] / self.Ny
        col = lambda a: torch.tensor(np.ascontiguousarray(a), device=dev)[:, None, None]  # noqa: E731
        dz, zc = np.diff(zf), 0.5 * (zf[1:] + zf[:-1])
        self.zc, self.zf, self.dzh = zc, zf, dz
        self.dz = col(dz)
        self.kappa = (case["ra"] * case["pr"]) ** -0.5
        d = np.concatenate([[zc[0] - zf[0]], np.diff(zc), [zf[-1] - zc[-1]]])
        cdn, cup = self.kappa / (dz * d[:-1]), self.kappa / (dz * d[1:])
        if case["adiabatic"]:
            cdn[0] = cup[-1] = 0.0
        self.cdn_h, self.cup_h = cdn, cup
        self.cdn, self.cup = col(cdn), col(cup)
        self.wlo, self.whi = col(dz[1:] / (dz[:-1] + dz[1:])), col(dz[:-1] / (dz[:-1] + dz[1:]))  # inner faces
        self.dc = col(np.diff(zc))
        if case["order"] == 4:
            self.f4 = [self._face4(np.linspace(0, case["lx"], self.Nx + 1), not self.w),
                       self._face4(np.linspace(0, case["ly"], self.Ny + 1), not self.w), self._face4(zf, False)]

    def _face4(self, X, periodic):
        """[(weights, cells)] of the face values 0 .. N-1 (periodic) or 1 .. N-1: cubic through cell averages."""
        N, L = len(X) - 1, X[-1] - X[0]
        out_w, out_c = [], []
        for f in range(0 if periodic else 1, N):
            cells = list(range(f - 2, f + 2))
            if not periodic:
                cells = [c for c in cells if 0 <= c < N]
            lo = [X[c % N] + L * (c // N) - X[f] for c in cells]
            hi = [X[c % N + 1] + L * (c // N) - X[f] for c in cells]
            s = hi[-1] - lo[0]
            A = [[(b ** (p + 1) - a ** (p + 1)) / ((p + 1) * (b - a)) for a, b in zip(np.array(lo) / s, np.array(hi) / s)]
                 for p in range(len(cells))]
            w = np.linalg.solve(np.array(A), np.eye(len(cells))[0])
            out_w.append(list(w) + [0.0] * (4 - len(cells)))
            out_c.append([c % N for c in cells] + [0] * (4 - len(cells)))
        return torch.tensor(np.array(out_w), device=self.dev), torch.tensor(np.array(out_c), device=self.dev)

    def refine(self, U, V, W):
        """Dense faces of the coarse ones: split of the outer faces, then the slab, row and cell balances."""
        c, ax, ay, az = self.case, self.ax, self.ay, self.az
        mx, my, mz, nx, ny, nz = c["mx"], c["my"], c["mz"], c["nx"], c["ny"], c["nz"]
        DX, DY = self.dx * mx, self.dy * my

        def up(a, dim):  # the face on the far side of every cell
            return a.narrow(dim, 1, a.shape[dim] - 1) if self.w else torch.roll(a, -1, dim)

        def near(a, dim):
            return a.narrow(dim, 0, a.shape[dim] - 1) if self.w else a

        Uz, Vz = az.split(U, 0), az.split(V, 0)
        div = ((up(Uz, 2) - near(Uz, 2)) / DX + (up(Vz, 1) - near(Vz, 1)) / DY) * self.dz
        div = div.reshape(nz, mz, ny, nx)
        planes = [W[1:]]
        for b in range(mz - 1, 0, -1):
            planes.append(planes[-1] + div[:, b])
        Wc = torch.cat([torch.stack([W[:-1]] + planes[:0:-1], 1).reshape(self.Nz, ny, nx), W[-1:]])
        Wy = ay.split(Wc, 1)
        Ws = ax.split(Wy, 2)
        Uo = ay.split(Uz, 1)                                           # [Nz][Ny][coarse x faces]
        dU = ((up(Uo, 2) - near(Uo, 2)) / DX).reshape(self.Nz, ny, my, nx)
        dW = ((Wy[1:] - Wy[:-1]) / self.dz).reshape(self.Nz, ny, my, nx)
        rows = [near(Vz, 1)]
        for b in range(my - 1):
            rows.append(rows[-1] - self.dy * (dU[:, :, b] + dW[:, :, b]))
        Vc = torch.stack(rows, 2).reshape(self.Nz, self.Ny, nx)
        if self.w:
            Vc = torch.cat([Vc, Vz[:, -1:]], 1)
        Vs = ax.split(Vc, 2)
        d = ((up(Vs, 1) - near(Vs, 1)) / self.dy + (Ws[1:] - Ws[:-1]) / self.dz).reshape(self.Nz, self.Ny, nx, mx)
        cols = [near(Uo, 2)]
        for b in range(mx - 1):
            cols.append(cols[-1] - self.dx * d[..., b])
        Us = torch.stack(cols, 3).reshape(self.Nz, self.Ny, self.Nx)
        if self.w:
            Us = torch.cat([Us, Uo[:, :, -1:]], 2)
        return Us, Vs, Ws

    def _value(self, T, dim):
        """Advected face values: periodic faces 0 .. N-1, else the inner ones."""
        periodic = dim != 0 and not self.w
        if self.case["order"] == 4:
            w, cells = self.f4[2 - dim]
            shape = [1, 1, 1]
            shape[dim] = len(w)
            return sum(T.index_select(dim, cells[:, p]) * w[:, p].reshape(shape) for p in range(4))
        if periodic:
            return 0.5 * (T + torch.roll(T, 1, dim))
        n = T.shape[dim] - 1
        lo, hi = T.narrow(dim, 0, n), T.narrow(dim, 1, n)
        return self.wlo * lo + self.whi * hi if dim == 0 else 0.5 * (lo + hi)

    def advect(self, vel, T):
        out = 0.0
        for v, dim, h in ((vel[0], 2, self.dx), (vel[1], 1, self.dy), (vel[2], 0, self.dz)):
            f = self._value(T, dim)
            if dim != 0 and not self.w:
                f = v * f
                out = out - (torch.roll(f, -1, dim) - f) / h
            else:
                f = v.narrow(dim, 1, T.shape[dim] - 1) * f
                z = torch.zeros_like(f.narrow(dim, 0, 1))
                out = out - torch.diff(torch.cat([z, f, z], dim), dim=dim) / h
        return out

    def diffuse(self, T, vertical=True):
        out = 0.0
        for dim, h in ((2, self.dx), (1, self.dy)):
            if self.w:
                g = torch.diff(T, dim=dim)
                z = torch.zeros_like(g.narrow(dim, 0, 1))
                out = out + torch.diff(torch.cat([z, g, z], dim), dim=dim) * (self.kappa / h ** 2)
            else:
                out = out + (torch.roll(T, 1, dim) - 2 * T + torch.roll(T, -1, dim)) * (self.kappa / h ** 2)
        return out + self.diffuse_z(T) if vertical else out

    def diffuse_z(self, T):
        below = torch.cat([torch.full_like(T[:1], 0.5), T[:-1]])
        above = torch.cat([T[1:], torch.full_like(T[:1], -0.5)])
        return self.cdn * (below - T) + self.cup * (above - T)

    def solve_z(self, r, h):
        """(1 - h Lz) x = r with Lz the homogeneous vertical diffusion."""
        lo, up = -h * self.cdn_h, -h * self.cup_h
        di = 1 + h * (self.cdn_h + self.cup_h)
        c, x = np.zeros(self.Nz), [None] * self.Nz
        for k in range(self.Nz):
            den = di[k] - (lo[k] * c[k - 1] if k else 0.0)
            c[k] = up[k] / den
            x[k] = (r[k] - lo[k] * x[k - 1]) / den if k else r[k] / den
        for k in range(self.Nz - 2, -1, -1):
            x[k] = x[k] - c[k] * x[k + 1]
        return torch.stack(x)

    def step(self, vel, Tm, T, s):
        a, b, g = (0.0, 1.0, self.dt) if s == 0 else (0.5, 0.5, 1.5 * self.dt) if (s + 1) % 50 == 0 else (1.0, 0.0, 2 * self.dt)
        if not self.case["implicit"]:
            return a * Tm + b * T + g * (self.advect(vel, T) + self.diffuse(Tm))
        bz = torch.zeros_like(T)
        if not self.case["adiabatic"]:
            bz[0] += 0.5 * self.cdn[0]
            bz[-1] -= 0.5 * self.cup[-1]
        r = a * Tm + b * T + g * (self.advect(vel, T) + self.diffuse(Tm, False) + 0.5 * self.diffuse_z(Tm) + 0.5 * bz)
        return self.solve_z(r, 0.5 * g)

    def nu(self, T):
        return torch.stack([((0.5 - T[0]) / (self.zc[0] - self.zf[0])).mean(), ((T[-1] + 0.5) / (self.zf[-1] - self.zc[-1])).mean()])

    def moments(self, T):
        v = (self.dz * self.dx * self.dy).expand_as(T)
        total = (T * v).sum()
        mean = total / v.sum()
        return total, mean, ((T - mean) ** 2 * v).sum() / v.sum()

    def upscale(self, T):
        c = self.case
        t = (T * self.dz).reshape(c["nz"], c["mz"], c["ny"], c["my"], c["nx"], c["mx"]).sum((1, 3, 5))
        return t / (self.dz.reshape(c["nz"], c["mz"]).sum(1)[:, None, None] * c["my"] * c["mx"])

    def profiles(self, T, Ws):
        up = self._value(T, 0) * Ws[1:-1] / self.kappa - torch.diff(T, dim=0) / self.dc
        nu = self.nu(T)
        nu_z = torch.cat([nu[:1], up.mean((1, 2)), nu[1:]])
        s = 0.0
        for dim, h, area in ((2, self.dx, self.dy * self.dz), (1, self.dy, self.dx * self.dz)):
            d = torch.diff(T, dim=dim) if self.w else T - torch.roll(T, 1, dim)
            s = s + (d * d * area / h).sum()
        d = torch.diff(T, dim=0)
        s = s + (d * d / self.dc).sum() * self.dx * self.dy
        if not self.case["adiabatic"]:
            s = s + self.dx * self.dy * (((T[0] - 0.5) ** 2).sum() / (self.zc[0] - self.zf[0]) + ((T[-1] + 0.5) ** 2).sum() / (self.zf[-1] - self.zc[-1]))
        return nu_z, s / (self.case["lx"] * self.case["ly"])

    def cfl(self, vel, c):
        U, V, W = (v.abs() for v in vel)
        far = lambda a, dim: torch.maximum(a.narrow(dim, 0, a.shape[dim] - 1), a.narrow(dim, 1, a.shape[dim] - 1)) if self.w else torch.maximum(a, torch.roll(a, -1, dim))  # noqa: E731
        return c / (far(U, 2) / self.dx + far(V, 1) / self.dy + torch.maximum(W[1:], W[:-1]) / self.dz).amax()


def exact(case, seed):
    vel, T0, dt = _inputs(case, seed)
    x = _Exact(case, dt, T0.device)
    T0 = T0.double()
    kind = case["kind"]
    if kind == "adjoint":
        leaves = [t.detach().clone().requires_grad_(True) for t in (T0, *vel[0])]
        dense = x.refine(*leaves[1:])
        wnu, wvar = _loss_weights(case)
        Tm = T = leaves[0]
        loss = 0.0
        for s in range(case["steps"] + 1):
            if wnu[s]:
                loss = loss + wnu[s] * x.nu(T)[0]
            if wvar[s]:
                loss = loss + wvar[s] * x.moments(T)[2]
            if s < case["steps"]:
                Tm, T = T, x.step(dense, Tm, T, s)
        loss.backward()
        return {"loss": loss.detach(), "gT0": leaves[0].grad, "gU": leaves[1].grad, "gV": leaves[2].grad, "gW": leaves[3].grad}
    dense = [x.refine(*v) for v in vel]
    if kind == "refine":
        return list(dense[0])
    if kind == "diagnose":
        total, mean, var = x.moments(T0)
        nu = x.nu(T0)
        nu_z, nu_T = x.profiles(T0, dense[0][2])
        stats = dict(nu_bot=nu[0], nu_top=nu[1], mean=mean, var=var, integral=total)
        return {"dt": x.cfl(dense[0], 0.3).reshape(1), "stats": torch.stack([stats[k] for k in sorted(stats)]), "nu_z": nu_z,
                "nu_T": nu_T.reshape(1), "Tc": x.upscale(T0)}
    Tm, T, s = T0, T0, 0
    nus, Tcs = [], []
    for i in range(case["steps"]):
        if kind == "temporal":
            A, B = dense[i % 2], dense[(i + 1) % 2]
            for q in range(case["mt"]):
                Tm, T = T, x.step([p + q / case["mt"] * (r - p) for p, r in zip(A, B)], Tm, T, s)
                s += 1
        else:
            Tm, T = T, x.step(dense[i % len(dense)], Tm, T, s)
            s += 1
        if kind == "coupled":
            nus.append(x.nu(T))
            Tcs.append(x.upscale(T))
    out = {"T": T, "Tprev": Tm}
    if case["precision"] == "f64":
        out["nu"] = torch.stack(nus) if nus else x.nu(T).reshape(1, 2)
    if kind == "coupled":
        out["Tc"] = torch.stack(Tcs)
    return out
