"""Performance cases of the Richards solver: what a program that uses the
library has it do, through its public entry points.

Kinds of work
  run       ``Solver.run`` over a fixed simulated window from a given state
            (state upload, time steps, state read-back, water balance);
  assemble  ``Solver.assemble``: closures and the Picard system at two heads;
  solve     ``Solver.solve``: one linear system from a given start;
  ensemble  ``Ensemble.run``: independent columns and blocks of uneven size;
  network   ``Network.forward`` / ``Network.loss_grad`` of the warm start.

Sizes come from the repository's own workloads: the 1-D loam column, the
128 x 128 x 64 heterogeneous box, the 512 x 512 x 64 watershed, the tilted
slope, the uneven ensemble and the warm start's training volumes, with ragged
and odd relatives of each.  Inputs are synthetic and made on the device from
the seed alone.

``exact`` restates the method in plain torch at 64 bits (Picard, backward
Euler, conjugate gradients to a hundredth of the solver's tolerance); it uses
nothing of this repository.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1809_10895_gb300 import rf

F64 = torch.float64


def _dev():
    return torch.device("cuda", torch.cuda.current_device())


# ----------------------------------------------------------------- the cases
def listed():
    return [
        # The paper's 1-D infiltration column (200 cells of 5 mm, ponded loam)
        # through its first simulated seconds: the smallest problem, all latency.
        dict(name="column_fp64", kind="run", ground="column", nx=1, ny=1, nz=200, precision="fp64", picard="chord",
             steps=4, dt=1.0),
        # A small block with no size a multiple of anything, as a test or a
        # calibration run steps many times.
        dict(name="box_small_fp64", kind="run", ground="box", nx=33, ny=31, nz=29, precision="fp64", picard="chord",
             steps=6, dt=60.0),
        # The heterogeneous box at its configured size under rain, the
        # ordinary production run on the paper's FP64 path.
        dict(name="box_fp64", kind="run", ground="box", nx=128, ny=128, nz=64, precision="fp64", picard="chord",
             steps=4, dt=60.0),
        # The benchmark's masked watershed in a storm, full size, FP64: the
        # headline workload and the largest case.
        dict(name="watershed_fp64", kind="run", ground="watershed", nx=512, ny=512, nz=64, precision="fp64",
             picard="chord", steps=2, dt=120.0),
        # The same ground on the mixed-precision path (FP32 inner solve inside
        # FP64 defect correction), a smaller catchment.
        dict(name="watershed_mixed", kind="run", ground="watershed", nx=384, ny=320, nz=64, precision="mixed",
             picard="chord", steps=3, dt=120.0),
        # The paper's tilted slope at half its printed plan resolution, an odd
        # row length, modified Picard, mixed precision.
        dict(name="slope_mixed_modified", kind="run", ground="slope", nx=425, ny=211, nz=50, precision="mixed",
             picard="modified", steps=3, dt=120.0),
        # One assembled Picard system with its closures, as a program that
        # drives its own linear solver asks for it; ragged sizes.
        dict(name="assemble_fp64", kind="assemble", ground="box", nx=251, ny=243, nz=61, precision="fp64", dt=60.0),
        # One linear solve of a saturated, anisotropic block: many CG
        # iterations on the FP64 path ...
        dict(name="solve_fp64", kind="solve", ground="saturated", nx=256, ny=192, nz=64, precision="fp64", dt=60.0),
        # ... and on the mixed path.
        dict(name="solve_mixed", kind="solve", ground="saturated", nx=256, ny=256, nz=64, precision="mixed", dt=60.0),
        # Many small independent problems of uneven size at once (parameter
        # studies), mixed precision with the vertical-line preconditioner.
        dict(name="ensemble_mixed", kind="ensemble", n=32, side=10, nz_max=250, precision="mixed", precond="zline",
             t_end=1.0),
        # The learned warm start's guess for a half-million-cell block ...
        dict(name="network_forward", kind="network", mode="forward", D=32, H=128, W=128),
        # ... and a training evaluation (loss and all gradients) of it.
        dict(name="network_gradient", kind="network", mode="gradient", D=32, H=128, W=128),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["run", "run", "run", "run", "assemble", "solve", "solve", "ensemble", "network"])
    if kind == "run":
        ground = rng.choice(["column", "box", "box", "watershed", "watershed", "slope"])
        prec = rng.choice(["fp64", "mixed"])
        if ground == "column":
            return dict(kind="run", ground="column", nx=1, ny=1, nz=_log_int(rng, 60, 400), precision=prec,
                        picard="chord", steps=rng.randint(2, 6), dt=1.0)
        if ground == "box":
            s = _log_int(rng, 24, 200)
            return dict(kind="run", ground="box", nx=s, ny=max(8, int(s * rng.uniform(0.6, 1.1))),
                        nz=rng.randint(24, 72), precision=prec, picard=rng.choice(["chord", "modified"]),
                        steps=rng.randint(2, 5), dt=60.0)
        nx, ny = _log_int(rng, 96, 480), _log_int(rng, 96, 480)
        if ground == "watershed":
            return dict(kind="run", ground="watershed", nx=nx, ny=ny, nz=rng.randint(48, 64), precision=prec,
                        picard="chord", steps=2, dt=120.0)
        return dict(kind="run", ground="slope", nx=nx, ny=ny, nz=rng.randint(30, 50), precision=prec,
                    picard=rng.choice(["chord", "modified"]), steps=2, dt=120.0)
    if kind == "assemble":
        return dict(kind="assemble", ground=rng.choice(["box", "watershed"]), nx=_log_int(rng, 24, 400),
                    ny=_log_int(rng, 24, 400), nz=rng.randint(24, 64), precision=rng.choice(["fp64", "mixed"]), dt=60.0)
    if kind == "solve":
        return dict(kind="solve", ground="saturated", nx=_log_int(rng, 24, 300), ny=_log_int(rng, 24, 300),
                    nz=rng.randint(24, 64), precision=rng.choice(["fp64", "mixed"]), dt=60.0)
    if kind == "ensemble":
        return dict(kind="ensemble", n=rng.randint(6, 40), side=rng.randint(3, 10), nz_max=rng.randint(80, 250),
                    precision="mixed", precond=rng.choice(["zline", "jacobi"]), t_end=1.0)
    return dict(kind="network", mode=rng.choice(["forward", "gradient"]), D=rng.randint(8, 32),
                H=rng.randint(24, 128), W=rng.randint(24, 128))


# ------------------------------------------------------------------- grounds
LOAM = dict(model="vg", theta_r=0.078, theta_s=0.43, alpha=3.6, n=1.56, Ks=2.89e-6, S=1e-5)


def _gen(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed))
    return g


def _uniform(g, lo, hi):
    return float(lo + (hi - lo) * torch.rand((), generator=g, device=g.device, dtype=F64))


def _smooth_field(g, shape, corr):
    """Unit-variance correlated noise: white noise under an exponential-type
    spectrum with correlation length corr (cells) per axis."""
    f = torch.fft.rfftn(torch.randn(shape, generator=g, device=g.device, dtype=F64))
    k2 = torch.zeros((), device=g.device, dtype=F64)
    for ax, n in enumerate(shape):
        k = torch.fft.rfftfreq(n, device=g.device, dtype=F64) if ax == len(shape) - 1 else \
            torch.fft.fftfreq(n, device=g.device, dtype=F64)
        v = [1] * len(shape)
        v[ax] = k.numel()
        k2 = k2 + (2.0 * math.pi * corr * k.reshape(v)) ** 2
    f = f * (1.0 + k2) ** (-(len(shape) + 1) / 4.0)
    x = torch.fft.irfftn(f, s=shape)
    return (x - x.mean()) / x.std()


def _ground(case, seed):
    """Mesh, soils, fields, boundaries, parameters and heads of a case as a
    plain dict; fields are (nz, ny, nx) device tensors, z up."""
    g = _gen(seed)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    shape = (nz, ny, nx)
    dev = g.device
    G = dict(shape=shape, z_bottom=0.0, active=None, zone=None, Ks=None, grav=(0.0, 0.0, 1.0), t0=0.0,
             prm=dict(tol_picard=1e-6, tol_cg=1e-10, precision=case["precision"], dt0=case["dt"], dt_max=case["dt"],
                      picard_form=case.get("picard", "chord")))
    kind = case["ground"]
    if kind == "column":
        dz = 0.005
        G.update(d=(1.0, 1.0, dz), soils=[dict(LOAM)])
        h = torch.full(shape, _uniform(g, -1.1, -0.9), device=dev, dtype=F64)
        G["bcs"] = [("zmax", "dirichlet", 0.0), ("zmin", "free_drainage", None)]
        G["prm"].update(tol_cg=1e-12, f_grow=1.2, f_shrink=1.2, dt_max=600.0)
        G["h0"] = h
        return G
    if kind == "box":
        d = 0.25
        z = ((torch.arange(nz, device=dev, dtype=F64) + 0.5) * d).reshape(nz, 1, 1)
        top = nz * d
        G.update(d=(d, d, d), soils=[dict(model="vg", theta_r=0.05, theta_s=0.40, alpha=2.0, n=1.8, Ks=1e-5, S=1e-5)])
        G["Ks"] = torch.exp(math.log(1e-5) + _smooth_field(g, shape, 8.0))
        z_wt = top - min(10.0, 0.75 * top)
        # an hour into the rain: hydrostatic below a wetting front
        front = _uniform(g, 0.6, 1.2) + 0.2 * _smooth_field(g, shape[1:], 8.0)
        s = torch.sigmoid((front - (top - z)) / 0.3)
        h = (z_wt - z) * torch.ones(shape, device=dev, dtype=F64)
        G["h0"] = torch.maximum(h, h + s * (-0.8 - h)).contiguous()
        G["bcs"] = [("zmax", "flux", 1e-6), ("zmin", "dirichlet", z_wt)]
        G["t0"] = 3600.0
        return G
    if kind == "watershed":
        dx, dz = 10.0, 0.5
        z = ((torch.arange(nz, device=dev, dtype=F64) + 0.5) * dz).reshape(nz, 1, 1)
        hm = _smooth_field(g, (ny, nx), 40.0)
        hm = (hm - hm.min()) / (hm.max() - hm.min())
        surf = 0.5 * nz * dz * (1.0 + hm)
        act = z < surf
        soils = [dict(model="vg", theta_r=0.05, theta_s=0.40, alpha=_uniform(g, 0.5, 3.0), n=_uniform(g, 1.45, 2.5),
                      Ks=10.0 ** _uniform(g, -6.0, -4.0), S=1e-5) for _ in range(4)]
        zone = torch.clamp(torch.arange(nz, device=dev) // max(nz // 4, 1), max=3).to(torch.uint8)
        G.update(d=(dx, dx, dz), soils=soils, active=act,
                 zone=zone.reshape(nz, 1, 1).expand(shape).contiguous())
        # hydrostatic above a water table at the bottom, moister near the surface
        depth = surf - z
        h = -z * torch.ones(shape, device=dev, dtype=F64)
        s = torch.exp(-torch.clamp(depth, min=0.0) / _uniform(g, 0.8, 1.5))
        h = h + s * 0.5 * (-3.0 - h) * (h < -3.0)
        G["h0"] = torch.where(act, h, torch.zeros((), device=dev, dtype=F64)).contiguous()
        G["bcs"] = [("zmax", "flux", _uniform(g, 2.0, 4.0) * 1e-3 / 3600.0), ("zmin", "seepage", None)]
        G["t0"] = 11 * 3600.0
        return G
    if kind == "slope":
        a, b = math.radians(20.0), math.radians(3.0)
        G.update(d=(2.0, 2.0, 0.2), soils=[dict(LOAM)],
                 grav=(math.sin(a), math.cos(a) * math.sin(b), math.cos(a) * math.cos(b)))
        z = ((torch.arange(nz, device=dev, dtype=F64) + 0.5) * 0.2).reshape(nz, 1, 1)
        depth = nz * 0.2 - z
        h = torch.full(shape, -10.0, device=dev, dtype=F64) + 0.3 * _smooth_field(g, shape, 6.0)
        # rain has wetted the upper decimetres; the river keeps its bank moist
        h = h + (torch.exp(-depth / _uniform(g, 0.3, 0.6)) * 7.0)
        x = ((torch.arange(nx, device=dev, dtype=F64) + 0.5) * 2.0).reshape(1, 1, nx)
        h = h + torch.exp(-x / 6.0) * (-1.0 - h)
        G["h0"] = h.contiguous()
        G["bcs"] = [("xmin", "dirichlet", 0.0), ("zmax", "flux", 2e-7)]
        G["prm"].update(tol_picard=1e-3)
        return G
    # saturated: hydrostatic head above a Dirichlet bottom, log-normal Ks,
    # 10:1 anisotropic cells
    dz = 0.1
    z = ((torch.arange(nz, device=dev, dtype=F64) + 0.5) * dz).reshape(nz, 1, 1)
    G.update(d=(1.0, 1.0, dz), soils=[dict(model="vg", theta_r=0.05, theta_s=0.4, alpha=2.0, n=1.8, Ks=1e-4, S=1e-4)])
    G["Ks"] = torch.exp(math.log(1e-4) + 1.0 * torch.randn(shape, generator=g, device=dev, dtype=F64))
    G["h0"] = ((nz * dz + 2.0) - z + 0.2 * _smooth_field(g, shape, 6.0)).contiguous()
    G["bcs"] = [("zmin", "dirichlet", nz * dz + 1.5), ("zmax", "flux", 5e-5)]
    G["prm"].update(tol_cg=1e-12, tol_inner=1e-4)
    return G


def _heads(case, seed, G):
    """h^k and h^n of an assemble case: the state and a later iterate."""
    g = _gen(seed + 7777)
    hn = G["h0"]
    hk = hn + 0.05 * _smooth_field(g, G["shape"], 4.0) * (0.2 + torch.abs(hn))
    return hk.reshape(-1).contiguous(), hn.reshape(-1).contiguous()


def _solver(G):
    nz, ny, nx = G["shape"]
    act = None if G["active"] is None else G["active"].reshape(-1).to(torch.uint8).cpu().numpy()
    s = rf.Solver(nx, ny, nz, *G["d"], G["z_bottom"], act, params=rf.default_params(grav=G["grav"], **G["prm"]))
    s.set_soils(G["soils"], None if G["zone"] is None else G["zone"].reshape(-1).cpu().numpy(),
                None if G["Ks"] is None else G["Ks"].reshape(-1).cpu().numpy())
    for face, type_, v in G["bcs"]:
        s.set_bc(face, type_, None, v)
    return s


# ------------------------------------------------------------------ ensemble
def _instances(case, seed):
    """Instance sizes belong to the case (fixed); soils and heads to the seed."""
    sizes = np.random.default_rng(1234 + case["n"] + 100 * case["side"])
    rng = np.random.default_rng(seed)
    out = []
    for _ in range(case["n"]):
        nx, ny = (int(v) for v in sizes.integers(1, case["side"] + 1, 2))
        nz = int(sizes.integers(50, case["nz_max"] + 1))
        out.append(dict(nx=nx, ny=ny, nz=nz, h0=float(rng.uniform(-3.0, -0.1)),
                        soil=dict(model="vg", theta_r=0.05, theta_s=0.40, alpha=float(rng.uniform(0.5, 5.0)),
                                  n=float(rng.uniform(1.2, 2.5)), Ks=float(10 ** rng.uniform(-7, -4)), S=1e-5)))
    return out


# ------------------------------------------------------------------- network
NET_LAYERS = [(4, 32)] + [(32, 32)] * 8 + [(32, 1)]


def _net_inputs(case, seed):
    g = _gen(seed)
    rng = np.random.default_rng(seed)
    parts = []
    for li, (ci, co) in enumerate(NET_LAYERS):
        std = math.sqrt(2.0 / (27 * ci)) * (0.3 if li and li % 2 == 0 else 1.0)
        parts += [rng.normal(0.0, std, 27 * ci * co), 0.01 * rng.normal(size=co)]
    theta = np.concatenate(parts).astype(np.float32)
    shape = (case["D"], case["H"], case["W"])
    f = torch.stack([-1.0 + 0.5 * _smooth_field(g, shape, 8.0), _smooth_field(g, shape, 8.0),
                     torch.zeros(shape, device=g.device, dtype=F64),
                     torch.full(shape, _uniform(g, -1.0, 1.0), device=g.device, dtype=F64)], dim=-1)
    f[-1, :, :, 2] = 1.0
    x = f.to(torch.float32)[None].contiguous()
    target = (0.5 * _smooth_field(g, shape, 4.0)).to(torch.float32)[None].contiguous()
    return theta, x, target


# ------------------------------------------------------------- prepare / run
def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        insts = []
        for c in _instances(case, seed):
            s = c["soil"]
            insts.append(rf.rf_ens_instance(c["nx"], c["ny"], c["nz"], 0.01, 0.01, 0.01,
                                            rf.rf_soil(0, s["theta_r"], s["theta_s"], s["alpha"], s["n"], s["Ks"],
                                                       s["S"]),
                                            c["h0"], rf.BC_TYPES["dirichlet"], -0.01, rf.BC_TYPES["free_drainage"],
                                            0.0))
        e = rf.Ensemble(insts, params=rf.default_params(precision=case["precision"], precond=case["precond"]))
        return dict(kind=kind, e=e, n=case["n"], t_end=case["t_end"])
    if kind == "network":
        theta, x, target = _net_inputs(case, seed)
        net = rf.Network()
        net.set_params(theta)
        y = torch.empty(x.shape[:4], dtype=torch.float32, device=x.device)
        return dict(kind=kind, mode=case["mode"], net=net, x=x, target=target, y=y)
    G = _ground(case, seed)
    s = _solver(G)
    st = dict(kind=kind, s=s, h0=G["h0"].reshape(-1), t0=G["t0"])
    if kind == "run":
        st.update(t_end=G["t0"] + case["steps"] * case["dt"], out=torch.empty_like(st["h0"]))
    else:
        hk, hn = _heads(case, seed, G)
        st.update(hk=hk, hn=hn, dt=case["dt"])
        if kind == "assemble":
            st["out"] = {k: torch.empty_like(hk) for k in ("K", "theta", "c", "b", "diag")}
        else:
            s.assemble(hk, hn, case["dt"])      # the system that the solve works on
            st["x"] = torch.empty_like(hk)
    return st


def run(st):
    kind = st["kind"]
    if kind == "run":
        s = st["s"]
        s.set_state_device(st["h0"], st["t0"])
        s.run(st["t_end"])
        s.get_state_device(st["out"])
        mb = s.mass_balance()
        return dict(h=st["out"], inflow=mb["inflow_cum"], storage=mb["storage"])
    if kind == "assemble":
        st["s"].assemble(st["hk"], st["hn"], st["dt"], **st["out"])
        return st["out"]
    if kind == "solve":
        st["x"].copy_(st["hk"])
        st["s"].solve(st["x"])
        return st["x"]
    if kind == "ensemble":
        e = st["e"]
        e.reset()
        e.run(st["t_end"])
        return [e.get(i)[0] for i in range(st["n"])]
    if st["mode"] == "forward":
        st["net"].forward(st["x"], st["y"])
        return st["y"]
    loss, grad = st["net"].loss_grad(st["x"], st["target"])
    return dict(loss=loss, grad=grad)


# --------------------------------------------------------------------- work
def work(case):
    """Each input read once and each output written once per pass; for
    iterations, per time step (run) or per assembled system (solve).  Flops:
    closures (about 100 per cell) and operator applications (about 20) that
    one Picard iteration with one CG iteration needs."""
    kind = case["kind"]
    if kind == "network":
        vox = case["D"] * case["H"] * case["W"]
        fl = 2.0 * 27 * (4 * 32 + 8 * 32 * 32 + 32) * vox
        by = vox * (16 + 4) + 4 * 225793
        if case["mode"] == "forward":
            return dict(bytes=by, flops=fl)
        return dict(bytes=by + 4 * 225793 + 8 * vox, flops=3.0 * fl)
    if kind == "ensemble":
        cells = sum(c["nx"] * c["ny"] * c["nz"] for c in _instances(case, 0))
        steps = max(1.0, case["t_end"])
        return dict(bytes=16.0 * cells * steps, flops=160.0 * cells * steps)
    n = case["nx"] * case["ny"] * case["nz"]
    if case["ground"] == "watershed":
        n = 0.75 * n
    if kind == "run":
        # h, Ks, zone and flags read, h written, a step
        return dict(bytes=26.0 * n * case["steps"], flops=160.0 * n * case["steps"])
    if kind == "assemble":
        # h^k, h^n, Ks, zone, flags read; five arrays written
        return dict(bytes=66.0 * n, flops=240.0 * n)
    # diagonal, three face coefficients, right side and start read, x written
    return dict(bytes=56.0 * n, flops=40.0 * n)


# -------------------------------------------------- the method in plain torch
class _Ref:
    """Picard / backward-Euler finite volumes on (nz, ny, nx) tensors."""

    def __init__(self, G):
        self.G = G
        self.shape = G["shape"]
        dx, dy, dz = G["d"]
        self.V = dx * dy * dz
        self.A = dict(x=dy * dz, y=dx * dz, z=dx * dy)
        self.dist = dict(x=dx, y=dy, z=dz)
        self.ax = dict(x=2, y=1, z=0)
        self.grav = dict(zip("xyz", G["grav"]))
        dev = G["h0"].device
        one = torch.ones(self.shape, device=dev, dtype=F64)
        self.act = torch.ones(self.shape, device=dev, dtype=torch.bool) if G["active"] is None else G["active"]
        zone = torch.zeros(self.shape, device=dev, dtype=torch.long) if G["zone"] is None else G["zone"].long()
        self.soil = {k: torch.tensor([s[k] for s in G["soils"]], device=dev, dtype=F64)[zone]
                     for k in ("theta_r", "theta_s", "alpha", "n", "Ks", "S")}
        self.Ks = self.soil["Ks"] if G["Ks"] is None else G["Ks"] * one
        p = dict(tol_picard=1e-6, tol_cg=1e-10, f_grow=1.3, f_shrink=1.3, n_inc=10, n_small=3, n_max=8)
        p.update(G["prm"])
        self.p = p
        self.modified = p["picard_form"] == "modified"
        # boundary faces: (face, outward sign, cells)
        self.bfaces = {}
        for a, lo, hi in (("x", "xmin", "xmax"), ("y", "ymin", "ymax"), ("z", "zmin", "zmax")):
            for face, sgn in ((lo, -1), (hi, 1)):
                m = torch.zeros(self.shape, device=dev, dtype=torch.bool)
                m.select(self.ax[a], 0 if sgn < 0 else self.shape[self.ax[a]] - 1)[...] = True
                if a == "z":        # a vertical face towards an inactive cell too
                    if sgn > 0:
                        m[:-1] |= ~self.act[1:]
                    else:
                        m[1:] |= ~self.act[:-1]
                self.bfaces[face] = (a, sgn, m & self.act)

    def closure(self, h):
        s = self.soil
        sat = h >= 0.0
        u = torch.where(sat, torch.ones_like(h), -s["alpha"] * h)
        m = 1.0 - 1.0 / s["n"]
        nl = s["n"] * torch.log(u)
        x = torch.exp(nl)
        l1 = torch.log1p(x)
        se = torch.exp(-m * l1)
        omy = -torch.expm1(-m * torch.log1p(torch.exp(-nl)))     # 1 - (x/(1+x))^m
        ys = torch.exp(-m * torch.log1p(torch.exp(-nl)))
        dth = s["theta_s"] - s["theta_r"]
        th = torch.where(sat, s["theta_s"] + s["S"] * h, s["theta_r"] + dth * se)
        K = torch.where(sat, self.Ks, self.Ks * torch.sqrt(se) * omy * omy)
        C = torch.where(sat, s["S"] * torch.ones_like(h), dth * s["alpha"] * s["n"] * m * ys / (1.0 + x))
        z = torch.zeros((), device=h.device, dtype=F64)
        return torch.where(self.act, th, z), torch.where(self.act, K, z), torch.where(self.act, C, z)

    def boundary(self, hn, K):
        """Per boundary face: (cells, transmissibility, head, explicit inflow)."""
        out = []
        for face, type_, v in self.G["bcs"]:
            a, sgn, m = self.bfaces[face]
            A = self.A[a]
            zero = torch.zeros_like(K)
            g = sgn * self.grav[a]
            if type_ == "seepage":
                m, type_, v = m & (hn >= 0.0), "dirichlet", 0.0
            if type_ == "dirichlet":
                KD = torch.where(m, self.closure(torch.full_like(K, v))[1], zero)
                T = KD * A / (0.5 * self.dist[a])
                out.append((T, v, g * KD * A))
            elif type_ == "flux":
                out.append((zero, 0.0, torch.where(m, v * A * torch.ones_like(K), zero)))
            else:                   # free drainage
                out.append((zero, 0.0, torch.where(m, g * K * A, zero)))
        return out

    def assemble(self, hk, hn, dt, thk, thn, K, C):
        dh = hk - hn
        chord = torch.abs(dh) > 1e-10
        if self.modified:
            c = self.V / dt * C
            b = c * hk - self.V / dt * (thk - thn)
        else:
            Cc = torch.where(chord, (thk - thn) / torch.where(chord, dh, torch.ones_like(dh)), C)
            c = self.V / dt * Cc
            b = c * hn
        diag = c.clone()
        T = {}
        for a in "xyz":
            ax, n = self.ax[a], self.shape[self.ax[a]]
            T[a] = None
            if n < 2:
                continue
            lo, hi = torch.narrow(K, ax, 0, n - 1), torch.narrow(K, ax, 1, n - 1)
            both = torch.narrow(self.act, ax, 0, n - 1) & torch.narrow(self.act, ax, 1, n - 1)
            Kb = torch.where(both, 0.5 * (lo + hi), torch.zeros_like(lo))
            T[a] = Kb * self.A[a] / self.dist[a]
            torch.narrow(diag, ax, 0, n - 1).add_(T[a])
            torch.narrow(diag, ax, 1, n - 1).add_(T[a])
            gr = Kb * (self.A[a] * self.grav[a])
            torch.narrow(b, ax, 0, n - 1).add_(gr)
            torch.narrow(b, ax, 1, n - 1).sub_(gr)
        for Tb, hD, q in self.boundary(hn, K):
            diag = diag + Tb
            b = b + Tb * hD + q
        z = torch.zeros((), device=hk.device, dtype=F64)
        return torch.where(self.act, c, z), torch.where(self.act, b, z), torch.where(self.act, diag, z), T

    def apply(self, diag, T, x):
        y = diag * x
        for a in "xyz":
            if T[a] is None:
                continue
            ax, n = self.ax[a], self.shape[self.ax[a]]
            torch.narrow(y, ax, 0, n - 1).sub_(T[a] * torch.narrow(x, ax, 1, n - 1))
            torch.narrow(y, ax, 1, n - 1).sub_(T[a] * torch.narrow(x, ax, 0, n - 1))
        return y

    def solve(self, diag, T, b, x, tol):
        """Jacobi-preconditioned conjugate gradients, restarted once so that
        the residual it stops on is the true one."""
        di = torch.where(self.act, 1.0 / torch.where(self.act, diag, torch.ones_like(diag)), torch.zeros_like(diag))
        x = torch.where(self.act, x, torch.zeros_like(x))
        bb = float(torch.linalg.vector_norm(b))
        for _ in range(2):
            r = b - self.apply(diag, T, x)
            z = di * r
            p, rz = z.clone(), (r * z).sum()
            for _ in range(20000):
                if float(torch.linalg.vector_norm(r)) <= tol * bb:
                    break
                q = self.apply(diag, T, p)
                al = rz / (p * q).sum()
                x = x + al * p
                r = r - al * q
                z = di * r
                rn = (r * z).sum()
                p = z + (rn / rz) * p
                rz = rn
        return x

    def run(self, h, t, t_end):
        """(h, inflow, storage) at t_end under EBATS."""
        p, inflow = self.p, 0.0
        h = torch.where(self.act, h, torch.zeros_like(h))
        thn, K, C = self.closure(h)
        dtn, easy = min(p["dt0"], p["dt_max"]), 0
        tol = lambda s: 1e-9 * max(1.0, abs(s))  # noqa: E731
        while t < t_end - tol(t_end):
            dt = min(dtn, t_end - t)
            hk, thk, Kk, Ck, conv = h, thn, K, C, False
            for it in range(1, p["n_max"] + 1):
                c, b, diag, T = self.assemble(hk, h, dt, thk, thn, Kk, Ck)
                x = self.solve(diag, T, b, hk, 1e-2 * p["tol_cg"])
                Kold = Kk
                thk, Kk, Ck = self.closure(x)
                dmax = float(torch.where(self.act, torch.abs(x - hk), torch.zeros_like(x)).max())
                hk = x
                if dmax <= p["tol_picard"]:
                    conv = True
                    break
            if not conv:
                dtn, easy = dt / p["f_shrink"], 0
                continue
            for Tb, hD, q in self.boundary(h, Kold):
                inflow += dt * float(torch.clamp(Tb * (hD - hk) + q, min=0.0).sum())
            h, thn, K, C = hk, thk, Kk, Ck
            t = t_end if abs(t + dt - t_end) <= tol(t + dt) else t + dt
            easy = easy + 1 if it <= p["n_small"] else 0
            if easy >= p["n_inc"]:
                dtn, easy = min(dtn * p["f_grow"], p["dt_max"]), 0
        return h, inflow, self.V * float(thn.sum())


def _exact_network(case, seed):
    theta, x, target = _net_inputs(case, seed)
    th = torch.tensor(theta, device=x.device, dtype=F64, requires_grad=case["mode"] == "gradient")
    layers, o = [], 0
    for ci, co in NET_LAYERS:
        W = th[o:o + 27 * ci * co].reshape(co, 3, 3, 3, ci).permute(0, 4, 1, 2, 3)
        o += 27 * ci * co
        layers.append((W, th[o:o + co]))
        o += co
    conv = lambda a, l: torch.nn.functional.conv3d(a, l[0], l[1], padding=1)  # noqa: E731
    a = torch.relu(conv(x.double().permute(0, 4, 1, 2, 3), layers[0]))
    for k in range(4):
        a = torch.relu(conv(torch.relu(conv(a, layers[1 + 2 * k])), layers[2 + 2 * k]) + a)
    y = conv(a, layers[-1])[:, 0]
    if case["mode"] == "forward":
        return y.detach()
    loss = ((y - target.double()) ** 2).mean()
    loss.backward()
    return dict(loss=float(loss.detach()), grad=th.grad.cpu().numpy())


def exact(case, seed):
    kind = case["kind"]
    if kind == "network":
        return _exact_network(case, seed)
    if kind == "ensemble":
        # the two smallest instances; the others have no value here
        insts = _instances(case, seed)
        order = sorted(range(len(insts)), key=lambda i: insts[i]["nx"] * insts[i]["ny"] * insts[i]["nz"])[:2]
        out = [None] * len(insts)
        for i in order:
            c = insts[i]
            shape = (c["nz"], c["ny"], c["nx"])
            G = dict(shape=shape, d=(0.01, 0.01, 0.01), active=None, zone=None, Ks=None, grav=(0.0, 0.0, 1.0),
                     soils=[c["soil"]], bcs=[("zmax", "dirichlet", -0.01), ("zmin", "free_drainage", None)],
                     h0=torch.full(shape, c["h0"], device=_dev(), dtype=F64),
                     prm=dict(dt0=1.0, dt_max=600.0, picard_form="chord"))
            out[i] = _Ref(G).run(G["h0"], 0.0, case["t_end"])[0].reshape(-1).cpu().numpy()
        return out
    G = _ground(case, seed)
    R = _Ref(G)
    if kind == "run":
        h, inflow, storage = R.run(G["h0"], G["t0"], G["t0"] + case["steps"] * case["dt"])
        return dict(h=h.reshape(-1), inflow=inflow, storage=storage)
    hk, hn = (a.reshape(G["shape"]) for a in _heads(case, seed, G))
    thn = R.closure(hn)[0]
    thk, K, C = R.closure(hk)
    c, b, diag, T = R.assemble(hk, hn, case["dt"], thk, thn, K, C)
    if kind == "assemble":
        K = torch.where(R.act, K, torch.full_like(K, -1.0))      # inactive cells carry -1
        return {k: v.reshape(-1) for k, v in dict(K=K, theta=thk, c=c, b=b, diag=diag).items()}
    return R.solve(diag, T, b, hk, 1e-2 * G["prm"]["tol_cg"]).reshape(-1)
