"""The performance cases of the library: what its users have it do, through the public entry points.

Families (the key "family" of a case):
  flow    gks.Solver on a rectilinear grid: copy a state in, take time steps, copy the state out
  corner  the same on a body-fitted grid (Solver.set_nodes): a wall-clustered compression corner
  steady  gks.SteadySolver: multigrid cycles on that corner
  faces   gks.face_flux: interface fluxes of the caller's own reconstruction
  serve   serve.Server: a burst of independent solves of mixed sizes

exact() restates the scheme in 64-bit torch: generic polynomial moments of the Maxwellians (every
monomial's moment a product of one-dimensional ones) on whole-grid arrays.  Single-precision runs
return float32 (what such a run resolves), double-precision runs float64.
"""
import itertools
import math

import numpy as np
import torch

from paper_1302_2132_gb300 import gks, inputs, serve

GAMMA = 1.4
CFL = 0.5


def listed():
    return [
        # the shock tube every user starts with, in the checking precision; the smallest call: each
        # step is a few hundred faces, so latency and launches count
        dict(name="sod_400_fp64", family="flow", flow="sod", dim=1, nx=400, ny=1, nz=1, model="none",
             precision="fp64", expand="directional", recon="muscl2", limiter="vanleer", steps=145),
        # a small 2D solve (the small end of the serving mix) run by itself
        dict(name="quadrant_64_fp32", family="flow", flow="quadrant", dim=2, nx=64, ny=64, nz=1, model="none",
             precision="fp32", expand="multid", recon="muscl2", limiter="minmod", steps=97),
        # the headline: decaying turbulence, k-epsilon, FP32 flux with the IEEE double state
        dict(name="turb_1024_acc64", family="flow", flow="turbulence", dim=2, nx=1024, ny=1024, nz=1, model="keps",
             precision="fp32_acc64", expand="multid", recon="muscl2", limiter="vanleer", steps=49),
        # the same flow in double precision (verification runs)
        dict(name="turb_512_fp64", family="flow", flow="turbulence", dim=2, nx=512, ny=512, nz=1, model="keps",
             precision="fp64", expand="multid", recon="muscl2", limiter="vanleer", steps=7),
        # shock / boundary layer on a stretched grid: wall, Dirichlet inflow and top, k-omega, C_a > 0
        dict(name="shock_bl_1024x384_acc64", family="flow", flow="boundary_layer", dim=2, nx=1024, ny=384, nz=1,
             model="komega", precision="fp32_acc64", expand="multid", recon="muscl2", limiter="vanleer", steps=49),
        # 3D turbulence, larger than the L2 cache (the largest case)
        dict(name="turb3d_160_acc64", family="flow", flow="turbulence", dim=3, nx=160, ny=160, nz=160, model="keps",
             precision="fp32_acc64", expand="multid", recon="muscl2", limiter="vanleer", steps=7),
        # fifth-order reconstruction on an odd, non-square grid, float-pair state
        dict(name="turb_weno5_603x501_fp32", family="flow", flow="turbulence", dim=2, nx=603, ny=501, nz=1,
             model="keps", precision="fp32", expand="multid", recon="weno5", limiter="vanleer", steps=49),
        # k and omega transported with the flow
        dict(name="transport_512_fp32", family="flow", flow="turbulence", dim=2, nx=512, ny=512, nz=1,
             model="komega_transport", precision="fp32", expand="multid", recon="muscl2", limiter="vanleer", steps=49),
        # the paper's fine corner grid, time-accurate
        dict(name="corner_528x136_fp32", family="corner", nx=528, ny=136, precision="fp32", steps=97),
        # the paper's own mode: steady solver on the same grid, local time steps, LU-SGS, four levels
        dict(name="steady_528x136_fp32", family="steady", nx=528, ny=136, precision="fp32", levels=4, cycles=20),
        # stateless interface fluxes for a caller with its own reconstruction
        dict(name="faces_3d_400k_fp32", family="faces", dim=3, count=400000, precision="fp32", expand="multid"),
        # serving: a burst of solves, half 1D and half 2D
        dict(name="serve_16_fp32", family="serve", count=16, mix=4000, precision="fp32"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same families and ranges."""
    family = rng.choice(["flow1", "flow2", "flow2", "flow2", "flow3", "corner", "steady", "faces", "serve"])
    if family == "flow1":
        return dict(family="flow", flow=rng.choice(["sod", "turbulence"]), dim=1, nx=_log(rng, 100, 8192), ny=1, nz=1,
                    model="none", precision=rng.choice(["fp64", "fp32", "fp32_acc64"]), expand="directional",
                    recon="muscl2",
                    limiter=rng.choice(["minmod", "vanleer"]), steps=rng.randint(50, 145))
    if family == "flow2":
        flow = rng.choice(["turbulence", "quadrant", "boundary_layer"])
        precision = rng.choice(["fp64", "fp32", "fp32", "fp32_acc64", "fp32_acc64"])
        top = 512 if precision == "fp64" else 1024
        model = {"turbulence": rng.choice(["keps", "none", "komega_transport"]), "quadrant": "none",
                 "boundary_layer": "komega"}[flow]
        recon = "muscl2"
        if precision != "fp32_acc64" and model != "komega_transport":
            recon = rng.choice(["muscl2", "muscl2", "muscl3", "weno5"])
        if flow == "boundary_layer":
            nx, ny = _log(rng, 64, top), _log(rng, 45, 384)
        else:
            nx, ny = _log(rng, 48, top), _log(rng, 48, top)
        return dict(family="flow", flow=flow, dim=2, nx=nx, ny=ny, nz=1, model=model, precision=precision,
                    expand=rng.choice(["multid", "multid", "directional"]), recon=recon,
                    limiter=rng.choice(["vanleer", "minmod"]), steps=rng.randint(3, 7) if precision == "fp64"
                    else rng.randint(10, 49))
    if family == "flow3":
        precision = rng.choice(["fp64", "fp32", "fp32_acc64"])
        top = 64 if precision == "fp64" else 160
        return dict(family="flow", flow="turbulence", dim=3, nx=_log(rng, 20, top), ny=_log(rng, 20, top),
                    nz=_log(rng, 20, top), model=rng.choice(["keps", "none"]), precision=precision,
                    expand=rng.choice(["multid", "directional"]), recon="muscl2", limiter="vanleer",
                    steps=rng.randint(2, 6))
    if family == "corner":
        precision = rng.choice(["fp32", "fp32", "fp32_acc64", "fp64"])
        return dict(family="corner", nx=_log(rng, 96, 528 if precision == "fp64" else 1056),
                    ny=_log(rng, 48, 136 if precision == "fp64" else 272), precision=precision,
                    steps=rng.randint(5, 9) if precision == "fp64" else rng.randint(30, 97))
    if family == "steady":
        return dict(family="steady", nx=16 * rng.randint(8, 66), ny=8 * rng.randint(6, 34),
                    precision=rng.choice(["fp32", "fp32", "fp64"]), levels=rng.choice([3, 4]), cycles=rng.randint(5, 12))
    if family == "faces":
        precision = rng.choice(["fp32", "fp64"])
        return dict(family="faces", dim=rng.choice([1, 2, 3]), count=_log(rng, 1000, 400000), precision=precision,
                    expand=rng.choice(["directional", "multid"]))
    return dict(family="serve", count=rng.randint(4, 20), mix=rng.randint(1, 1 << 20), precision="fp32")


# ---- inputs ------------------------------------------------------------------------------------------
def _shape(case):
    return (case["nz"], case["ny"], case["nx"])[3 - case["dim"]:]


def _turbulence(case, gen, dev):
    """Random-phase solenoidal velocity with E(k) ~ k^4 exp(-2 (k/k0)^2) on [0, 2 pi)^dim at turbulent
    Mach 0.3 (0.5 in 3D), rho = 1, p = 1/gamma; log-normal k and epsilon of a few Fourier modes."""
    D, shape = case["dim"], _shape(case)
    k0 = 4.0 if D == 3 else 8.0
    kk = torch.meshgrid(*[torch.fft.fftfreq(n, d=1.0 / n, device=dev, dtype=torch.float64) for n in shape],
                        indexing="ij")[::-1]  # kk[0] along x, the last array axis
    k2 = sum(k * k for k in kk)
    km = torch.where(k2 == 0, torch.ones_like(k2), k2).sqrt()
    amp = torch.sqrt(km ** 4 * torch.exp(-2.0 * (km / k0) ** 2) / km ** (D - 1)) * (k2 > 0)
    uh = [torch.fft.fftn(torch.randn(shape, generator=gen, device=dev, dtype=torch.float64)) * amp for _ in range(D)]
    if D > 1:
        dot = sum(u * k for u, k in zip(uh, kk)) / km ** 2
        uh = [u - dot * k for u, k in zip(uh, kk)]
    vel = [torch.fft.ifftn(u).real for u in uh]
    urms = torch.sqrt(sum((v * v).mean() for v in vel))
    mach = 0.5 if D == 3 else 0.3
    one = torch.ones(shape, device=dev, dtype=torch.float64)
    prim = torch.stack([one] + [v * (mach / urms) for v in vel] + [one / GAMMA])
    x = torch.meshgrid(*[torch.arange(n, device=dev, dtype=torch.float64) * (2 * math.pi / n) for n in shape],
                       indexing="ij")

    def field(ref):
        s = torch.zeros(shape, device=dev, dtype=torch.float64)
        for _ in range(8):
            r = torch.randn(2 + D, generator=gen, device=dev, dtype=torch.float64).tolist()
            s += r[0] * torch.cos(sum(round(2 * q) * c for q, c in zip(r[2:], x)) + 3.0 * r[1])
        return (ref * torch.exp(0.5 * s / math.sqrt(8))).float().double()

    k_ref = 1.5 * mach * mach
    f1, f2 = field(k_ref), field(0.09 * k_ref * k_ref / 2e-5)
    if case["model"] == "komega_transport":
        f2 = (f2 / (0.09 * f1)).float().double()
    return dict(prim=prim, f1=f1, f2=f2, dx=[np.full(n, 2 * math.pi / n) for n in shape[::-1]], bc=[[0, 0]] * D,
                bc_prim=None, mu=1e-5, T_wall=1.0, C_a=0.0)


def _flow_inputs(case, seed, dev):
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    rng = np.random.default_rng(int(seed))
    D, shape = case["dim"], _shape(case)
    if case["flow"] == "turbulence":
        s = _turbulence(case, gen, dev)
        if case["model"] == "none":
            s["f1"] = s["f2"] = None
        return s
    if case["flow"] == "sod":
        n = case["nx"]
        left = (np.arange(n) + 0.5) / n < 0.5
        r, p = rng.uniform(0.9, 1.1, 2), rng.uniform(0.9, 1.1, 2)
        prim = np.stack([np.where(left, r[0], 0.125 * r[1]), np.zeros(n), np.where(left, p[0], 0.1 * p[1])])
        return dict(prim=torch.tensor(prim, device=dev), f1=None, f2=None, dx=[np.full(n, 1.0 / n)], bc=[[1, 1]],
                    bc_prim=None, mu=1e-5, T_wall=1.0, C_a=1.0)
    if case["flow"] == "quadrant":
        nx, ny = case["nx"], case["ny"]
        q = ((np.arange(nx) + 0.5) / nx >= 0.5).astype(int)[None, :] + 2 * ((np.arange(ny) + 0.5) / ny >= 0.5).astype(int)[:, None]
        st = np.stack([rng.uniform(0.1, 1.5, 4), rng.uniform(-0.8, 0.8, 4), rng.uniform(-0.8, 0.8, 4),
                       rng.uniform(0.1, 1.5, 4)])
        return dict(prim=torch.tensor(st[:, q], device=dev), f1=None, f2=None,
                    dx=[np.full(nx, 1.0 / nx), np.full(ny, 1.0 / ny)], bc=[[1, 1], [1, 1]], bc_prim=None, mu=1e-4,
                    T_wall=1.0, C_a=0.5)
    s = inputs.shock_boundary_layer(case["nx"], case["ny"])
    return dict(prim=_stirred(s["prim"], gen, dev), f1=torch.tensor(s["f1"], device=dev),
                f2=torch.tensor(s["f2"], device=dev), dx=s["dx"], bc=s["bc"], bc_prim=s["bc_prim"], mu=s["mu"],
                T_wall=s["T_wall"], C_a=0.5)


def _stirred(prim, gen, dev):
    """A profile with one percent of smooth disturbances in density, velocity and pressure."""
    p = torch.tensor(prim, device=dev)
    ny, nx = p.shape[1:]
    y = torch.arange(ny, device=dev, dtype=torch.float64)[:, None] * (2 * math.pi / ny)
    x = torch.arange(nx, device=dev, dtype=torch.float64)[None, :] * (2 * math.pi / nx)
    for v in range(4):
        r = torch.randn((3, 4), generator=gen, device=dev, dtype=torch.float64).tolist()
        s = sum(q[0] * torch.cos(round(2 * q[1]) * x + round(2 * q[2]) * y + 3.0 * q[3]) for q in r)
        p[v] += (p[v] if v != 2 else p[1]) * (0.01 * torch.tanh(s))
    return p


def _corner_inputs(case, seed, dev):
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    s = inputs.compression_corner(case["nx"], case["ny"])
    return dict(prim=_stirred(s["prim"], gen, dev), f1=torch.tensor(s["f1"], device=dev),
                f2=torch.tensor(s["f2"], device=dev), nodes=s["nodes"], bc=s["bc"], bc_prim=s["bc_prim"], mu=s["mu"],
                T_wall=s["T_wall"], C_a=0.5)


FACES = dict(dt=1e-3, mu=2e-5, C_a=0.4)


def _face_records(case, seed, dev):
    """Faces between states of any contrast, one third of them nearly equal, the relaxation time from
    zero to tens of time steps; records in the layout of gks_face_flux."""
    gen = torch.Generator(device=dev).manual_seed(int(seed))
    D, n = case["dim"], case["count"]
    nv = D + 2
    uni = lambda lo, hi, *s: lo + (hi - lo) * torch.rand((n,) + s, generator=gen, device=dev, dtype=torch.float64)

    def cons():
        rho, U, p = uni(0.3, 2.0), uni(-1.5, 1.5, D), uni(0.2, 2.0)
        return torch.cat([rho[:, None], rho[:, None] * U, (p / (GAMMA - 1) + 0.5 * rho * (U * U).sum(1))[:, None]], 1)

    nrm = lambda *s: torch.randn((n,) + s, generator=gen, device=dev, dtype=torch.float64)
    wl, wr = cons(), cons()
    wr = torch.where((uni(0, 1) < 0.33)[:, None], wl * (1 + 1e-4 * nrm(nv)), wr)
    h, sl, sr = uni(0.002, 0.05)[:, None], nrm(nv), nrm(nv)
    tt = nrm(2 * (D - 1) * nv)
    tau = torch.where(uni(0, 1) < 0.3, torch.zeros(n, device=dev, dtype=torch.float64),
                      FACES["dt"] * torch.exp(uni(-7.0, 3.0)))
    return torch.cat([wl, wr, wl - 0.5 * h * sl, wr + 0.5 * h * sr, sl, sr, tt, 0.5 * h, 0.5 * h, tau[:, None]],
                     1).contiguous()


SERVE = dict(gamma=GAMMA, mu=1e-4, C_a=0.5, cfl=CFL, limiter="vanleer", expand="multid")


def _requests(case, seed):
    """Half 1D, half 2D, sizes log-uniform as in the serving stream (2D up to 256^2), shorter runs: the
    sizes and step counts from the case's mix, the states from the seed."""
    out = []
    for i in range(case["count"]):
        rng, sizes = np.random.default_rng([int(seed), i]), np.random.default_rng([case["mix"], i])
        if i % 2 == 0:
            n = int(round(math.exp(sizes.uniform(math.log(256), math.log(4096)))))
            s = inputs.sod_1d(n) if i % 4 == 0 else inputs.turbulence_1d(n, seed=int(rng.integers(1 << 30)))
            if i % 4 == 0:
                s["prim"][2] *= rng.uniform(0.9, 1.1)
                s.update(lo=[0.0], hi=[1.0])
        else:
            n = int(round(math.exp(sizes.uniform(math.log(64), math.log(256)))))
            if i % 4 == 1:
                s = inputs.riemann_quadrant(n, seed=int(rng.integers(1 << 30)))
                s.update(lo=[0.0, 0.0], hi=[1.0, 1.0])
            else:
                s = inputs.turbulence(n, 2, seed=int(rng.integers(1 << 30)), k0=min(8.0, n / 8.0))
                s.update(lo=[0.0, 0.0], hi=[2 * math.pi, 2 * math.pi])
        s["nsteps"] = int(sizes.integers(40, 121))
        out.append(s)
    return out


# ---- the measured calls -------------------------------------------------------------------------------
def _out_type(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def prepare(case, seed):
    f = case["family"]
    dev = torch.device("cuda")
    if f == "serve":
        return dict(case=case, reqs=_requests(case, seed),
                    srv=serve.Server(precision=case["precision"], arena_bytes=1 << 30, max_cells=512 * 512))
    if f == "faces":
        return dict(case=case, recs=_face_records(case, seed, dev))
    if f == "flow":
        s = _flow_inputs(case, seed, dev)
        n = (case["nx"], case["ny"], case["nz"])[:case["dim"]]
        solver = gks.Solver(case["dim"], n, s["bc"], dx=s["dx"], bc_data=s["bc_prim"], gamma=GAMMA, mu=s["mu"],
                            T_wall=s["T_wall"], turb_model=case["model"], C_a=s["C_a"], limiter=case["limiter"],
                            expand=case["expand"], precision=case["precision"], reconstruction=case["recon"])
    else:
        s = _corner_inputs(case, seed, dev)
        n = (case["nx"], case["ny"])
        kw = dict(bc_data=s["bc_prim"], gamma=GAMMA, mu=s["mu"], T_wall=s["T_wall"], turb_model="komega",
                  C_a=s["C_a"], limiter="vanleer", expand="directional", precision=case["precision"])
        if f == "steady":
            solver = gks.SteadySolver(n, s["bc"], s["nodes"], levels=case["levels"], **kw)
        else:
            solver = gks.Solver(2, n, s["bc"], dx=[np.ones(n[0]), np.ones(n[1])], **kw)
            solver.set_nodes(s["nodes"])
    st = dict(case=case, solver=solver, prim=s["prim"].reshape(-1).contiguous())
    transport = case.get("model") == "komega_transport"
    if s["f1"] is not None:
        f1, f2 = s["f1"].reshape(-1).contiguous(), s["f2"].reshape(-1).contiguous()
        if transport:  # set with every new state
            st.update(f1=f1, f2=f2)
        else:
            solver.set_turbulence(f1, f2)
    if f != "steady":
        st["out"] = torch.empty(st["prim"].numel(), dtype=_out_type(case), device=dev)
        if transport:
            st["k"], st["om"] = (torch.empty(f1.numel(), dtype=_out_type(case), device=dev) for _ in range(2))
    return st


def run(state):
    case = state["case"]
    f = case["family"]
    if f == "faces":
        F, tau = gks.face_flux(case["dim"], state["recs"], FACES["dt"], gamma=GAMMA, mu=FACES["mu"],
                               C_a=FACES["C_a"], precision=case["precision"], expand=case["expand"])
        return {"F": F.to(_out_type(case)), "tau": tau.to(_out_type(case))}
    if f == "serve":
        srv = state["srv"]
        ids = [srv.submit(r, **SERVE) for r in state["reqs"]]
        srv.wait_all(600)
        return [srv.poll(i)[1].astype(np.float32) for i in ids]
    solver = state["solver"]
    solver.set_state(state["prim"], layout="soa_prim")
    if f == "steady":
        k = case["cycles"] // 4
        res = [solver.cycles(k, cfl=1.0, cfl_flux=0.5), solver.cycles(case["cycles"] - k, cfl=4.0, cfl_flux=0.5)]
        kind = np.float64 if case["precision"] == "fp64" else np.float32
        return {"W": solver.get_state().astype(kind), "res": np.concatenate(res).astype(kind)}
    if "f1" in state:
        solver.set_turbulence(state["f1"], state["f2"])
    solver.step(nsteps=case["steps"], cfl=CFL)
    out = {"W": solver.get_state(out=state["out"])}
    if "k" in state:
        out["k"], out["omega"] = solver.get_turbulence(state["k"], state["om"])
    return out


# Arithmetic of one interface flux and of one cell (slopes, relaxation time, update) in the closed
# form of the scheme, by dimension: what a pass has to compute whatever the layout.
_FLUX = {1: 350.0, 2: 650.0, 3: 1000.0}
_CELL = {1: 50.0, 2: 150.0, 3: 250.0}


def work(case):
    f = case["family"]
    if f == "faces":
        D, n = case["dim"], case["count"]
        nv = D + 2
        size = 8.0 if case["precision"] == "fp64" else 4.0
        return {"bytes": n * (8.0 * (6 * nv + 2 * (D - 1) * nv + 3) + size * (nv + 1)), "flops": n * _FLUX[D]}
    if f == "serve":
        # half 1D of about 1150 cells, half 2D of about 128^2, eighty steps
        h = case["count"] / 2.0
        return {"bytes": h * (1150 * 3 + 128 * 128 * 4) * 12.0,
                "flops": 80 * h * (1150 * (_FLUX[1] + _CELL[1]) + 128 * 128 * (2 * _FLUX[2] + _CELL[2]))}
    D = case.get("dim", 2)
    cells = float(case["nx"] * case["ny"] * case.get("nz", 1))
    passes = case["steps"] if f != "steady" else case["cycles"] * 3.0
    size = 8.0 if case["precision"] == "fp64" or f == "steady" else 4.0
    fields = 16.0 if case.get("model") == "komega_transport" else 0.0
    return {"bytes": cells * ((D + 2) * (8.0 + size) + fields + (2 * size if fields else 0.0)),
            "flops": passes * cells * (D * _FLUX[D] + _CELL[D])}


# ---- the scheme in 64 bits ----------------------------------------------------------------------------
class _Maxwellian:
    """Moments of a Maxwellian of state w: <u^i v^j w^k xi^(2l)> over the full line or a half line of u."""

    def __init__(self, w, K):
        D = len(w) - 2
        self.D, self.rho = D, w[0]
        self.U = [w[1 + d] / w[0] for d in range(D)]
        self.il = (2 * w[D + 1] / w[0] - sum(u * u for u in self.U)) / (K + D)  # 1 / (2 lambda)
        self.tang = [self._line(u, 6) for u in self.U[1:]]
        self.xi = [1.0, K * self.il, K * (K + 2) * self.il ** 2]
        self.K = K

    def _line(self, U, n, m0=None, m1=None):
        m = [torch.ones_like(U) if m0 is None else m0, U if m1 is None else m1]
        while len(m) < n + 1:
            m.append(U * m[-1] + (len(m) - 1) * self.il * m[-2])
        return m

    def full(self):
        return self._line(self.U[0], 7)

    def half(self, sign):
        lam = 0.5 / self.il
        m0 = 0.5 * torch.erfc(-sign * torch.sqrt(lam) * self.U[0])
        m1 = self.U[0] * m0 + sign * 0.5 * torch.exp(-lam * self.U[0] ** 2) / torch.sqrt(math.pi * lam)
        return self._line(self.U[0], 7, m0, m1)

    def moment(self, line, poly, shift=0):
        """<u^shift poly> for poly = {(i, j, .., l): coefficient}."""
        total = 0.0
        for e, c in poly.items():
            t = line[e[0] + shift]
            for d in range(self.D - 1):
                if e[1 + d]:
                    t = t * self.tang[d][e[1 + d]]
            if e[-1]:
                t = t * self.xi[e[-1]]
            total = total + c * t
        return total

    def slope(self, r):
        """a with <(a . psi) psi> = r, as a polynomial."""
        D, U, il = self.D, self.U, self.il
        R = [r[1 + d] - U[d] * r[0] for d in range(D)]
        q = sum(u * u for u in U) + (self.K + D) * il
        aE = (2 * r[D + 1] - q * r[0] - 2 * sum(u * x for u, x in zip(U, R))) / ((self.K + D) * il * il)
        a = [None] + [R[d] / il - U[d] * aE for d in range(D)]
        a[0] = r[0] - 0.5 * aE * q - sum(u * x for u, x in zip(U, a[1:]))
        return a + [aE]


def _psi(D):
    unit = lambda d, n: tuple(n if k == d else 0 for k in range(D + 1))
    out = [{unit(0, 0): 1.0}] + [{unit(d, 1): 1.0} for d in range(D)]
    return out + [{unit(d, 1 if d == D else 2): 0.5 for d in range(D + 1)}]


def _dot(a, psi):
    poly = {}
    for c, p in zip(a, psi):
        for e, v in p.items():
            poly[e] = poly.get(e, 0.0) + c * v
    return poly


def _times(p, q):
    out = {}
    for (e, a), (f, b) in itertools.product(p.items(), q.items()):
        k = tuple(x + y for x, y in zip(e, f))
        out[k] = out.get(k, 0.0) + a * b
    return out


def _amom(g, line, poly, psi, axis=0):
    """<c (a . psi) psi_m>, c the velocity along the axis (0 normal; None: 1)."""
    D = g.D
    out = []
    for p in psi:
        q = _times(poly, p)
        if axis is None or axis == 0:
            out.append(g.moment(line, q, 0 if axis is None else 1))
        else:
            e = tuple(1 if k == axis else 0 for k in range(D + 1))
            out.append(g.moment(line, _times(q, {e: 1.0})))
    return out


def _time_integrals(dt, tau):
    x = dt / tau
    s = torch.full_like(x, 1.0 / math.factorial(21))
    xs = torch.clamp(x, max=1.0)
    for m in range(20, 2, -1):
        s = 1.0 / math.factorial(m) - xs * s
    p3 = s
    p2 = 0.5 - xs * p3
    p1 = 1.0 - xs * p2
    e = 1.0 - xs * p1
    series = [dt * xs * p2, -dt * dt * xs * (p2 - 2 * p3), dt * dt * xs * p3, dt * p1, tau * dt * (e - 2 * p1),
              -tau * dt * p1, dt * dt * p2]
    e = torch.exp(-x)
    q = tau * (1.0 - e)
    T2 = 0.5 * dt * dt - tau * dt + tau * q
    closed = [dt - q, -tau * dt * (1 + e) + 2 * tau * q, T2, q, tau * dt * e - 2 * tau * q, -tau * q,
              tau * dt - tau * q]
    T = [torch.where(x < 1.0, a, b) for a, b in zip(series[:6], closed[:6])]
    # ratios to Dn = dt^2/2 - T2, formed where they do not vanish with tau
    y = tau / dt
    yq = y * (1.0 - e)
    big = [(2 * yq - 1 - e) / (1 - yq), (e - 2 * yq) / (1 - yq), -yq / (1 - yq)]
    small = [series[k] / series[6] for k in (1, 4, 5)]
    return T, [torch.where(x < 1.0, a, b) for a, b in zip(small, big)]


def _flux(wl, wr, cl, cr, sl, sr, tl, tr, dxl, dxr, tau_t, dt, mu, C_a):
    """Time-integrated flux in the face frame; tl, tr per tangential axis (empty: directional)."""
    D = len(wl) - 2
    K = 2.0 / (GAMMA - 1.0) - D
    psi = _psi(D)
    one = {tuple([0] * (D + 1)): 1.0}
    gl, gr = _Maxwellian(wl, K), _Maxwellian(wr, K)
    hl, hr = gl.half(1.0), gr.half(-1.0)
    w0 = [gl.rho * a + gr.rho * b for a, b in zip(_amom(gl, hl, one, psi, None), _amom(gr, hr, one, psi, None))]
    g0 = _Maxwellian(w0, K)
    pl, pr, p0 = gl.rho * gl.il, gr.rho * gr.il, g0.rho * g0.il
    tau = mu / p0 + tau_t + C_a * torch.abs(pr - pl) / (pr + pl) * dt
    T, (r1, r4, r5) = _time_integrals(dt, tau)
    rhs = [0.0] * (D + 2)
    F = [0.0] * (D + 2)

    def add(to, s, m):
        for k in range(D + 2):
            to[k] = to[k] + s * m[k]

    for g, line, s, t in ((gl, hl, sl, tl), (gr, hr, sr, tr)):
        a = _dot(g.slope([x / g.rho for x in s]), psi)
        b = [_dot(g.slope([x / g.rho for x in q]), psi) for q in t]
        full = g.full()
        r = [-x for x in _amom(g, full, a, psi)]
        for q, c in enumerate(b):
            add(r, -1.0, _amom(g, full, c, psi, 1 + q))
        A = _dot(g.slope(r), psi)
        w = g.rho / g0.rho
        u = {tuple([1] + [0] * D): 1.0}
        add(F, T[3] * g.rho, _amom(g, line, one, psi))
        for poly, axis, cr_, cf in [(a, 0, r4, T[4]), (A, None, r5, T[5])] + [(c, 1 + q, r4, T[4]) for q, c in enumerate(b)]:
            add(rhs, cr_ * w, _amom(g, line, poly, psi, axis))
            add(F, cf * g.rho, _amom(g, line, _times(poly, u), psi, axis))
    full, pos = g0.full(), g0.half(1.0)
    neg = g0.half(-1.0)
    u = {tuple([1] + [0] * D): 1.0}
    abar = [(pos, [(x - c) / (dxl * g0.rho) for x, c in zip(w0, cl)], 0),
            (neg, [(c - x) / (dxr * g0.rho) for x, c in zip(w0, cr)], 0)]
    abar += [(full, [0.5 * (x + y) / g0.rho for x, y in zip(tl[q], tr[q])], 1 + q) for q in range(len(tl))]
    for line, r, axis in abar:
        poly = _dot(g0.slope(r), psi)
        add(rhs, r1, _amom(g0, line, poly, psi, axis))
        add(F, T[1] * g0.rho, _amom(g0, line, _times(poly, u), psi, axis))
    Ab = _dot(g0.slope(rhs), psi)
    add(F, T[2] * g0.rho, _amom(g0, full, Ab, psi))
    add(F, T[0] * g0.rho, _amom(g0, full, one, psi))
    return F, tau


def _limit(kind, a, b):
    if kind == "minmod":
        return 0.5 * (torch.sign(a) + torch.sign(b)) * torch.minimum(a.abs(), b.abs())
    ab = a * b
    return torch.where(ab > 0, 2 * ab / torch.where(ab > 0, a + b, torch.ones_like(ab)), torch.zeros_like(ab))


def _pressure(W):
    D = len(W) - 2
    return (GAMMA - 1) * (W[D + 1] - 0.5 * sum(W[1 + d] ** 2 for d in range(D)) / W[0])


def _cons(prim):
    D = len(prim) - 2
    q = sum(prim[1 + d] ** 2 for d in range(D))
    return [prim[0]] + [prim[0] * prim[1 + d] for d in range(D)] + [prim[D + 1] / (GAMMA - 1) + 0.5 * prim[0] * q]


def _wall_image(w, T_wall):
    D = len(w) - 2
    p = _pressure(w)
    rho = p / (T_wall * T_wall / (p / w[0]))
    U = [-w[1 + d] / w[0] for d in range(D)]
    return [rho] + [rho * u for u in U] + [p / (GAMMA - 1) + 0.5 * rho * sum(u * u for u in U)]


H = 3  # ghost layers


def _ghosts(W, ax, s, side):
    """The H ghost layers of one side along array axis ax, outward order as in the padded array."""
    n = W[0].shape[ax]
    bc = s["bc"][s["D"] - 1 - ax][side]
    take = lambda idx: [w.index_select(ax, torch.tensor(idx, device=w.device)) for w in W]
    edge = 0 if side == 0 else n - 1
    if bc == 0:
        return take([(i - H) % n for i in range(H)] if side == 0 else [i % n for i in range(H)])
    if bc == 2:
        return _wall_image(take([H - 1 - i for i in range(H)] if side == 0 else [n - 1 - i for i in range(H)]), s["T_wall"])
    if bc == 3:
        d = _cons(list(torch.tensor(np.asarray(s["bc_prim"][s["D"] - 1 - ax][side]), device=W[0].device).T))
        other = 1 - ax  # (two-dimensional boundary data)
        m = W[0].shape[other]
        if m != d[0].numel():
            d = [torch.cat([x[:1].expand(H), x, x[-1:].expand(H)]) for x in d]
        return [x.unsqueeze(ax).expand([H if a == ax else m for a in range(2)]) for x in d]
    return take([edge] * H)


def _pad(W, s, axes=None):
    """Ghost cells: the last grid axis first (array axis 0), then towards x."""
    for ax in range(s["D"]) if axes is None else axes:
        lo, hi = _ghosts(W, ax, s, 0), _ghosts(W, ax, s, 1)
        W = [torch.cat([a, w, b], dim=ax) for a, w, b in zip(lo, W, hi)]
    return W


def _pad_field(f, s):
    for ax in range(s["D"]):
        n = f.shape[ax]
        idx = [i % n if s["bc"][s["D"] - 1 - ax][0] == 0 else min(max(i, 0), n - 1) for i in range(-H, n + H)]
        f = f.index_select(ax, torch.tensor(idx, device=f.device))
    return f


def _cut(f, ax, lo, hi):
    """f[lo : n + hi] along ax (n the padded length)."""
    return f.narrow(ax, lo, f.shape[ax] + hi - lo)


def _shifted(f, ax, k):
    """Neighbour k cells up along ax (periodic roll: only cells away from the padded edge are used)."""
    return torch.roll(f, -k, ax)


def _tau_t(model, P, f1, f2, grads, beta_star=0.09, C_mu=0.09):
    p = _pressure(P)
    S = torch.sqrt(2 * sum((0.5 * (grads[a][b] + grads[b][a])) ** 2 for a in range(len(grads)) for b in range(len(grads))))
    nu, eta = (C_mu * f1 * f1 / f2, S * f1 / f2) if model == "keps" else (f1 / f2, S / (beta_star * f2))
    t = P[0] * nu / (p * torch.sqrt(1 + eta * eta))
    return torch.where((f1 > 0) & (f2 > 0), t, torch.zeros_like(t))


def _muscl3(a, b, c):
    dm, dp = b - a, c - b
    return b + _limit("minmod", dm, 4 * dp) / 6 + _limit("minmod", dp, 4 * dm) / 3


def _weno5(a, b, c, d, e):
    q = [(2 * a - 7 * b + 11 * c) / 6, (-b + 5 * c + 2 * d) / 6, (2 * c + 5 * d - e) / 6]
    be = [13 / 12 * (a - 2 * b + c) ** 2 + 0.25 * (a - 4 * b + 3 * c) ** 2,
          13 / 12 * (b - 2 * c + d) ** 2 + 0.25 * (b - d) ** 2,
          13 / 12 * (c - 2 * d + e) ** 2 + 0.25 * (3 * c - 4 * d + e) ** 2]
    al = [g / (1e-6 + x) ** 2 for g, x in zip((0.1, 0.6, 0.3), be)]
    return sum(x * y for x, y in zip(al, q)) / sum(al)


def _physical(w):
    return (w[0] > 0) & (_pressure(w) > 0)


def _rect_run(case, s, dev, steps, mu, C_a, limiter, recon, expand, model):
    """Time steps on a rectilinear grid; returns conservative variables (and rho k, rho omega)."""
    D = case["dim"]
    s = dict(s, D=D)
    W = _cons(list(s["prim"]))
    transport = model == "komega_transport"
    f1, f2 = s["f1"], s["f2"]
    wid = []  # ghosted widths along each grid axis, shaped for broadcasting
    for d in range(D):
        w = np.asarray(s["dx"][d], dtype=np.float64)
        n = len(w)
        if s["bc"][d][0] == 0:
            g = [w[i % n] for i in range(-H, n + H)]
        else:
            g = [w[min(-i - 1, n - 1)] if i < 0 else (w[max(2 * n - 1 - i, 0)] if i >= n else w[i]) for i in range(-H, n + H)]
        wid.append(torch.tensor(np.array(g), device=dev).reshape([-1 if a == D - 1 - d else 1 for a in range(D)]))
    if transport:
        rk, rw = W[0] * f1, W[0] * f2
    for _ in range(steps):
        P = _pad(W, s)
        rate = sum((torch.abs(W[1 + d] / W[0]) + torch.sqrt(GAMMA * _pressure(W) / W[0])) / _cut(wid[d], D - 1 - d, H, -H)
                   for d in range(D))
        dt = CFL / rate.max()
        U = [P[1 + d] / P[0] for d in range(D)]
        diff = lambda f, d: (_shifted(f, D - 1 - d, 1) - _shifted(f, D - 1 - d, -1)) / (
            0.5 * _shifted(wid[d], D - 1 - d, -1) + wid[d] + 0.5 * _shifted(wid[d], D - 1 - d, 1))
        if model == "none":
            tau_c = torch.zeros_like(P[0])
        else:
            k_, o_ = (_pad_field(rk / W[0], s), _pad_field(rw / W[0], s)) if transport else (_pad_field(f1, s), _pad_field(f2, s))
            grads = [[diff(U[b], d) for b in range(D)] for d in range(D)]
            tau_c = _tau_t("keps" if model == "keps" else "komega", P, k_, o_, grads)

        def slopes(f, d):
            ax = D - 1 - d
            dm = 0.5 * (_shifted(wid[d], ax, -1) + wid[d])
            dp = 0.5 * (_shifted(wid[d], ax, 1) + wid[d])
            return _limit(limiter, (f - _shifted(f, ax, -1)) / dm, (_shifted(f, ax, 1) - f) / dp)

        sl_all = [[slopes(w, d) for w in P] for d in range(D)]
        new = list(W)
        mass = []
        for d in range(D):
            ax = D - 1 - d
            order = [0] + [1 + d] + [1 + e for e in range(D) if e != d] + [D + 1]
            n = W[0].shape[ax]

            def side(f, k, ax=ax, n=n):  # cell of face index 0..n: cell index face - 1 + k, other axes interior
                for a in range(D):
                    f = f.narrow(a, H - 1 + k, n + 1) if a == ax else f.narrow(a, H, f.shape[a] - 2 * H)
                return f

            def wside(k):
                return wid[d].narrow(ax, H - 1 + k, n + 1)

            c = {k: [side(P[v], k) for v in order] for k in ((-2, -1, 0, 1, 2, 3) if recon == "weno5" else (-1, 0, 1, 2))}
            cl, cr = c[0], c[1]
            hl, hr = wside(0), wside(1)
            if recon == "muscl2":
                sl, sr = [side(sl_all[d][v], 0) for v in order], [side(sl_all[d][v], 1) for v in order]
                wl, wr = [a + 0.5 * hl * b for a, b in zip(cl, sl)], [a - 0.5 * hr * b for a, b in zip(cr, sr)]
            else:
                if recon == "muscl3":
                    wl = [_muscl3(x, y, z) for x, y, z in zip(c[-1], c[0], c[1])]
                    wr = [_muscl3(x, y, z) for x, y, z in zip(c[2], c[1], c[0])]
                else:
                    wl = [_weno5(*x) for x in zip(c[-2], c[-1], c[0], c[1], c[2])]
                    wr = [_weno5(*x) for x in zip(c[3], c[2], c[1], c[0], c[-1])]
                sl, sr = [2 * (a - b) / hl for a, b in zip(wl, cl)], [2 * (b - a) / hr for a, b in zip(wr, cr)]
            okl, okr = _physical(wl), _physical(wr)
            wl, sl = [torch.where(okl, a, b) for a, b in zip(wl, cl)], [torch.where(okl, a, 0.0) for a in sl]
            wr, sr = [torch.where(okr, a, b) for a, b in zip(wr, cr)], [torch.where(okr, a, 0.0) for a in sr]
            tl, tr = [], []
            if expand == "multid":
                for e in range(D):
                    if e != d:
                        tl.append([side(sl_all[e][v], 0) for v in order])
                        tr.append([side(sl_all[e][v], 1) for v in order])
            F, _ = _flux(wl, wr, cl, cr, sl, sr, tl, tr, 0.5 * hl, 0.5 * hr, 0.5 * (side(tau_c, 0) + side(tau_c, 1)), dt,
                         mu, C_a)
            h = _cut(wid[d], ax, H, -H)
            for v, f in zip(order, F):
                new[v] = new[v] - (f.narrow(ax, 1, n) - f.narrow(ax, 0, n)) / h
            mass.append((F[0], side, hl, hr, h, ax, n, d))
        if transport:
            rk, rw = _komega_step(P, U, k_, o_, rk, rw, new[0], mass, slopes, diff, dt, mu, D)
        W = new
    return (W, rk / W[0], rw / W[0]) if transport else (W, None, None)


def _komega_step(P, U, k, om, rk, rw, rho_new, mass, slopes, diff, dt, mu, D):
    """Wilcox 2006 k-omega after the flow step (two-dimensional: no vortex stretching)."""
    beta_star, alpha, beta0, sigma, sigma_star, sigma_do, C_lim = 0.09, 13 / 25, 0.0708, 0.5, 0.6, 0.125, 7 / 8
    inner = lambda f: f[tuple(slice(H, -H) for _ in range(D))]
    out = [rk, rw]
    for fr, side, hl, hr, h, ax, n, d in mass:
        rl, rr = side(P[0], 0), side(P[0], 1)
        md = P[0] * k / om
        mface = 0.5 * (side(md, 0) + side(md, 1))
        for q, (f, sg) in enumerate(((k, sigma_star), (om, sigma))):
            s = slopes(f, d)
            a, b = side(f, 0), side(f, 1)
            phil = a + 0.5 * side(s, 0) * (hl - fr / rl)
            phir = b - 0.5 * side(s, 1) * (hr + fr / rr)
            G = fr * torch.where(fr >= 0, phil, phir) - dt * (mu + sg * mface) * (b - a) / (0.5 * hl + 0.5 * hr)
            out[q] = out[q] - (G.narrow(ax, 1, n) - G.narrow(ax, 0, n)) / h
    g = [[inner(diff(U[b], a)) for b in range(D)] for a in range(D)]
    gk, gw = [inner(diff(k, a)) for a in range(D)], [inner(diff(om, a)) for a in range(D)]
    rho, k0, w0 = inner(P[0]), inner(k), inner(om)
    div = sum(g[a][a] for a in range(D))
    Sm = [[0.5 * (g[a][b] + g[b][a]) for b in range(D)] for a in range(D)]
    SS = sum(Sm[a][b] ** 2 for a in range(D) for b in range(D))
    Sb = sum((Sm[a][b] - (div / 3 if a == b else 0.0)) ** 2 for a in range(D) for b in range(D))
    X = 2 * SS - 2 / 3 * div * div
    wt = torch.maximum(w0, C_lim * torch.sqrt(2 * Sb / beta_star))
    cross = sum(a * b for a, b in zip(gk, gw))
    rk = out[0] + dt * (rho * k0 / wt * X - 2 / 3 * rho * k0 * div)
    rw = out[1] + dt * (alpha * rho * w0 / wt * X - 2 / 3 * alpha * rho * w0 * div
                        + torch.where(cross > 0, sigma_do, 0.0) * rho / w0 * cross)
    return torch.clamp(rk / (1 + dt * beta_star * w0), min=0.0), torch.maximum(rw / (1 + dt * beta0 * w0), rho_new * 1e-12)


def _corner_metrics(nodes, dev):
    """Per face along i and j: normal, length, centroid distances of the four-cell stencil, centroid to
    midpoint distances; cell areas.  Ghost centroids mirror through the boundary face midpoint."""
    X = np.asarray(nodes)
    cen = 0.25 * (X[:-1, :-1] + X[:-1, 1:] + X[1:, 1:] + X[1:, :-1])
    d1, d2 = X[1:, 1:] - X[:-1, :-1], X[1:, :-1] - X[:-1, 1:]
    area = 0.5 * (d1[..., 0] * d2[..., 1] - d2[..., 0] * d1[..., 1])
    faces = []
    for a in (0, 1):  # 0: i-faces, 1: j-faces
        if a == 0:
            e, m, ax = X[1:] - X[:-1], 0.5 * (X[1:] + X[:-1]), 1
        else:
            e, m, ax = X[:, 1:] - X[:, :-1], 0.5 * (X[:, 1:] + X[:, :-1]), 0
        L = np.sqrt((e ** 2).sum(-1))
        nrm = np.stack([e[..., 1], -e[..., 0]], -1) / L[..., None] * (1 if a == 0 else -1)
        lo, hi = m.take([0], ax), m.take([-1], ax)
        g = np.concatenate([2 * lo - cen.take([1, 0], ax), cen, 2 * hi - cen.take([-1, -2], ax)], ax)
        n = cen.shape[ax]
        c = [g.take(range(k, k + n + 1), ax) for k in range(4)]
        dist = lambda p, q: np.sqrt(((p - q) ** 2).sum(-1))
        rec = [nrm[..., 0], nrm[..., 1], L, dist(c[0], c[1]), dist(c[1], c[2]), dist(c[2], c[3]), dist(m, c[1]), dist(m, c[2])]
        faces.append([torch.tensor(np.ascontiguousarray(r), device=dev) for r in rec])
    return faces, torch.tensor(area, device=dev)


def _corner_run(case, s, dev):
    faces, area = _corner_metrics(s["nodes"], dev)
    s = dict(s, D=2)
    W = _cons(list(s["prim"]))
    ny, nx = W[0].shape
    ends = lambda f, ax: (f.narrow(ax, 0, f.shape[ax] - 1), f.narrow(ax, 1, f.shape[ax] - 1))
    for _ in range(case["steps"]):
        U = [W[1] / W[0], W[2] / W[0]]
        c = torch.sqrt(GAMMA * _pressure(W) / W[0])
        rate = 0.0
        for ax, rec in ((1, faces[0]), (0, faces[1])):
            for q in (0, 1):
                r = [ends(x, ax)[q] for x in rec[:3]]
                rate = rate + (torch.abs(U[0] * r[0] + U[1] * r[1]) + c) * r[2]
        dt = CFL / (0.5 * rate / area).max()
        line = {1: _pad(W, s, [1]), 0: _pad(W, s, [0])}  # ghosts along one axis at a time
        grads = [[0.0, 0.0], [0.0, 0.0]]
        for ax, rec in ((1, faces[0]), (0, faces[1])):
            P, n = line[ax], W[0].shape[ax]
            for b in range(2):
                u = P[1 + b] / P[0]
                uf = 0.5 * (u.narrow(ax, H - 1, n + 1) + u.narrow(ax, H, n + 1))
                for a in range(2):
                    lo, hi = ends(uf * rec[a] * rec[2], ax)
                    grads[a][b] = grads[a][b] + (hi - lo) / area
        tau_c = _tau_t("komega", W, s["f1"], s["f2"], grads)
        new = list(W)
        for ax, rec in ((1, faces[0]), (0, faces[1])):
            nx_, ny_, L, d01, d12, d23, dl, dr = rec
            P, n = line[ax], W[0].shape[ax]
            st = []
            for k in range(4):
                w = [p.narrow(ax, H - 2 + k, n + 1) for p in P]
                st.append([w[0], w[1] * nx_ + w[2] * ny_, -w[1] * ny_ + w[2] * nx_, w[3]])
            sl = [_limit("vanleer", (b - a) / d01, (c2 - b) / d12) for a, b, c2 in zip(*st[:3])]
            sr = [_limit("vanleer", (b - a) / d12, (c2 - b) / d23) for a, b, c2 in zip(*st[1:])]
            cl, cr = st[1], st[2]
            wl, wr = [a + dl * b for a, b in zip(cl, sl)], [a - dr * b for a, b in zip(cr, sr)]
            okl, okr = _physical(wl), _physical(wr)
            wl, sl = [torch.where(okl, a, b) for a, b in zip(wl, cl)], [torch.where(okl, a, 0.0) for a in sl]
            wr, sr = [torch.where(okr, a, b) for a, b in zip(wr, cr)], [torch.where(okr, a, 0.0) for a in sr]
            t = torch.cat([tau_c.narrow(ax, 0, 1), tau_c, tau_c.narrow(ax, n - 1, 1)], ax)
            t = 0.5 * (t.narrow(ax, 0, n + 1) + t.narrow(ax, 1, n + 1))
            F, _ = _flux(wl, wr, cl, cr, sl, sr, [], [], dl, dr, t, dt, s["mu"], s["C_a"])
            F = [F[0] * L, (F[1] * nx_ - F[2] * ny_) * L, (F[1] * ny_ + F[2] * nx_) * L, F[3] * L]
            for v in range(4):
                lo, hi = ends(F[v], ax)
                new[v] = new[v] - (hi - lo) / area
        W = new
    return W


def _flat(W):
    return torch.stack(W).reshape(-1)


def exact(case, seed):
    f = case["family"]
    dev = torch.device("cuda")
    if f == "steady":
        return None  # hundreds of dependent sweeps and eleven residuals a cycle: minutes in plain torch
    if f == "faces":
        r = _face_records(case, seed, dev)
        D = case["dim"]
        nv = D + 2
        col = lambda o: [r[:, o + v] for v in range(nv)]
        m = case["expand"] == "multid"
        tl = [col((6 + q) * nv) for q in range(D - 1)] if m else []
        tr = [col((6 + D - 1 + q) * nv) for q in range(D - 1)] if m else []
        dt = torch.full_like(r[:, 0], FACES["dt"])
        F, tau = _flux(col(0), col(nv), col(2 * nv), col(3 * nv), col(4 * nv), col(5 * nv), tl, tr, r[:, -3], r[:, -2],
                       r[:, -1], dt, FACES["mu"], FACES["C_a"])
        return {"F": torch.stack(F, 1), "tau": tau}
    if f == "serve":
        out = []
        for q in _requests(case, seed):
            s = dict(prim=torch.tensor(q["prim"], device=dev), f1=None, f2=None, dx=q["dx"], bc=q["bc"], bc_prim=None,
                     T_wall=1.0)
            W, _, _ = _rect_run(dict(dim=q["dim"]), s, dev, q["nsteps"], SERVE["mu"], SERVE["C_a"], "vanleer", "muscl2",
                                "multid", "none")
            out.append(_flat(W))
        return out
    if f == "corner":
        return {"W": _flat(_corner_run(case, _corner_inputs(case, seed, dev), dev))}
    s = _flow_inputs(case, seed, dev)
    W, k, om = _rect_run(case, s, dev, case["steps"], s["mu"], s["C_a"], case["limiter"], case["recon"], case["expand"],
                         case["model"])
    out = {"W": _flat(W)}
    if k is not None:
        out["k"], out["omega"] = k.reshape(-1), om.reshape(-1)
    return out
