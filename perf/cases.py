"""Performance cases of the porous-convection library: the calls a program makes while it solves.

A solve is the same everywhere: create a lattice (or a batch, or a server), set its medium and
its initial fields, then repeat "advance a chunk of time steps, look at the residual and the wall
Nusselt number, read the fields".  Each case is one such chunk through the Python entry points,
over the sizes, storage formats, lattices and boundary sets of this repository's configurations,
tests and benchmark.  Initial fields and porosity fields come from the seed.

`exact` advances the same equations (Liu & He, arXiv:1611.03329) in 64-bit PyTorch, with dense
moment matrices and no code of the library.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1611_03329_gb300 as gb

# ---- the cases -------------------------------------------------------------------------------
# kind "lattice": one lattice.  setup: cavity (halfway walls, hot and cold x faces), channel
# (velocity inlet, convective outflow), melting (enthalpy model), nodes (cavity with the paper's
# node walls).  field: heterogeneous porosity.  monitor: residual and Nusselt number each chunk.


def _lattice(name, setup, nx, ny, nz, steps, storage="fp32", q=19, scheme="pingpong", field=False,
             monitor=False):
    return dict(name=name, kind="lattice", setup=setup, nx=nx, ny=ny, nz=nz, steps=steps,
                storage=storage, q=q, scheme=scheme, field=field, monitor=monitor)


def listed():
    return [
        # the smallest configured solve (32^3 cavity), monitored every 100 steps: launches count
        _lattice("cavity_32", "cavity", 32, 32, 32, 100, monitor=True),
        # a grid-convergence size: odd and ragged extents, in single precision
        _lattice("cavity_63x61x59", "cavity", 63, 61, 59, 100, monitor=True),
        # the benchmark's channel in both storage formats it is run in
        _lattice("channel_256_fp32", "channel", 256, 64, 64, 100),
        _lattice("channel_256_fp16", "channel", 256, 64, 64, 100, storage="fp16"),
        # the precision sweep: heterogeneous cavity, BF16 deviations
        _lattice("field_cavity_128_bf16", "cavity", 128, 128, 128, 50, storage="bf16", field=True,
                 monitor=True),
        # the largest configured solve
        _lattice("field_cavity_256_fp32", "cavity", 256, 256, 256, 20, field=True),
        # one population copy updated in place, chosen where memory is short
        _lattice("cavity_160_aa", "cavity", 160, 160, 160, 40, scheme="aa"),
        # the enthalpy model of solid-liquid phase change
        _lattice("melting_64", "melting", 64, 64, 64, 100, monitor=True),
        # the D3Q15 flow lattice on the benchmark's channel shape
        _lattice("channel_192_d3q15", "channel", 192, 48, 48, 100, q=15),
        # the paper's own node walls (a 64-spacing cavity has 65 sites)
        _lattice("nodes_65", "nodes", 65, 65, 65, 100, monitor=True),
        # the batch configuration: 64 independent cavities of mixed edges
        dict(name="batch_64_cavities", kind="batch", count=64, edges="32,48,64,96,128", pick=2016,
             steps=20),
        # a served stream of small solves, from submission to the final fields on the host
        dict(name="serve_16_small", kind="serve", count=16, edges="16,24,32,40,48", pick=5,
             max_steps=300, chunk=100),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: most are single lattices, some batches and served streams."""
    kind = rng.choice(["lattice"] * 8 + ["batch", "serve"])
    if kind == "batch":
        edges = rng.choice(["32,48,64", "32,48,64,96,128", "24,33,40,57", "64,96,128"])
        return dict(kind="batch", count=_log_int(rng, 4, 64), edges=edges,
                    pick=rng.randrange(1 << 20), steps=rng.randint(10, 20))
    if kind == "serve":
        edges = rng.choice(["16,24,32,40,48", "16,17,31,48", "32,48,64"])
        return dict(kind="serve", count=rng.randint(4, 16), edges=edges,
                    pick=rng.randrange(1 << 20), max_steps=rng.choice([100, 200, 300]),
                    chunk=rng.choice([50, 100]))
    setup = rng.choice(["cavity", "cavity", "channel", "channel", "melting", "nodes"])
    storage, q, scheme, field = "fp32", 19, "pingpong", False
    if setup == "cavity":
        storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
        field = rng.random() < 0.4
        if storage == "fp32" and rng.random() < 0.25:
            scheme = "aa"
    elif setup == "channel":
        storage = rng.choice(["fp32", "fp32", "fp16", "bf16"])
        if storage == "fp32" and rng.random() < 0.3:
            q = 15
    top = {"cavity": 224, "channel": 80, "melting": 128, "nodes": 128}[setup]
    w = _log_int(rng, 24, top)
    shape = rng.choice(["even", "any"])
    if setup == "channel":
        nx, ny, nz = 4 * w, w, w
    elif shape == "even":
        w += w & 1
        nx = ny = nz = w
    else:  # ragged: every extent its own, odd ones among them
        nx, ny, nz = (max(17, w + rng.randint(-7, 7)) for _ in range(3))
    steps = rng.randint(20, 100)
    steps = max(5, min(steps, int(1.5e8 / (nx * ny * nz))))
    return dict(kind="lattice", setup=setup, nx=nx, ny=ny, nz=nz, steps=steps, storage=storage, q=q,
                scheme=scheme, field=field, monitor=rng.random() < 0.5)


# ---- problems --------------------------------------------------------------------------------
_COLLIDE_FLOPS = {19: 460, 15: 400}  # flow and temperature collision of one site


def _problem(case):
    """The problem dictionary of a lattice case (no porosity field yet)."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    pb = dict(nx=nx, ny=ny, nz=nz, storage=case["storage"], q=case["q"], scheme=case["scheme"],
              T0=0.5)
    if case["setup"] == "channel":
        pb.update(mapping="channel", Re=10.0, u0=0.01, Pr=0.71, Ri=1.0, Da=1e-3, phi=0.7, F_phi=-1.0,
                  flow_bc=[2, 3, 1, 1, 0, 0], heat_bc=[2, 3, 2, 2, 0, 0],
                  face_T=[0.0, 0.0, 0.0, 1.0, 0.0, 0.0],
                  face_u=[(0.01, 0.0, 0.0)] + [(0.0, 0.0, 0.0)] * 5, T_init=0.0,
                  gravity_axis=1, gravity_sign=-1)
        return pb
    pb.update(mapping="cavity", Ra=1e5, Da=1e-2, Pr=0.71, phi=0.6, F_phi=-1.0, L=float(nx),
              flow_bc=[1] * 6, heat_bc=[2, 2, 1, 1, 1, 1], face_T=[1.0, 0.0, 0.0, 0.0, 0.0, 0.0],
              T_init=0.5, gravity_axis=2, gravity_sign=-1)
    if case["setup"] == "melting":
        pb.update(Da=None, phi=1.0, F_phi=0.0, enthalpy=True, T_m=0.5, St=1.0, T_init=0.0)
    if case["setup"] == "nodes":
        pb.update(L=float(nx - 1), flow_bc=[4] * 6, heat_bc=[4, 4, 5, 5, 5, 5])
    return pb


def _generator(seed):
    g = torch.Generator(device=_dev())
    g.manual_seed(int(seed))
    return g


def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _smooth(shape, gen, modes=3):
    """A smooth random field of unit size: a few sine products with random factors and phases."""
    out = torch.zeros(shape, dtype=torch.float64, device=_dev())
    r = torch.rand((modes, 7), generator=gen, device=_dev(), dtype=torch.float64).cpu()
    for m in range(modes):
        parts = []
        for a in range(3):
            x = (torch.arange(shape[a], dtype=torch.float64, device=_dev()) + 0.5) / shape[a]
            k = 1 + int(3 * float(r[m, 2 * a]))
            sh = [1, 1, 1]
            sh[a] = shape[a]
            parts.append(torch.sin(math.pi * k * x + 2 * math.pi * float(r[m, 2 * a + 1])).reshape(sh))
        out += (2 * float(r[m, 6]) - 1) * parts[0] * parts[1] * parts[2]
    return out


def _initial(pb, case_setup, gen):
    """Initial temperature and velocity (host, FP64): the problem's own state, disturbed."""
    shape = (pb["nz"], pb["ny"], pb["nx"])
    if case_setup == "melting":
        T = (0.5 + 0.4 * _smooth(shape, gen)).clamp(0.0, 1.0)
    else:
        T = (pb["T_init"] + 0.1 * _smooth(shape, gen)).clamp(0.0, 1.0)
    u = torch.stack([0.004 * _smooth(shape, gen) for _ in range(3)])
    if case_setup == "melting":
        u.zero_()
    return T.cpu().numpy(), u.cpu().numpy()


def _porosity(shape, gen):
    """Gaussian random porosity: mean 0.6, std 0.05, clipped to [0.4, 0.9], correlated over L/16."""
    w = torch.randn(shape, generator=gen, device=_dev(), dtype=torch.float64)
    f = torch.fft.fftn(w)
    for a, n in enumerate(shape):
        k = torch.fft.fftfreq(n, device=_dev(), dtype=torch.float64)
        sh = [1, 1, 1]
        sh[a] = n
        f = f * torch.exp(-0.5 * (2 * math.pi * k * max(shape) / 16.0) ** 2).reshape(sh)
    f = torch.fft.ifftn(f).real
    f = (f - f.mean()) / f.std()
    return (0.6 + 0.05 * f).clamp(0.4, 0.9).float().cpu().numpy()


def _lattice_inputs(case, seed):
    gen = _generator(seed)
    pb = _problem(case)
    if case["field"]:
        pb["phi_field"] = _porosity((pb["nz"], pb["ny"], pb["nx"]), gen)
    T, u = _initial(pb, case["setup"], gen)
    return pb, T, u


def _many(case, seed, served):
    """The problems of a batch or a served stream: sizes from the case, physics from the seed."""
    pick = np.random.Generator(np.random.PCG64(case["pick"]))
    edges = [int(e) for e in case["edges"].split(",")]
    rng = np.random.Generator(np.random.PCG64(seed))
    out = []
    for k in range(case["count"]):
        n = int(pick.choice(edges))
        kind = float(pick.uniform())
        base = dict(setup="cavity", nx=n, ny=n, nz=n, storage="fp32", q=19, scheme="pingpong",
                    field=False)
        if served and kind < 0.1:
            base["setup"] = "melting"
        elif served and kind < 0.4:
            base.update(setup="channel", nx=2 * n, ny=max(16, n // 2), nz=max(16, n // 2))
        pb = _problem(base)
        if base["setup"] == "cavity":
            pb.update(phi=float(rng.uniform(0.4, 0.9)), Da=float(10 ** rng.uniform(-5, -1)),
                      Ra=float(10 ** rng.uniform(3, 6)))
        elif base["setup"] == "channel":
            pb["Da"] = float(10 ** rng.uniform(-3, -2))
        else:
            pb["Ra"] = float(10 ** rng.uniform(4, 6))
        out.append(pb)
    return out


def _sites(pb):
    return pb["nx"] * pb["ny"] * pb["nz"]


# ---- what a program has, and one pass of it --------------------------------------------------
def prepare(case, seed):
    if case["kind"] == "serve":
        # the server is created once by a program and kept; its requests are host data
        stream = torch.cuda.Stream()
        pbs = _many(case, seed, True)
        n = sum(_sites(p) for p in pbs)
        return dict(case=case, stream=stream, pbs=pbs,
                    server=gb.Server(chunk=case["chunk"], stream=stream.cuda_stream),
                    u=np.zeros(3 * n, np.float32), T=np.zeros(n, np.float32))
    stream = torch.cuda.Stream()
    if case["kind"] == "batch":
        pbs = _many(case, seed, False)
        lats = []
        gen = _generator(seed)
        for pb in pbs:
            lat = gb.Lattice(pb, stream=stream.cuda_stream)
            T, u = _initial(pb, "cavity", gen)
            lat.init_equilibrium(T_field=T, u_field=u)
            lats.append(lat)
        batch = gb.Batch(lats, stream=stream.cuda_stream)
        n = sum(_sites(p) for p in pbs)
        state = dict(case=case, stream=stream, lats=lats, batch=batch)
    else:
        pb, T, u = _lattice_inputs(case, seed)
        lat = gb.Lattice(pb, stream=stream.cuda_stream)
        lat.init_equilibrium(T_field=T, u_field=u)
        if case["monitor"]:
            lat.residual()  # the snapshot that the first chunk is compared with
        n = _sites(pb)
        state = dict(case=case, stream=stream, lats=[lat])
    with torch.cuda.stream(stream):
        state.update(rho=torch.empty(n, device="cuda"), u=torch.empty(3 * n, device="cuda"),
                     T=torch.empty(n, device="cuda"))
    return state


def _monitored(case):
    """Whether the wall Nusselt number is read too: on the D3Q19 halfway-wall problems."""
    return case["q"] == 19 and case["setup"] != "nodes"


def _face(case):
    return 3 if case["setup"] == "channel" else 0  # the hot wall


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        return _serve(state)
    out = {}
    if case["kind"] == "batch":
        state["batch"].step(case["steps"])
    else:
        lat = state["lats"][0]
        lat.step(case["steps"])
        if case["monitor"]:
            out["r_u"], out["r_T"] = lat.residual()
            if _monitored(case):
                out["nu"], out["nu_profile"], out["nu_mp"] = lat.nusselt(_face(case))
    at = 0
    for lat in state["lats"]:
        lat.macros_device(state["rho"].data_ptr() + 4 * at, state["u"].data_ptr() + 12 * at,
                          state["T"].data_ptr() + 4 * at)
        at += lat.ns
    out.update(rho=state["rho"], u=state["u"], T=state["T"])
    return out


def _serve(state):
    srv, case = state["server"], state["case"]
    at, ids = 0, []
    for pb in state["pbs"]:
        rid = srv.submit(pb, tol=1e-4, max_steps=case["max_steps"])
        n = _sites(pb)
        srv.set_output(rid, state["u"][3 * at:3 * (at + n)], state["T"][at:at + n])
        at += n
        ids.append(rid)
    while sum(srv.advance()) > 0:
        pass
    res = {r["id"]: r for r in srv.poll()}
    rows = [res[i] for i in ids]
    return dict(steps=np.array([r["steps"] for r in rows]), u=state["u"], T=state["T"],
                nu=np.array([r["nu_avg"] for r in rows], np.float32))


def work(case):
    """Bytes and operations of one pass.  A time step reads the populations of the previous one
    and writes its own (the unit of the lattice Boltzmann method's roofline: 208 bytes a site on
    D3Q19 + D3Q7 in FP32); the fields read out at the end are written once."""
    if case["kind"] == "lattice":
        n = case["nx"] * case["ny"] * case["nz"]
        elem = 4 if case["storage"] == "fp32" else 2
        step = 2 * (case["q"] + 7) * elem + (8 if elem == 2 else 0) + (4 if case["field"] else 0)
        fields = (case["q"] + 7) * elem + 20 + (4 if case["field"] else 0)
        return dict(bytes=n * (case["steps"] * step + fields),
                    flops=n * case["steps"] * _COLLIDE_FLOPS[case["q"]])
    n = sum(_sites(pb) for pb in _many(case, 0, case["kind"] == "serve"))
    steps = case["steps"] if case["kind"] == "batch" else case["max_steps"]
    return dict(bytes=n * (208 * steps + 124), flops=n * steps * _COLLIDE_FLOPS[19])


# ---- the same in 64 bits ---------------------------------------------------------------------
_E19 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1),
        (1, 1, 0), (-1, 1, 0), (1, -1, 0), (-1, -1, 0), (1, 0, 1), (-1, 0, 1), (1, 0, -1),
        (-1, 0, -1), (0, 1, 1), (0, -1, 1), (0, 1, -1), (0, -1, -1)]
_E15 = _E19[:7] + [(x, y, z) for z in (1, -1) for y in (1, -1) for x in (1, -1)]


def _moment_rows(q, e):
    """The orthogonal moment basis of Eqs. A1 / A2 as polynomials of the velocities."""
    x, y, z = (np.array([v[a] for v in e], float) for a in range(3))
    c2 = x * x + y * y + z * z
    one = np.ones(q)
    if q == 19:
        return np.stack([one, 19 * c2 - 30, (21 * c2 * c2 - 53 * c2 + 24) / 2,
                         x, (5 * c2 - 9) * x, y, (5 * c2 - 9) * y, z, (5 * c2 - 9) * z,
                         3 * x * x - c2, (3 * c2 - 5) * (3 * x * x - c2),
                         y * y - z * z, (3 * c2 - 5) * (y * y - z * z),
                         x * y, y * z, z * x,
                         (y * y - z * z) * x, (z * z - x * x) * y, (x * x - y * y) * z])
    return np.stack([one, c2 - 2, (15 * c2 * c2 - 55 * c2 + 32) / 2,
                     x, (5 * c2 - 13) * x / 2, y, (5 * c2 - 13) * y / 2, z, (5 * c2 - 13) * z / 2,
                     3 * x * x - c2, y * y - z * z, x * y, y * z, z * x, x * y * z])


class _Exact:
    """One lattice in FP64: dense moment matrices, streaming by shifts, faces on their slabs."""

    def __init__(self, pb, T, u):
        self.pb, q = pb, pb["q"]
        dev = _dev()
        f8 = dict(dtype=torch.float64, device=dev)
        self.e = _E19 if q == 19 else _E15
        self.w = ([1 / 3] + [1 / 18] * 6 + [1 / 36] * 12) if q == 19 else ([2 / 9] + [1 / 9] * 6 + [1 / 72] * 8)
        self.opp = [self.e.index(tuple(-c for c in v)) for v in self.e]
        M = _moment_rows(q, self.e)
        self.M = torch.tensor(M, **f8)
        self.Mi = torch.tensor(np.linalg.inv(M), **f8)
        N = np.array([[1] * 7, [0, 1, -1, 0, 0, 0, 0], [0, 0, 0, 1, -1, 0, 0], [0, 0, 0, 0, 0, 1, -1],
                      [0, 1, 1, 1, 1, 1, 1], [0, 1, 1, -1, -1, 0, 0], [0, 1, 1, 0, 0, -1, -1]], float)
        self.N, self.Ni = torch.tensor(N, **f8), torch.tensor(np.linalg.inv(N), **f8)
        self.shape = (pb["nz"], pb["ny"], pb["nx"])
        self.ns = _sites(pb)
        # lattice units: Eq. 56 (cavity) or Eq. 51 (channel), Eqs. 7, 32, 41
        L = float(pb.get("L") or (pb["ny"] if pb["mapping"] == "channel" else pb["nx"]))
        if pb["mapping"] == "channel":
            nu, gbeta = L * pb["u0"] / pb["Re"], pb["Ri"] * pb["u0"] ** 2 / L
        else:
            nu = 0.1 * L * math.sqrt(3 * pb["Pr"]) / math.sqrt(pb["Ra"]) / 3
            gbeta = 0.01 / 3 / L
        self.nu, self.L = nu, L
        snu = 1 / (0.5 + 3 * nu)
        s = ([1, 1.1, 1.1, 1, 1.1, 1, 1.1, 1, 1.1, snu, 1.1, snu, 1.1, snu, snu, snu, 1.2, 1.2, 1.2]
             if q == 19 else [1, 1.1, 1.1, 1, 1.1, 1, 1.1, 1, 1.1] + [snu] * 5 + [1.2])
        self.s = torch.tensor(s, **f8)[:, None]
        self.alpha = nu / pb["Pr"]
        self.buoy = [0.0, 0.0, 0.0]
        self.buoy[pb["gravity_axis"]] = -pb["gravity_sign"] * gbeta
        # medium: Eq. 6 (Kozeny-Carman K around the mean porosity, Ergun's F_phi)
        K = pb["Da"] * L * L if pb["Da"] else math.inf
        if pb.get("phi_field") is not None:
            p = torch.tensor(pb["phi_field"], **f8).reshape(-1)
            pm = float(p.mean())
            K = K * (p ** 3 / (1 - p) ** 2) / (pm ** 3 / (1 - pm) ** 2)
            self.phi = p
        else:
            self.phi = torch.full((1,), pb["phi"], **f8)
            K = torch.full((1,), K, **f8)
        F = 1.75 / torch.sqrt(150 * self.phi ** 3) if pb["F_phi"] < 0 else pb["F_phi"]
        self.cd, self.cf = self.phi * nu / K, self.phi * F / torch.sqrt(K)
        self.melt = bool(pb.get("enthalpy"))
        # the layer of node-wall sites: its site, the fluid site beside it, its face temperature
        self.wall = None
        if 4 in pb["flow_bc"]:
            c = [t.reshape(-1) for t in torch.meshgrid(*[torch.arange(n, device=dev) for n in self.shape],
                                                       indexing="ij")][::-1]
            nx, ny, nz = pb["nx"], pb["ny"], pb["nz"]
            on = torch.zeros(self.ns, dtype=torch.bool, device=dev)
            cf, Tw = [t.clone() for t in c], torch.full((self.ns,), math.nan, **f8)
            for f in range(5, -1, -1):
                at = c[f // 2] == (0 if f % 2 == 0 else (nx, ny, nz)[f // 2] - 1)
                on |= at
                cf[f // 2] = cf[f // 2] + at.long() * (1 if f % 2 == 0 else -1)
                if pb["heat_bc"][f] == 4:
                    Tw = torch.where(at, torch.full_like(Tw, pb["face_T"][f]), Tw)
            idx = on.nonzero().reshape(-1)
            self.wall = (idx, (cf[0] + nx * (cf[1] + ny * cf[2]))[idx], Tw[idx])
        T, u = torch.tensor(T, **f8).reshape(-1), torch.tensor(u, **f8).reshape(3, -1)
        self.f = self.feq(torch.ones(self.ns, **f8), u)
        if self.melt:  # phase-pure enthalpy: solid at or below the melting point
            En = torch.where(T <= 0.5, T, T + 1.0)
            self.g = self.geq(T, u, En)
        else:
            self.g = self.geq(T, u)
        self.hist = None
        if pb["flow_bc"][1] == 3:
            self.hist = {i: self.grid(self.f)[i][:, :, -1].clone() for i in range(q) if self.e[i][0] == -1}
            self.hist["g"] = self.grid(self.g)[2][:, :, -1].clone()

    def grid(self, a):
        return a.reshape((a.shape[0],) + self.shape)

    def feq(self, rho, u, phi=None):
        phi = self.phi if phi is None else phi
        uu = (u * u).sum(0)
        out = []
        for w, e in zip(self.w, self.e):
            eu = e[0] * u[0] + e[1] * u[1] + e[2] * u[2]
            out.append(w * (rho + 3 * eu + (4.5 * eu * eu - 1.5 * uu) / phi))
        return torch.stack(out)

    def geq(self, T, u, En=None):  # varpi = 1/2, sigma = 1
        g0 = 0.5 * T if En is None else En - 0.5 * T
        return torch.stack([g0] + [T / 12 + 0.5 * T * (e[0] * u[0] + e[1] * u[1] + e[2] * u[2])
                                   for e in _E19[1:7]])

    def pulled(self, keep):
        """Streamed populations of every site (Eqs. 10, 35 with the face rules)."""
        pb, U = self.pb, 0.01
        F, G = self.grid(self.f), self.grid(self.g)
        f, g, hist = torch.empty_like(F), torch.empty_like(G), {}

        def slabs(e):
            for a in range(3):
                if e[a]:
                    face = 2 * a + (0 if e[a] == 1 else 1)
                    if pb["flow_bc"][face] not in (0, 4):
                        sl = [slice(None)] * 3
                        sl[2 - a] = slice(0, 1) if e[a] == 1 else slice(-1, None)
                        yield face, tuple(sl)

        for i, e in enumerate(self.e):
            f[i] = torch.roll(F[i], (e[2], e[1], e[0]), (0, 1, 2))
            here = F[self.opp[i]]
            cut = list(slabs(e))
            order = {3: 0, 2: 1, 1: 2}  # a later rule wins: outflow, velocity face, wall
            for face, sl in sorted(cut, key=lambda t: order[pb["flow_bc"][t[0]]]):
                kind = pb["flow_bc"][face]
                if kind == 3:
                    inner = torch.roll(F[i], (e[2], e[1]), (0, 1))[sl]
                    f[i][sl] = (self.hist[i].unsqueeze(2) + U * inner) / (1 + U)
                else:
                    uw = pb["face_u"][face] if kind == 2 else (0, 0, 0)
                    f[i][sl] = here[sl] + 6 * self.w[i] * sum(a * b for a, b in zip(e, uw))
        if self.hist is not None:
            # the outlet's density is anchored to 1 through the populations the outflow set
            col = f[:, :, :, -1]
            via = torch.zeros_like(col)
            for i, e in enumerate(self.e):
                if e[0] == -1:
                    y = torch.arange(self.shape[1], device=col.device)
                    ok = torch.ones_like(y, dtype=torch.bool)
                    if e[1] and pb["flow_bc"][2 if e[1] == 1 else 3] != 0:
                        ok = y != (0 if e[1] == 1 else self.shape[1] - 1)
                    via[i] = self.w[i] * ok[None, :]
            col += via * (1 - col.sum(0)) / via.sum(0)
            hist = {i: col[i].clone() for i, e in enumerate(self.e) if e[0] == -1}
        for i, e in enumerate(_E19[:7]):
            g[i] = torch.roll(G[i], (e[2], e[1], e[0]), (0, 1, 2))
            here = G[self.opp[i]]
            for face, sl in slabs(e):
                kind = pb["heat_bc"][face]
                if kind == 3:
                    g[i][sl] = (self.hist["g"].unsqueeze(2) + U * G[i][sl]) / (1 + U)
                    hist["g"] = g[i][sl][:, :, 0].clone()
                else:
                    g[i][sl] = here[sl] if kind == 1 else pb["face_T"][face] / 6 - here[sl]
        if keep and self.hist is not None:
            self.hist = hist
        return f.reshape(len(self.e), -1), g.reshape(7, -1)

    def temperature(self, g):
        n = g.sum(0)
        if not self.melt:
            return n, torch.ones_like(n), n
        return torch.where(n <= 0.5, n, torch.where(n >= 1.5, n - 1.0, torch.full_like(n, 0.5))), \
            (n - 0.5).clamp(0, 1), n

    def medium(self, at):
        return (t if t.numel() == 1 else t[at] for t in (self.phi, self.cd, self.cf))

    def state(self, f, g, at):
        """rho, u, T, body force, liquid fraction and enthalpy (Eqs. 5, 25, 27-28, 39, B8-B9)."""
        phi, cd, cf = self.medium(at)
        T, fl, En = self.temperature(g)
        G = torch.stack([b * (T - 0.5) for b in self.buoy])
        e = torch.tensor(self.e, dtype=torch.float64, device=f.device).T
        v = e @ f + 0.5 * phi * G
        l0, l1 = 0.5 + 0.25 * cd, 0.5 * cf
        u = v / (l0 + torch.sqrt(l0 * l0 + l1 * v.norm(dim=0)))
        if self.melt:
            u = u * (fl >= 0.5)
        return f.sum(0), u, T, G, fl, En

    def collide(self, f, g, at, wall_u=None):
        phi, cd, cf = self.medium(at)
        rho, u, T, G, fl, En = self.state(f, g, at)
        if wall_u is not None:
            u = wall_u
        F = phi * G - (cd + cf * u.norm(dim=0)) * u
        uF, q = (u * F).sum(0), len(self.e)
        c = 2 / 3 if q == 19 else 7 / 3
        z = torch.zeros_like(rho)
        a = 2 * u[0] * F[0] - u[1] * F[1] - u[2] * F[2]
        b = u[1] * F[1] - u[2] * F[2]
        mixed = [(u[0] * F[1] + u[1] * F[0]) / phi, (u[1] * F[2] + u[2] * F[1]) / phi,
                 (u[0] * F[2] + u[2] * F[0]) / phi]
        flux = [F[0], -c * F[0], F[1], -c * F[1], F[2], -c * F[2]]
        if q == 19:  # Eq. 23
            S = [z, 38 * uF / phi, -11 * uF / phi] + flux + [2 * a / phi, -a / phi, 2 * b / phi, -b / phi] \
                + mixed + [z, z, z]
        else:  # Eq. 17
            S = [z, 2 * uF / phi, -10 * uF / phi] + flux + [2 * a / phi, 2 * b / phi] + mixed + [z]
        m, meq = self.M @ f, self.M @ self.feq(rho, u, phi)
        fo = self.Mi @ (m - self.s * (m - meq) + (1 - 0.5 * self.s) * torch.stack(S))
        if self.melt:  # the solid rests
            fo = torch.where(fl >= 0.5, fo, torch.tensor(self.w, dtype=torch.float64, device=f.device)[:, None] * rho)
        za = 1 / (0.5 + 6 * self.alpha)
        n = self.N @ g
        neq = torch.stack([En, T * u[0], T * u[1], T * u[2], 0.5 * T, z, z])
        zeta = torch.tensor([1, za, za, za, 1.2, 1.2, 1.2], dtype=torch.float64, device=f.device)[:, None]
        return fo, self.Ni @ (n - zeta * (n - neq))

    def node(self, f, g, full):
        """Node-wall sites by non-equilibrium extrapolation from the fluid site beside them."""
        idx, beside, Tw = self.wall
        ff, gg = f[:, beside], g[:, beside]
        rho, u, T, _, _, _ = self.state(ff, gg, beside)
        T_b = torch.where(torch.isnan(Tw), T, Tw)
        rest = torch.zeros_like(u)
        pb_, pf_ = list(self.medium(idx))[0], list(self.medium(beside))[0]
        fb = ff + self.feq(rho, rest, pb_) - self.feq(rho, u, pf_)
        gb_ = gg + self.geq(T_b, rest) - self.geq(T, u)
        if not full:
            return rho, rest, T_b
        return self.collide(fb, gb_, idx, wall_u=rest)

    def step(self):
        f, g = self.pulled(True)
        for lo in range(0, self.ns, 1 << 21):
            at = slice(lo, min(self.ns, lo + (1 << 21)))
            self.f[:, at], self.g[:, at] = self.collide(f[:, at], g[:, at], at)
        if self.wall is not None:
            self.f[:, self.wall[0]], self.g[:, self.wall[0]] = self.node(f, g, True)

    def fields(self):
        f, g = self.pulled(False)
        rho, u, T = (torch.empty(n, self.ns, dtype=torch.float64, device=f.device) for n in (1, 3, 1))
        for lo in range(0, self.ns, 1 << 21):
            at = slice(lo, min(self.ns, lo + (1 << 21)))
            rho[0, at], u[:, at], T[0, at] = self.state(f[:, at], g[:, at], at)[:3]
        if self.wall is not None:
            i = self.wall[0]
            rho[0, i], u[:, i], T[0, i] = self.node(f, g, False)
        return rho[0], u, T[0]

    def nusselt(self, T, face):
        """Eqs. 53-55 on a fixed-temperature halfway wall: mean, profile, centre value."""
        a, hi = face // 2, face % 2
        T = T.reshape(self.shape).movedim(2 - a, 0)
        T0, T1 = (T[-1], T[-2]) if hi else (T[0], T[1])
        p = (self.L * (8 * self.pb["face_T"][face] - 9 * T0 + T1) / 3)
        p = p.mean(0) if a != 2 else p.mean(0)  # over z for x and y faces, over y for z faces
        n = p.numel()
        return float(p.mean()), p.cpu().numpy(), float(p[n // 2] if n % 2 else (p[n // 2 - 1] + p[n // 2]) / 2)


def _change(a, b):
    return float((a - b).norm() / a.norm()) if float(a.norm()) > 0 else 0.0


def exact(case, seed):
    if case["kind"] == "lattice":
        sim = _Exact(*_lattice_inputs(case, seed))
        before = sim.fields() if case["monitor"] else None
        for _ in range(case["steps"]):
            sim.step()
        rho, u, T = sim.fields()
        out = {}
        if case["monitor"]:
            out["r_u"], out["r_T"] = _change(u, before[1]), _change(T, before[2])
            if _monitored(case):
                out["nu"], out["nu_profile"], out["nu_mp"] = sim.nusselt(T, _face(case))
        out.update(rho=rho, u=u.reshape(-1), T=T)
        return out
    us, Ts, rhos, nus = [], [], [], []
    gen = _generator(seed)
    for pb in _many(case, seed, case["kind"] == "serve"):
        if case["kind"] == "batch":
            sim = _Exact(pb, *_initial(pb, "cavity", gen))
            for _ in range(case["steps"]):
                sim.step()
            rho, u, T = sim.fields()
            rhos.append(rho)
        else:  # from rest, chunk by chunk, to the tolerance or the step limit
            shape = (pb["nz"], pb["ny"], pb["nx"])
            sim = _Exact(pb, np.full(shape, pb["T_init"]), np.zeros((3,) + shape))
            done, old = 0, None
            while True:
                for _ in range(case["chunk"]):
                    sim.step()
                done += case["chunk"]
                rho, u, T = sim.fields()
                if old and _change(u, old[0]) < 1e-4 and _change(T, old[1]) < 1e-4:
                    break
                if done >= case["max_steps"]:
                    break
                old = (u, T)
            nus.append(sim.nusselt(T, 0)[0])
        us.append(u.reshape(-1))
        Ts.append(T)
    u, T = torch.cat(us), torch.cat(Ts)
    if case["kind"] == "batch":
        return dict(rho=torch.cat(rhos), u=u, T=T)
    return dict(steps=None, u=u.cpu().numpy(), T=T.cpu().numpy(), nu=np.array(nus))
