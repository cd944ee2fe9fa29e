"""Performance cases: what a user of this library has it do, through its public calls.

A case is one solve (or one pool of solves) that is already set up; a pass advances it by
`steps` time steps and reads the result back, the way a program alternates between
stepping and looking.  The families cover the library's paths:

  box      periodic box with 1 % obstacles (the throughput workload), any storage type
  channel  channel between resting walls driven by a body force, the FP64 parity mode
  duct     square duct with a fixed sphere whose drag is read back (wall links, body sums)
  sediment closed box with a sphere sinking in it (particle update, fill/drain)
  mixed    ragged box with obstacles, closed in y, a moving lid: odd sizes, tracked wall
  law      another constitutive law or finite-volume variant in a box with obstacles
  noalloc  caller-owned device buffers (lbve_step_noalloc)
  cavity2d / mill2d   the two-dimensional path (lid-driven cavity, four-roll mill)
  pool     a serving mix stepped together, with the residuals the server looks at

`exact` evaluates the same steps from the method's equations in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

from paper_2009_12279_gb300 import lbve, serve, workloads

# ---------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------


def listed():
    return [
        # a start-up curve of the analytic channel: 512 cells, nothing but launch latency
        {"name": "channel_f64", "family": "channel", "nx": 4, "ny": 32, "nz": 4, "precision": "f64", "steps": 100},
        # a small box owned by a host framework that allows no device allocation
        {"name": "noalloc_f32", "family": "noalloc", "nx": 32, "ny": 32, "nz": 32, "precision": "f32", "steps": 10},
        # the paper's cavity (194^2 fluid cells) between two looks at its fields
        {"name": "cavity2d_f32", "family": "cavity2d", "nx": 194, "precision": "f32", "steps": 100},
        # a ragged mid-size domain with a moving lid and its drag
        {"name": "mixed_f32", "family": "mixed", "nx": 83, "ny": 57, "nz": 45, "precision": "f32", "steps": 40},
        # the fixed-sphere duct: drag history
        {"name": "duct128_f32", "family": "duct", "nx": 128, "precision": "f32", "steps": 20},
        # the sedimentation column: particle position and velocity history
        {"name": "sediment_f32", "family": "sediment", "nx": 64, "ny": 64, "nz": 256, "radius": 8.0,
         "precision": "f32", "steps": 40},
        # the headline throughput box
        {"name": "box512_f32", "family": "box", "nx": 512, "ny": 512, "nz": 512, "precision": "f32", "steps": 8},
        # the same in 16-bit storage at a size that is run more often
        {"name": "box256_bf16", "family": "box", "nx": 256, "ny": 256, "nz": 256, "precision": "bf16", "steps": 20},
        # Giesekus fluid with the transverse-overlap fluxes
        {"name": "giesekus_f32", "family": "law", "nx": 192, "ny": 160, "nz": 96, "precision": "f32",
         "law": "giesekus", "steps": 20},
        # FENE-P fluid
        {"name": "fene_f32", "family": "law", "nx": 100, "ny": 84, "nz": 60, "precision": "f32", "law": "fene",
         "steps": 20},
        # FP64 as a reference solution of a box
        {"name": "box_f64", "family": "box", "nx": 96, "ny": 80, "nz": 72, "precision": "f64", "steps": 10},
        # the server's pool between two looks at its residuals
        {"name": "pool48_bf16", "family": "pool", "members": 48, "mix": 0, "precision": "bf16", "steps": 25},
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    family = rng.choice(["box", "box", "box", "channel", "duct", "sediment", "mixed", "law", "noalloc", "cavity2d",
                         "mill2d", "pool"])
    reduced = rng.choice(["f32", "f32", "bf16", "f16"])
    steps = rng.randint(5, 40)
    if family == "box":
        # half of them with rows of whole 32-cell warps, half of any width
        nx = 32 * rng.randint(1, 16) if rng.random() < 0.5 else _side(rng, 17, 500)
        ny, nz = _side(rng, 15, 400), _side(rng, 15, 400)
        prec = rng.choice(["f32", "f32", "bf16", "f16", "f64"])
        if prec == "f64":
            nx, ny, nz = max(17, nx // 4), max(15, ny // 4), max(15, nz // 4)
        return {"family": family, "nx": nx, "ny": ny, "nz": nz, "precision": prec,
                "steps": min(steps, max(3, int(8 * 512 ** 3 / (nx * ny * nz * 2))))}
    if family == "channel":
        return {"family": family, "nx": rng.randint(3, 20), "ny": _side(rng, 18, 160), "nz": rng.randint(3, 20),
                "precision": rng.choice(["f64", reduced]), "steps": rng.randint(20, 200)}
    if family == "duct":
        return {"family": family, "nx": _side(rng, 24, 160), "precision": reduced, "steps": steps}
    if family == "sediment":
        r = round(rng.uniform(2.6, 9.0), 2)
        w = rng.randint(int(4 * r) + 10, 80)
        return {"family": family, "nx": w, "ny": w + rng.randint(0, 7), "nz": rng.randint(60, 200), "radius": r,
                "precision": reduced, "steps": steps}
    if family == "mixed":
        return {"family": family, "nx": _side(rng, 9, 200), "ny": _side(rng, 9, 150), "nz": _side(rng, 9, 150),
                "precision": rng.choice([reduced, "f64"]) if rng.random() < 0.3 else reduced, "steps": steps}
    if family == "law":
        return {"family": family, "nx": _side(rng, 20, 260), "ny": _side(rng, 16, 160), "nz": _side(rng, 16, 120),
                "precision": reduced, "law": rng.choice(["giesekus", "fene", "ctu", "divu"]), "steps": steps}
    if family == "noalloc":
        return {"family": family, "nx": _side(rng, 8, 80), "ny": _side(rng, 8, 80), "nz": _side(rng, 8, 80),
                "precision": reduced, "steps": 2 * rng.randint(1, 15)}
    if family in ("cavity2d", "mill2d"):
        return {"family": family, "nx": _side(rng, 30, 1000), "precision": rng.choice(["f32", "f32", "f64"]),
                "steps": rng.randint(10, 100)}
    return {"family": "pool", "members": rng.randint(3, 48), "mix": rng.randint(0, 10 ** 6), "precision": reduced,
            "steps": rng.randint(5, 30)}


# ---------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------
DEVICE = "cuda"


def _shape(case):
    f = case["family"]
    if f == "duct":
        return (case["nx"],) * 3
    return (case["nx"], case["ny"], case["nz"])


def _rng(seed):
    g = torch.Generator(device=DEVICE)
    g.manual_seed(int(seed))
    return g


def _uniform(g, shape, amplitude):
    return (torch.rand(shape, generator=g, device=DEVICE, dtype=torch.float64) * 2.0 - 1.0) * amplitude


def _obstacles(g, grid, fraction):
    return (torch.rand(grid, generator=g, device=DEVICE) < fraction).to(torch.uint8)


def _inputs(case, seed):
    """Geometry, parameters and initial fields of a three-dimensional case."""
    f = case["family"]
    nx, ny, nz = shape = _shape(case)
    grid = (nz, ny, nx)
    g = _rng(seed)
    i = {"shape": shape, "wall_vel": [], "particle": None, "rho": None, "tau": None}
    prm = dict(periodic=(1, 1, 1), eta=1.0 / 6.0, beta=0.5, lambda_p=1000.0, rho0=1.0, body_force=(0.0, 0.0, 0.0))
    if f == "box":
        i["flags"] = _obstacles(g, grid, 0.01)
        i["u"] = _uniform(g, (3,) + grid, 1e-3)
    elif f == "channel":
        i["flags"] = torch.from_numpy(workloads.channel_flags(shape, 1)).to(DEVICE)
        prm.update(periodic=(1, 0, 1), lambda_p=3000.0, body_force=(1e-6, 0.0, 0.0))
        i["u"] = _uniform(g, (3,) + grid, 1e-4)
    elif f == "duct":
        c = workloads.config_sphere_duct(nx, radius=12.0 * nx / 128.0)
        i["flags"] = torch.from_numpy(c["flags"]).to(DEVICE)
        i["wall_vel"] = c["wall_vel"]
        prm = dict(c["params"], lambda_p=max(c["params"]["lambda_p"], 10.0))
        i["u"] = _uniform(g, (3,) + grid, 1e-4)
    elif f == "sediment":
        # a light sphere that sinks at its Stokes velocity, Re = 0.1, in a closed box
        R, rho_p, eta = case["radius"], 1.2, 1.0 / 6.0
        v_st = 0.1 * eta / (2.0 * R)
        force = 6.0 * math.pi * eta * R * v_st
        flags = torch.ones(grid, dtype=torch.uint8, device=DEVICE)
        flags[1:-1, 1:-1, 1:-1] = 0
        i["flags"] = flags
        prm.update(periodic=(0, 0, 0), lambda_p=max(0.25 * R / v_st, 10.0))
        off = (torch.rand(3, generator=g, device=DEVICE, dtype=torch.float64) - 0.5).tolist()
        X = ((nx - 1) / 2.0 + off[0], (ny - 1) / 2.0 + off[1], nz - 3.0 * R + off[2])
        i["particle"] = dict(X=X, R=R, rho_p=rho_p, v=(0.0, 0.0, -v_st), Fext=(0.0, 0.0, -force))
        i["u"] = _uniform(g, (3,) + grid, 1e-5)
    elif f == "mixed":
        flags = _obstacles(g, grid, 0.03)
        flags[:, 0, :] = workloads.NOSLIP
        flags[:, -1, :] = workloads.WALL0
        i["flags"] = flags
        i["wall_vel"] = [(0.01, 0.0, -0.004)]
        prm.update(periodic=(1, 0, 1), lambda_p=300.0)
        i["u"] = _uniform(g, (3,) + grid, 1e-3)
        i["tau"] = _uniform(g, (6,) + grid, 1e-5)
    elif f == "law":
        i["flags"] = _obstacles(g, grid, 0.01)
        prm.update(lambda_p=500.0)
        prm.update({"giesekus": dict(giesekus_alpha=0.3, fv_terms=lbve.FV_FLUX | lbve.FV_SOURCE | lbve.FV_CTU),
                    "fene": dict(fene_L2=100.0),
                    "ctu": dict(fv_terms=lbve.FV_FLUX | lbve.FV_SOURCE | lbve.FV_CTU),
                    "divu": dict(fv_terms=lbve.FV_FLUX | lbve.FV_SOURCE | lbve.FV_DIVU)}[case["law"]])
        i["u"] = _uniform(g, (3,) + grid, 1e-3)
        i["tau"] = _uniform(g, (6,) + grid, 1e-6)
    elif f == "noalloc":
        i["flags"] = torch.zeros(grid, dtype=torch.uint8, device=DEVICE)
        i["u"] = _uniform(g, (3,) + grid, 1e-3)
    i["params"] = prm
    return i


def _inputs_2d(case, seed):
    n = case["nx"]
    g = _rng(seed)
    if case["family"] == "cavity2d":
        c = workloads.cavity2d(L=n, u0=1e-3)
        ub, force = c["ub"], None
    else:
        c = workloads.four_roll_mill2d(N=n)
        ub, force = None, c["force"]
    nx, ny = c["shape"]
    flags = c.get("flags")
    if flags is None:
        flags = np.zeros((ny, nx), np.uint8)
    return {"shape": c["shape"], "params": c["params"], "flags": flags, "ub": ub, "force": force,
            "u": _uniform(g, (2, ny, nx), 1e-4).cpu().numpy()}


def _requests(case):
    """The pool's requests: their shapes and parameters belong to the case, not to the seed."""
    r = np.random.default_rng(case["mix"])
    return [serve.make_request(k, r) for k in range(case["members"])]


def _pool_u(req, seed, k):
    nx, ny, nz = req.shape
    return _uniform(_rng(1000 * seed + k), (3, nz, ny, nx), 1e-5)


# ---------------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------------


def _solver(i, precision, stream=0):
    s = lbve.Solver(i["shape"], precision=precision, stream=stream, **i["params"])
    s.set_geometry(i["flags"].cpu().numpy(), i["wall_vel"])
    if i["particle"] is not None:
        s.add_particle(**i["particle"])
    torch.cuda.current_stream().synchronize()
    s.init_fields_device(u_ptr=i["u"].data_ptr(), tau_ptr=0 if i["tau"] is None else i["tau"].data_ptr())
    s.synchronize()
    return s


def _fields(shape):
    nx, ny, nz = shape
    new = lambda *k: torch.zeros(k + (nz, ny, nx), dtype=torch.float64, device=DEVICE)  # noqa: E731
    return {"rho": new(), "u": new(3), "tau": new(6)}


def prepare(case, seed):
    f = case["family"]
    st = {"family": f, "steps": case["steps"]}
    if f in ("cavity2d", "mill2d"):
        i = _inputs_2d(case, seed)
        s = lbve.Solver2D(i["shape"], precision=case["precision"], **i["params"])
        s.set_geometry(i["flags"], i["ub"])
        if i["force"] is not None:
            s.set_force_field(i["force"])
        s.init_fields(u=i["u"])
        st["solver"] = s
        return st
    if f == "pool":
        stream = torch.cuda.Stream()
        pool = lbve.Pool(case["precision"], stream=stream.cuda_stream)
        solvers, fields = [], []
        for k, req in enumerate(_requests(case)):
            s = serve.build_solver(req, case["precision"], stream.cuda_stream)
            u = _pool_u(req, seed, k)
            torch.cuda.synchronize()
            s.init_fields_device(u_ptr=u.data_ptr())
            s.synchronize()
            pool.admit(s)
            solvers.append(s)
            fields.append(_fields(req.shape))
        torch.cuda.synchronize()
        st.update(pool=pool, solvers=solvers, fields=fields, stream=stream)
        return st
    i = _inputs(case, seed)
    if f == "noalloc":
        nx, ny, nz = i["shape"]
        n = nx * ny * nz
        np_ = (n + 63) // 64 * 64
        st["params"] = lbve.make_params(i["shape"], precision=case["precision"], **i["params"])
        dt = {"f32": torch.float32, "bf16": torch.bfloat16, "f16": torch.float16}[case["precision"]]
        # the stored deviations f_i - w_i rho0 of the equilibrium at rho0 and u (FP16: times 2^15)
        scale = 2.0 ** 15 if case["precision"] == "f16" else 1.0
        fs = torch.zeros(19, np_, dtype=dt, device=DEVICE)
        fs[:, :n] = (_deviations(i["u"]).reshape(19, n) * scale).to(dt)
        st.update(f=fs, tau_a=torch.zeros(6, np_, device=DEVICE), tau_b=torch.zeros(6, np_, device=DEVICE),
                  flags=i["flags"], t=0)
        return st
    st["solver"] = _solver(i, case["precision"])
    st["fields"] = _fields(i["shape"])
    return st


def _read(s, out):
    s.read_fields_device(out["rho"].data_ptr(), out["u"].data_ptr(), out["tau"].data_ptr())
    return out


def run(st):
    f = st["family"]
    if f in ("cavity2d", "mill2d"):
        st["solver"].step(st["steps"])
        rho, u, tau = st["solver"].read_fields()
        return {"rho": rho, "u": u, "tau": tau}
    if f == "pool":
        st["pool"].step(st["steps"])
        res = st["pool"].residuals()
        fields = [_read(s, o) for s, o in zip(st["solvers"], st["fields"])]
        torch.cuda.current_stream().wait_stream(st["stream"])
        # one tensor per field: the members' fields one after another
        return {"residuals": res, "rho": torch.cat([o["rho"].reshape(-1) for o in fields]),
                "u": torch.cat([o["u"].reshape(-1) for o in fields]),
                "tau": torch.cat([o["tau"].reshape(-1) for o in fields])}
    if f == "noalloc":
        lbve.step_noalloc(st["params"], st["f"].data_ptr(), st["tau_a"].data_ptr(), st["tau_b"].data_ptr(),
                          st["flags"].data_ptr(), t0=st["t"], nsteps=st["steps"],
                          stream=torch.cuda.current_stream().cuda_stream)
        st["t"] += st["steps"]  # an even number of steps: the state stays in the plain layout and in tau_a
        return {"f": st["f"], "tau": st["tau_a"]}
    st["solver"].step(st["steps"])
    out = dict(_read(st["solver"], st["fields"]))
    if f in ("duct", "mixed"):
        out["forces"] = st["solver"].body_forces()
    if f == "sediment":
        out["particle"] = st["solver"].read_particle(0)
    return out


# ---------------------------------------------------------------------------------
# the least a pass has to do
# ---------------------------------------------------------------------------------


def work(case):
    """Per step and cell: every population, the stress and the flag read once, populations
    and stress written once; the fields read back at the end of the pass."""
    f = case["family"]
    pdf = {"f64": 8, "f32": 4, "bf16": 2, "f16": 2}[case["precision"]]
    real = 8 if case["precision"] == "f64" else 4
    if f in ("cavity2d", "mill2d"):
        n = (case["nx"] + 2) ** 2 if f == "cavity2d" else case["nx"] ** 2
        step = 2 * 9 * pdf + 2 * 3 * real + 1
        return {"bytes": n * (case["steps"] * step + 6 * 8 + 9 * pdf), "flops": 250.0 * n * case["steps"]}
    if f == "pool":
        n = sum(int(np.prod(r.shape)) for r in _requests(case))
    else:
        n = int(np.prod(_shape(case)))
    step = 2 * 19 * pdf + 2 * 6 * real + 1
    read = 0 if f == "noalloc" else 10 * 8 + 19 * pdf + 6 * real
    return {"bytes": float(n) * (case["steps"] * step + read), "flops": 650.0 * n * case["steps"]}


# ---------------------------------------------------------------------------------
# the method's equations in 64 bits
# ---------------------------------------------------------------------------------
_FLUX, _SOURCE, _CTU, _DIVU = 1, 2, 4, 8  # bits of fv_terms
_C3 = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1), (1, 1, 0), (-1, -1, 0),
       (1, -1, 0), (-1, 1, 0), (1, 0, 1), (-1, 0, -1), (1, 0, -1), (-1, 0, 1), (0, 1, 1), (0, -1, -1), (0, 1, -1),
       (0, -1, 1)]
_C2 = [(0, 0), (1, 0), (-1, 0), (0, 1), (0, -1), (1, 1), (-1, -1), (1, -1), (-1, 1)]
_T3 = {(0, 0): 0, (1, 1): 1, (2, 2): 2, (0, 1): 3, (0, 2): 4, (1, 2): 5}
_T2 = {(0, 0): 0, (1, 1): 1, (0, 1): 2}


def _weight(c):
    k = sum(v * v for v in c)
    return (4.0 / 9.0, 1.0 / 9.0, 1.0 / 36.0)[k] if len(c) == 2 else (1.0 / 3.0, 1.0 / 18.0, 1.0 / 36.0)[k]


def _opposite(i):
    return 0 if i == 0 else (i + 1 if i % 2 else i - 1)


def _dot(c, v):
    """c . v for a lattice direction; the number 0 when c is zero."""
    t = 0.0
    for k, s in enumerate(c):
        if s:
            t = t + s * v[k]
    return t


def _deviations(u):
    """feq_i(1, u) - w_i in three dimensions."""
    usq = sum(u[k] * u[k] for k in range(3))
    cu = [_dot(c, u) for c in _C3]
    return torch.stack([_weight(c) * (3.0 * q + 4.5 * q * q - 1.5 * usq) for c, q in zip(_C3, cu)])


class _Reference:
    """The coupled step on a grid with every field in float64: TRT lattice Boltzmann with
    Guo forcing, link bounce-back, finite-volume stress update; rigid spheres in three
    dimensions.  flags: 0 fluid; ub: velocity of the solid cells, or None."""

    def __init__(self, shape, params, flags, ub=None, force=None, u=None, tau=None):
        p = dict(beta=0.5, eta=1.0 / 6.0, lambda_p=1000.0, body_force=(0.0,) * len(shape),
                 fv_terms=_FLUX | _SOURCE, giesekus_alpha=0.0, fene_L2=0.0)
        p.update(params)
        self.d = d = len(shape)
        self.C, self.T = (_C3, _T3) if d == 3 else (_C2, _T2)
        self.flags, self.fluid = flags, flags == 0
        self.ub, self.force, self.p = ub, force, p
        self.eta_p, self.lam = p["beta"] * p["eta"], p["lambda_p"]
        nu = (1.0 - p["beta"]) * p["eta"]
        self.wp = 1.0 / (3.0 * nu + 0.5)
        self.wm = 1.0 / (3.0 / 16.0 / (1.0 / self.wp - 0.5) + 0.5)
        grid = tuple(reversed(shape))
        new = lambda *k: torch.zeros(k + grid, dtype=torch.float64, device=DEVICE)  # noqa: E731
        self.zero = new()
        u = new(d) if u is None else u
        self.f = self.equilibrium(torch.ones_like(self.zero), u)
        self.tau = new(len(self.T)) if tau is None else tau * self.fluid
        if p["fene_L2"]:
            s = 3.0 + self.lam * (self.tau[0] + self.tau[1] + self.tau[2]) / self.eta_p
            A = self.lam * self.tau / self.eta_p
            A[:3] += 1.0
            self.tau = A / (1.0 + s / p["fene_L2"]) * self.fluid
        self.forces = np.zeros((256, 3))
        self.particle = None

    def at(self, a, c):
        """a at r + c (periodic; a closed side's outer layer is solid on both ends)."""
        dims = [k for k in range(self.d) if c[k]]
        return torch.roll(a, [-c[k] for k in dims], [-1 - k for k in dims]) if dims else a

    def unit(self, k, s):
        return tuple(s if q == k else 0 for q in range(self.d))

    def t(self, i, j):
        return self.T[(min(i, j), max(i, j))]

    def equilibrium(self, rho, u):
        usq = sum(u[k] * u[k] for k in range(self.d))
        f = torch.empty((len(self.C),) + tuple(rho.shape), dtype=torch.float64, device=DEVICE)
        for i, c in enumerate(self.C):
            cu = _dot(c, u)
            f[i] = _weight(c) * rho * (1.0 + 3.0 * cu + 4.5 * cu * cu - 1.5 * usq)
        return f

    def stress(self):
        if not self.p["fene_L2"]:
            return self.tau
        A = self.tau
        fac = 1.0 / (1.0 - (A[0] + A[1] + A[2]) / self.p["fene_L2"])
        s = fac * A
        s[:3] -= 1.0
        return s * (self.eta_p / self.lam) * self.fluid

    def macroscopic(self):
        d, ts = self.d, self.stress()
        F = [self.zero + self.p["body_force"][j] for j in range(d)]
        if self.force is not None:
            F = [F[j] + self.force[j] for j in range(d)]
        for k in range(d):
            for s in (1, -1):
                c = self.unit(k, s)
                fl = self.at(self.fluid, c)
                for j in range(d):
                    a = ts[self.t(k, j)]
                    F[j] = F[j] + s * torch.where(fl, 0.5 * (a + self.at(a, c)), a)
        del ts
        rho = self.f.sum(0)
        rs = torch.where(self.fluid, rho, 1.0)
        u = []
        for k in range(d):
            j = 0.5 * F[k]
            for i, c in enumerate(self.C):
                if c[k]:
                    j = j + c[k] * self.f[i]
            u.append(torch.where(self.fluid, j / rs, 0.0))
        return rho, u, F

    def new_stress(self, u):
        d, p, A = self.d, self.p, self.tau
        flux, src = p["fv_terms"] & _FLUX, p["fv_terms"] & _SOURCE
        ctu = p["fv_terms"] & _CTU
        out = A.clone()
        G = [[None] * d for _ in range(d)]
        for k in range(d):
            face = {}
            for s in (1, -1):
                c = self.unit(k, s)
                fl = self.at(self.fluid, c)
                face[s] = [torch.where(fl, 0.5 * (u[j] + self.at(u[j], c)),
                                       self.zero if self.ub is None else self.at(self.ub[j], c)) for j in range(d)]
                if flux:
                    over = 1.0
                    if ctu:
                        for q in range(d):
                            if q != k:
                                over = over * (1.0 - u[q].abs())
                    vout = torch.where(fl, (s * u[k]).clamp(min=0.0) * over, 0.0)
                    vin = torch.where(fl, self.at((-s * u[k]).clamp(min=0.0) * over, c), 0.0)
                    for q in range(len(self.T)):
                        out[q] += vin * self.at(A[q], c) - vout * A[q]
            for j in range(d):
                G[k][j] = face[1][j] - face[-1][j]
        if src:
            for (i, j), q in self.T.items():
                S = 0.0
                for k in range(d):
                    S = S + A[self.t(i, k)] * G[k][j] + A[self.t(k, j)] * G[k][i]
                if p["fene_L2"]:
                    fac = 1.0 / (1.0 - (A[0] + A[1] + A[2]) / p["fene_L2"])
                    S = S - (fac * A[q] - (1.0 if i == j else 0.0)) / self.lam
                else:
                    S = S + self.eta_p / self.lam * (G[i][j] + G[j][i]) - A[q] / self.lam
                if p["giesekus_alpha"]:
                    g = p["giesekus_alpha"] / self.eta_p
                    for k in range(d):
                        S = S - g * A[self.t(i, k)] * A[self.t(k, j)]
                out[q] += S
        if p["fv_terms"] & _DIVU:
            div = sum(G[k][k] for k in range(d))
            for q in range(len(self.T)):
                out[q] += A[q] * div
        return out * self.fluid

    def collide(self, rho, u, F):
        A, B = 3.0 * (1.0 - 0.5 * self.wm), 1.0 - 0.5 * self.wp
        usq = sum(u[k] * u[k] for k in range(self.d))
        uF = sum(u[k] * F[k] for k in range(self.d))
        f = self.f
        f[0] += -self.wp * (f[0] - _weight(self.C[0]) * rho * (1.0 - 1.5 * usq)) - _weight(self.C[0]) * B * 3.0 * uF
        for i in range(1, len(self.C), 2):
            c = self.C[i]
            w, cu, cF = _weight(c), _dot(c, u), _dot(c, F)
            even = -self.wp * (0.5 * (f[i] + f[i + 1]) - w * rho * (1.0 + 4.5 * cu * cu - 1.5 * usq))
            even = even + w * B * (9.0 * cu * cF - 3.0 * uF)
            odd = -self.wm * (0.5 * (f[i] - f[i + 1]) - 3.0 * w * rho * cu) + w * A * cF
            f[i] += even + odd
            f[i + 1] += even - odd

    def step(self, n):
        for _ in range(n):
            if self.particle is not None:
                self.surface_velocity()
            rho, u, F = self.macroscopic()
            tau = self.new_stress(u)
            self.collide(rho, u, F)
            new = torch.empty_like(self.f)
            if self.forces is not None:
                self.forces[:] = 0.0
            moved = np.zeros(6)
            for i, c in enumerate(self.C):
                # f_i(r) comes from r - c_i, or back from r when r - c_i is solid
                o, back = _opposite(i), tuple(-v for v in c)
                if i == 0:
                    new[0] = self.f[0]
                    continue
                X = self.zero
                if self.ub is not None:
                    X = 6.0 * _weight(c) * rho * _dot(back, [self.at(b, back) for b in self.ub])
                link = ~self.at(self.fluid, back)
                new[i] = torch.where(link, self.f[o] - X, self.at(self.f[i], back))
                if self.d == 3 and self.tracked:
                    link &= self.fluid
                    m = torch.where(link, 2.0 * self.f[o] - X, 0.0)
                    owner = self.at(self.flags, back)
                    for fl in self.tracked:
                        s = torch.where(owner == fl, m, 0.0)
                        total = float(s.sum())
                        self.forces[fl] += [v * total for v in back]
                        if self.particle is not None and fl == 64:
                            for k in range(3):
                                moved[3 + k] += float((s * self.lever_cross(back, k)).sum())
            self.f, self.tau = new, tau
            if self.particle is not None:
                moved[:3] = self.forces[64]
                self.move(moved)

    # -- wall classes and one rigid sphere ------------------------------------------
    tracked = ()

    def set_walls(self, wall_vel):
        self.tracked = tuple(2 + k for k in range(len(wall_vel)))
        if len(wall_vel):
            self.ub = torch.zeros((3,) + tuple(self.zero.shape), dtype=torch.float64, device=DEVICE)
            for k, v in enumerate(wall_vel):
                for a in range(3):
                    self.ub[a] += (self.flags == 2 + k).double() * float(v[a])

    def add_sphere(self, X, R, rho_p, v=(0, 0, 0), Fext=(0, 0, 0)):
        m = rho_p * 4.0 / 3.0 * math.pi * R ** 3
        self.particle = dict(X=np.array(X, float), v=np.array(v, float), w=np.zeros(3), F=np.zeros(3), T=np.zeros(3),
                             dP=np.zeros(3), dL=np.zeros(3), m=m, I=0.4 * m * R * R, R=R, Fext=np.array(Fext, float))
        self.tracked = (64,)
        self.axes = [torch.arange(self.zero.shape[-1 - k], dtype=torch.float64, device=DEVICE).reshape(
            [-1 if q == 2 - k else 1 for q in range(3)]) for k in range(3)]
        inside = self.inside() & self.fluid
        self.flags = torch.where(inside, 64, self.flags).to(torch.uint8)
        self.fluid = self.flags == 0
        self.tau = self.tau * self.fluid

    def arm(self, shift=(0, 0, 0)):
        """Displacement of r + shift from the sphere's centre, per axis (the sphere's cells
        do not cross a periodic side in these cases)."""
        return [self.axes[k] + shift[k] - self.particle["X"][k] for k in range(3)]

    def lever_cross(self, c, k):
        d = self.arm(c)
        a, b = (k + 1) % 3, (k + 2) % 3
        return d[a] * c[b] - d[b] * c[a]

    def inside(self):
        d = self.arm()
        return d[0] * d[0] + d[1] * d[1] + d[2] * d[2] <= self.particle["R"] ** 2

    def surface(self):
        P, d = self.particle, self.arm()
        v, w = P["v"], P["w"]
        return [v[k] + w[(k + 1) % 3] * d[(k + 2) % 3] - w[(k + 2) % 3] * d[(k + 1) % 3] + self.zero
                for k in range(3)]

    def surface_velocity(self):
        on = self.flags == 64
        self.ub = torch.stack([torch.where(on, s, 0.0) for s in self.surface()])

    def move(self, FT):
        P = self.particle
        P["F"], P["T"] = FT[:3].copy(), FT[3:].copy()
        P["v"] = P["v"] + (P["F"] + P["Fext"]) / P["m"]
        P["w"] = P["w"] + P["T"] / P["I"]
        P["X"] = P["X"] + P["v"]
        P["dP"], P["dL"] = np.zeros(3), np.zeros(3)
        inside = self.inside()
        gone, made = self.fluid & inside, (self.flags == 64) & ~inside
        if not bool((gone | made).any()):
            return
        stable = self.fluid & ~gone
        faces = [self.unit(k, s) for k in range(3) for s in (1, -1)]
        nf = sum(self.at(stable, c).double() for c in faces)
        fresh = sum(self.at(self.tau * stable, c) for c in faces) / (nf + 1.0) * made
        nf1 = nf.clamp(min=1.0)
        give = (self.tau * gone - fresh) / nf1  # what each stable face neighbour gains
        tau = self.tau + sum(self.at(give, c) for c in faces)
        d = [a + self.zero for a in self.arm()]
        # deleted momentum to the sphere, the momentum of the new cells from it
        mom = [sum(c[k] * self.f[i] for i, c in enumerate(self.C) if c[k]) * gone for k in range(3)]
        rho = self.f.sum(0) * stable
        cnt = sum(self.at(stable, c).double() for c in self.C[1:])
        rho_bar = torch.where(cnt > 0, sum(self.at(rho, c) for c in self.C[1:]) / cnt.clamp(min=1.0), 1.0)
        us = self.surface()
        feq = self.equilibrium(rho_bar, us)
        mom = [mom[k] - rho_bar * us[k] * made for k in range(3)]
        for k in range(3):
            a, b = (k + 1) % 3, (k + 2) % 3
            P["dP"][k] = float(mom[k].sum())
            P["dL"][k] = float((d[a] * mom[b] - d[b] * mom[a]).sum())
        self.f = torch.where(made, feq, self.f)
        self.flags = torch.where(gone, 64, torch.where(made, 0, self.flags)).to(torch.uint8)
        self.fluid = self.flags == 0
        self.tau = torch.where(made, fresh, tau) * self.fluid
        P["v"] = P["v"] + P["dP"] / P["m"]
        P["w"] = P["w"] + P["dL"] / P["I"]

    def fields(self):
        rho, u, _ = self.macroscopic()
        return {"rho": rho * self.fluid, "u": torch.stack(u) * self.fluid, "tau": self.stress() * self.fluid}


def _reference(i):
    r = _Reference(i["shape"], i["params"], i["flags"], u=i["u"], tau=i["tau"])
    r.set_walls(i["wall_vel"])
    if i["particle"] is not None:
        r.add_sphere(**i["particle"])
    return r


def exact(case, seed):
    f = case["family"]
    if f in ("cavity2d", "mill2d"):
        i = _inputs_2d(case, seed)
        dev = lambda a: None if a is None else torch.as_tensor(a).to(DEVICE)  # noqa: E731
        r = _Reference(i["shape"], i["params"], dev(i["flags"]), ub=dev(i["ub"]), force=dev(i["force"]), u=dev(i["u"]))
        r.step(case["steps"])
        return {k: v.cpu().numpy() for k, v in r.fields().items()}
    if f == "pool":
        out = []
        for k, req in enumerate(_requests(case)):
            i = {"shape": req.shape, "params": req.params, "flags": torch.from_numpy(req.flags).to(DEVICE),
                 "wall_vel": req.wall_vel, "particle": req.particle, "u": _pool_u(req, seed, k), "tau": None}
            r = _reference(i)
            r.step(case["steps"])
            out.append(r.fields())
        return {"residuals": None, **{q: torch.cat([o[q].reshape(-1) for o in out]) for q in ("rho", "u", "tau")}}
    i = _inputs(case, seed)
    r = _reference(i)
    r.step(case["steps"])
    if f == "noalloc":
        n = r.zero.numel()
        pad = lambda a: torch.nn.functional.pad(a.reshape(-1, n), (0, (n + 63) // 64 * 64 - n))  # noqa: E731
        scale = 2.0 ** 15 if case["precision"] == "f16" else 1.0
        w = torch.tensor([_weight(c) for c in _C3], dtype=torch.float64, device=DEVICE).reshape(19, 1, 1, 1)
        return {"f": pad((r.f - w) * scale), "tau": pad(r.tau)}
    out = r.fields()
    if f in ("duct", "mixed"):
        out["forces"] = r.forces
    if f == "sediment":
        P = r.particle
        out["particle"] = {k: P[k] for k in ("X", "v", "w", "F", "T", "dP", "dL", "m", "I", "R")}
    return out
