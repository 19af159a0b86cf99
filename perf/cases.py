"""Performance cases of the gas-kinetic solver: the work that a user has it do,
through the public binding `paper_1802_00704_gb300.gks`, from the smallest
meshes to the benchmark's.

A case is a dict of plain values.  `kind` says which entry points a pass takes:

  steps      a time loop of the user's own: `step()` once per step;
  run        a time loop on the device: `run()` for a number of steps;
  batch      independent meshes in one handle: `batch_run()`;
  operators  the parts of a step for a time integrator of the user's own:
             `cfl_dt()`, `cls_reconstruct()`, `limit()` (where a limiter is
             configured) and `flux()`;
  points     the Gauss-point flux on its own: `point_flux()`.

The first three start every pass from the case's initial state with a cold
reconstruction, as a program does that is given a new initial state, so a pass
has the same answer whenever it runs.  `flow` names the test problem (the
paper's Sec. IV, on the jittered split-quad triangulations of the package's
`inputs`); a seed moves the mesh's nodes and changes the flow's parameters.
`preset` names the solver configuration (PRESETS).

`exact` is the scheme in plain torch in 64 bits, written from the paper's
equations (arXiv:1802.00704) with none of the package's arithmetic: polynomials
in the particle velocities are dictionaries of monomials, the moment matrices
are inverted by LU, and the reconstruction is solved by fixed-point iteration.
"""
import math
import random

import numpy as np
import torch

from paper_1802_00704_gb300 import gks, inputs

GAMMA = 1.4
CLS_W = 0.3
CFL = 0.3

# Solver configurations in use: the library's defaults, its FP64 options, and
# the mixed-precision settings of the benchmark with the knobs that the
# autotuner picks on its workloads.
_MIXED = dict(precision=gks.MIXED, basis_fp32=1, ilu_fp16=1, warm_extrap=2)
PRESETS = {
    "fp64": {},
    "fp64_extrap": dict(warm_extrap=2),
    "mixed": dict(_MIXED),
    "mixed_one_sweep": dict(_MIXED, ilu_sweeps=1, ilu_sweeps_bwd=2, inner_rtol=1e-4, gmres_m=8, flux_shape=1),
    "mixed_batch": dict(_MIXED, ilu_sweeps=1, inner_rtol=1e-6, gmres_m=12),
    "mixed_viscous": dict(_MIXED, inner_rtol=1e-5),
    "mixed_fp64_flux": dict(_MIXED, inner_rtol=1e-5, flux_lead=2),
}


def listed():
    return [
        # The accuracy test's coarsest mesh with the defaults, one call per step:
        # everything is latency and launches.
        dict(name="advection_800_fp64_steps", kind="steps", flow="advection", nx=20, ny=20, steps=10, preset="fp64"),
        # Sod's shock tube (6,400 triangles) with the shock detector and the DWBAP limiter.
        dict(name="sod_6400_fp64_dwbap", kind="run", flow="riemann", nx=400, ny=8, steps=10, preset="fp64_extrap",
             limiter=1),
        # The paper's second-order variant (acoustic pulse) on a mid-size mesh.
        dict(name="pulse_20k_fp64_order2", kind="run", flow="pulse", nx=100, ny=100, steps=10, preset="fp64",
             second_order=1),
        # The benchmark's FP64 leg: the third-order scheme in FP64 on a large mesh.
        dict(name="shock_vortex_400k_fp64", kind="run", flow="shock_vortex", nx=632, ny=316, steps=3, preset="fp64"),
        # Mixed precision untuned on the error sample's size, with odd sides.
        dict(name="shock_vortex_41k_mixed", kind="run", flow="shock_vortex", nx=203, ny=101, steps=10,
             preset="mixed"),
        # The headline workload, the largest mesh, with the autotuner's knobs.
        dict(name="shock_vortex_1m_mixed", kind="run", flow="shock_vortex", nx=1000, ny=500, steps=8,
             preset="mixed_one_sweep"),
        # The viscous cavity: no-slip walls, Prandtl number 0.72.
        dict(name="cavity_131k_mixed", kind="run", flow="cavity", nx=256, ny=256, steps=8, preset="mixed_viscous"),
        # A viscous flow whose viscous stress is wanted in FP64 (flux_lead = 2).
        dict(name="cavity_18k_mixed_fp64_flux", kind="run", flow="cavity", nx=95, ny=97, steps=8,
             preset="mixed_fp64_flux"),
        # Many uneven meshes at once with the robust limiter.
        dict(name="batch_64_mixed_robust", kind="batch", flow="batch", cases=64, t_min=1000, t_max=40000, steps=5,
             preset="mixed_batch", limiter=2),
        # The operators of a step on their own, FP64, no limiter, ragged sides.
        dict(name="operators_51k_fp64", kind="operators", flow="pulse", nx=161, ny=159, preset="fp64"),
        # ... and in mixed precision with the characteristic DWBAP limiter.
        dict(name="operators_12k_mixed_char", kind="operators", flow="riemann", nx=501, ny=12, preset="mixed",
             limiter=1, limit_char=1),
        # The flux function alone on an odd number of state pairs.
        dict(name="points_100k_fp64", kind="points", flow="smooth", points=100003, preset="fp64"),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _sides(rng, tri, aspect):
    """Quad counts with 2 nx ny near tri triangles and nx / ny near the aspect."""
    ny = max(5, int(round(math.sqrt(tri / (2.0 * aspect)))))
    return max(5, int(round(tri / (2.0 * ny)))), ny


def draw(rng):
    kind = rng.choice(["steps", "run", "run", "run", "batch", "operators", "points"])
    if kind == "points":
        return dict(kind=kind, flow="smooth", points=int(_log_uniform(rng, 1000, 400000)), preset="fp64")
    if kind == "batch":
        return dict(kind=kind, flow="batch", cases=rng.randint(8, 64), t_min=rng.randint(800, 2000),
                    t_max=rng.randint(8000, 40000), steps=rng.randint(3, 6), preset="mixed_batch", limiter=2)
    if kind == "steps":
        nx, ny = _sides(rng, _log_uniform(rng, 800, 20000), rng.uniform(0.7, 1.5))
        return dict(kind=kind, flow=rng.choice(["advection", "pulse"]), nx=nx, ny=ny, steps=rng.randint(5, 12),
                    preset=rng.choice(["fp64", "fp64_extrap", "mixed"]))
    flow = rng.choice(["advection", "riemann", "pulse", "shock_vortex", "cavity"])
    if kind == "operators":
        flow = rng.choice(["riemann", "pulse"])
    aspect = {"riemann": rng.uniform(20.0, 60.0), "shock_vortex": 2.0}.get(flow, rng.uniform(0.8, 1.25))
    presets = {"cavity": ["mixed_viscous", "mixed_viscous", "mixed_fp64_flux"],
               "shock_vortex": ["mixed", "mixed_one_sweep", "fp64"],
               "riemann": ["fp64_extrap", "mixed"]}.get(flow, ["fp64", "fp64_extrap", "mixed"])
    preset = rng.choice(presets)
    # the costly configurations (FP64 flux) up to 400,000 triangles, the others up to 1,000,000
    top = 400000 if preset.startswith("fp64") or preset == "mixed_fp64_flux" else 1000000
    top = {"riemann": 40000, "pulse": 200000, "cavity": min(top, 200000)}.get(flow, top)
    tri = _log_uniform(rng, {"cavity": 8000}.get(flow, 2000), top)
    nx, ny = _sides(rng, tri, aspect)
    c = dict(kind=kind, flow=flow, nx=nx, ny=ny, preset=preset)
    if kind == "run":
        c["steps"] = max(2, min(10, int((1.2e6 if top == 400000 else 8e6) / tri)))
    if flow == "riemann":
        c["limiter"] = rng.choice([1, 1, 2])
        c["limit_char"] = rng.choice([0, 1]) if c["limiter"] == 1 else 0
    if flow == "pulse" and preset.startswith("fp64"):
        c["second_order"] = rng.choice([0, 1])
    return c


# ---------------------------------------------------------------------------
# Inputs: meshes and initial cell averages.

def _averages(mesh, fields):
    """Cell averages of the primitive fields(x, y) -> rho, u, v, p (3 x 3 rule)."""
    return inputs.cell_average(mesh, lambda x, y: inputs.prim_to_cons(*fields(x, y), GAMMA), n=3)


def _advection(nx, ny, seed):
    r = random.Random(seed)
    k, amp, phase = r.choice([1, 2]), r.uniform(0.05, 0.2), r.uniform(0.0, 2.0 * math.pi)
    mesh = inputs.split_quad_mesh(nx, ny, 2.0, 2.0, seed=seed, periodic_x=True, periodic_y=True)

    def fields(x, y):
        one = np.ones_like(x)
        return 1.0 + amp * np.sin(k * math.pi * (x + y) + phase), one, one, one

    return mesh, _averages(mesh, fields)


def _riemann(nx, ny, seed, robust=False):
    """A Riemann strip: near Sod's data (density ratio 8, pressure ratio 10), or
    (robust limiter) any ratios from 2 to 10."""
    r = random.Random(seed)
    rr, rp, split = r.uniform(7.0, 8.0), r.uniform(9.0, 10.0), r.uniform(0.45, 0.55)
    if robust:
        rr, rp = r.uniform(2.0, 10.0), r.uniform(2.0, 10.0)
    left = inputs.prim_to_cons(np.float64(rr), np.float64(0.0), np.float64(0.0), np.float64(rp), GAMMA)
    right = inputs.prim_to_cons(np.float64(1.0), np.float64(0.0), np.float64(0.0), np.float64(1.0), GAMMA)
    mesh = inputs.split_quad_mesh(nx, ny, 1.0, ny / nx, seed=seed, periodic_y=True,
                                  bc={"left": (inputs.TAG_DIRICHLET, left), "right": (inputs.TAG_DIRICHLET, right)})

    def fields(x, y):
        m = x < split
        return np.where(m, rr, 1.0), 0.0 * x, 0.0 * x, np.where(m, rp, 1.0)

    return mesh, _averages(mesh, fields)


def _pulse(nx, ny, seed):
    r = random.Random(seed)
    eps, width = r.uniform(0.005, 0.02), r.uniform(0.06, 0.12)
    alpha = math.log(2.0) / width ** 2
    mesh = inputs.split_quad_mesh(nx, ny, 1.0, 1.0, seed=seed, periodic_x=True, periodic_y=True)

    def fields(x, y):
        one = np.ones_like(x)
        return one, 0.0 * x, 0.0 * x, 1.0 + eps * np.exp(-alpha * ((x - 0.5) ** 2 + (y - 0.5) ** 2))

    return mesh, _averages(mesh, fields)


def _shock_vortex(nx, ny, seed):
    """Stationary Mach-1.1 shock at x = 0.5 with an isentropic vortex upstream."""
    r = random.Random(seed)
    mach, eps, a = 1.1, r.uniform(0.2, 0.3), r.uniform(0.05, 0.075)
    yc = r.uniform(0.45, 0.55)
    u1 = mach * math.sqrt(GAMMA)
    rho2 = (GAMMA + 1.0) * mach ** 2 / ((GAMMA - 1.0) * mach ** 2 + 2.0)
    p2 = 1.0 + 2.0 * GAMMA / (GAMMA + 1.0) * (mach ** 2 - 1.0)
    u2 = u1 / rho2
    state = [inputs.prim_to_cons(*[np.float64(q) for q in s], GAMMA) for s in
             ((1.0, u1, 0.0, 1.0), (rho2, u2, 0.0, p2))]
    mesh = inputs.split_quad_mesh(nx, ny, 2.0, 1.0, seed=seed,
                                  bc={"left": (inputs.TAG_DIRICHLET, state[0]),
                                      "right": (inputs.TAG_OUTFLOW, state[1]),
                                      "bottom": (inputs.TAG_SLIP, np.zeros(4)), "top": (inputs.TAG_SLIP, np.zeros(4))})

    def fields(x, y):
        dx, dy = (x - 0.25) / a, (y - yc) / a
        e = np.exp(0.5 * (1.0 - dx * dx - dy * dy))
        temp = 1.0 - 0.5 * (GAMMA - 1.0) / GAMMA * (eps * e) ** 2
        rho = temp ** (1.0 / (GAMMA - 1.0))
        left = x < 0.5
        return (np.where(left, rho, rho2), np.where(left, u1 - eps * dy * e, u2), np.where(left, eps * dx * e, 0.0),
                np.where(left, rho * temp, p2))

    return mesh, _averages(mesh, fields)


def _cavity_mu(seed):
    return 0.15 * math.sqrt(GAMMA) / random.Random(seed).uniform(400.0, 1000.0)


def _cavity(nx, ny, seed):
    """Lid-driven cavity (lid Mach number 0.15) with a swirl that has set in."""
    r = random.Random(seed + 1)
    ul = 0.15 * math.sqrt(GAMMA)
    swirl, tilt = r.uniform(0.3, 0.6) * ul, r.uniform(-0.2, 0.2)
    wall, lid = np.array([0.0, 0.0, 1.0, 0.0]), np.array([ul, 0.0, 1.0, 0.0])
    mesh = inputs.split_quad_mesh(nx, ny, 1.0, 1.0, seed=seed,
                                  bc={"left": (inputs.TAG_NOSLIP, wall), "right": (inputs.TAG_NOSLIP, wall),
                                      "bottom": (inputs.TAG_NOSLIP, wall), "top": (inputs.TAG_NOSLIP, lid)})

    def fields(x, y):
        sx, sy = np.sin(math.pi * x), np.sin(math.pi * y)
        u = -swirl * sx * sx * np.sin(2.0 * math.pi * y) + ul * sx * y ** 12
        v = swirl * sy * sy * np.sin(2.0 * math.pi * x) * (1.0 + tilt * y)
        p = 1.0 - 0.5 * swirl ** 2 * (sx * sy) ** 2
        return p, u, v, p

    return mesh, _averages(mesh, fields)


_FLOWS = {"advection": _advection, "riemann": _riemann, "pulse": _pulse, "shock_vortex": _shock_vortex,
          "cavity": _cavity}


def _batch_meshes(case, seed):
    """Log-uniform sizes; even members advect a wave, odd ones are Riemann strips
    (the sizes do not depend on the seed)."""
    r = random.Random(case["cases"])
    out = []
    for c in range(case["cases"]):
        t = _log_uniform(r, case["t_min"], case["t_max"])
        if c % 2 == 0:
            n = max(5, int(round(math.sqrt(t / 2.0))))
            out.append(_advection(n, n, seed * 1009 + c))
        else:
            out.append(_riemann(max(5, int(round(t / 16.0))), 8, seed * 1009 + c, robust=True))
    return out


def _physics(case, seed):
    """The handle's options beyond the preset."""
    kw = {k: case[k] for k in ("limiter", "limit_char", "second_order") if case.get(k)}
    if case["flow"] == "cavity":
        kw.update(mu=_cavity_mu(seed), prandtl=0.72)
    return kw


def _point_rows(case, seed):
    """State pairs in their face frames, (n, 6, 4) each: smooth flow data with
    small jumps; derivatives of a flow resolved by some tens of cells."""
    g = torch.Generator().manual_seed(seed)
    n = case["points"]

    def rand(*shape):
        return torch.rand(*shape, generator=g, dtype=torch.float64) * 2.0 - 1.0

    rho, u, v, p = 1.0 + 0.3 * rand(n), 0.8 * rand(n), 0.5 * rand(n), 1.0 + 0.3 * rand(n)
    rows = []
    for _ in range(2):
        f = torch.stack([rho * (1.0 + 0.02 * rand(n)), u + 0.02 * rand(n), v + 0.02 * rand(n),
                         p * (1.0 + 0.02 * rand(n))])
        val = torch.stack([f[0], f[0] * f[1], f[0] * f[2], f[3] / (GAMMA - 1.0) + 0.5 * f[0] * (f[1] ** 2 + f[2] ** 2)])
        rows.append(torch.cat([val.T[:, None], rand(n, 2, 4), 4.0 * rand(n, 3, 4)], dim=1).contiguous())
    return rows[0], rows[1], 0.01


def prepare(case, seed):
    dev = torch.device("cuda")
    s = {"case": dict(case)}
    if case["kind"] == "points":
        wl, wr, s["dt"] = _point_rows(case, seed)
        s["wl"], s["wr"] = wl.to(dev), wr.to(dev)
        return s
    kw = dict(PRESETS[case["preset"]], **_physics(case, seed))
    if case["kind"] == "batch":
        pairs = _batch_meshes(case, seed)
        s["mesh"] = gks.GksMesh.batch([m for m, _ in pairs], **kw)
        w0 = np.concatenate([w for _, w in pairs], axis=1)
    else:
        mesh, w0 = _FLOWS[case["flow"]](case["nx"], case["ny"], seed)
        s["mesh"] = gks.GksMesh(mesh, **kw)
    s["w0"] = torch.from_numpy(w0.copy()).to(dev)
    s["w"] = torch.empty_like(s["w0"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "points":
        return gks.point_flux(s["wl"], s["wr"], s["dt"])
    m = s["mesh"]
    m.reset_warm_start()
    if kind == "operators":
        w = s["w0"]
        dt = m.cfl_dt(w)
        coef, _ = m.cls_reconstruct(w)
        out = {"dt": dt, "coef": coef}
        if case.get("limiter"):
            coef, out["flags"] = m.limit(w, coef)
            out["limited"] = coef
        out["flux"], _ = m.flux(w, coef, dt)
        return out
    w = s["w"]
    w.copy_(s["w0"])
    if kind == "steps":
        dts = [m.step(w)["dt"] for _ in range(case["steps"])]
        return {"w": w, "dt": np.array(dts)}
    if kind == "run":
        info = m.run(w, max_steps=case["steps"])
        return {"w": w, "t": info["t"], "steps": info["steps"]}
    info = m.batch_run(w, max_steps=case["steps"])
    return {"w": w, "t": info["t"], "status": info["status"], "steps": info["steps"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without.

def _sizes(case):
    """(triangles, faces) of the case."""
    if case["kind"] == "batch":
        r = random.Random(case["cases"])
        tri = 0
        for c in range(case["cases"]):
            t = _log_uniform(r, case["t_min"], case["t_max"])
            tri += 2 * max(5, int(round(math.sqrt(t / 2.0)))) ** 2 if c % 2 == 0 else 16 * max(5, int(round(t / 16.0)))
    else:
        tri = 2 * case["nx"] * case["ny"]
    return tri, 3 * tri // 2


def work(case):
    """Bytes: the state read and written, the reconstruction's operator (24 values
    and 3 indices per triangle), the pivot blocks of its preconditioner (25 values)
    and the geometry of the faces (11 values, 2 indices), once per step; where the
    coefficients are asked for, those (20 values, once out, once in), and the face
    fluxes.  Operations: one application of the operator and the preconditioner
    (2 x 400 per triangle) and 1,500 per Gauss point of a face, the fewest of the
    moment sums of Eqs. (8)-(15)."""
    if case["kind"] == "points":
        return {"bytes": case["points"] * 8 * (48 + 4), "flops": 1500.0 * case["points"]}
    tri, faces = _sizes(case)
    f = 4 if case["preset"].startswith("mixed") else 8
    step = tri * (64 + f * 49 + 12) + faces * (8 * 11 + 8)
    flops = tri * 800.0 + 2 * faces * 1500.0
    if case["kind"] == "operators":
        return {"bytes": step + tri * 160 * (4 if case.get("limiter") else 2) + faces * 32, "flops": flops}
    return {"bytes": step * case["steps"], "flops": flops * case["steps"]}


# ---------------------------------------------------------------------------
# The scheme in 64 bits.  Polynomials in u, v, z = xi.xi are dictionaries
# {(a, b, c): coefficient tensor}; a slope s stands for s0 + s1 u + s2 v + s3 e.

def _psi(s):
    return {(0, 0, 0): s[0], (1, 0, 0): s[1], (0, 1, 0): s[2], (2, 0, 0): 0.5 * s[3], (0, 2, 0): 0.5 * s[3],
            (0, 0, 1): 0.5 * s[3]}


def _add(*polys):
    out = {}
    for p in polys:
        for k, c in p.items():
            out[k] = out[k] + c if k in out else c
    return out


def _scale(f, p):
    return {k: f * c for k, c in p.items()}


def _times(p, q):
    out = {}
    for (a, b, c), x in p.items():
        for (d, e, f), y in q.items():
            k = (a + d, b + e, c + f)
            out[k] = out[k] + x * y if k in out else x * y
    return out


def _shift(p, a, b=0):
    return {(i + a, j + b, k): c for (i, j, k), c in p.items()}


class _Maxwell:
    """Moments of a Maxwellian (density 1); side 0 the whole line in u, +1 u > 0, -1 u < 0."""

    def __init__(self, w, side=0, like=None):
        self.rho, self.U, self.V = w[0], w[1] / w[0], w[2] / w[0]
        self.p = (GAMMA - 1.0) * (w[3] - 0.5 * self.rho * (self.U ** 2 + self.V ** 2))
        self.h = self.p / self.rho                      # variance of each velocity component
        self.K = 2.0 / (GAMMA - 1.0) - 2.0
        one = torch.ones_like(self.U)
        if side == 0:
            u0, u1 = one, self.U
        else:
            q = torch.sqrt(2.0 * self.h)
            u0 = 0.5 * torch.special.erfc(-side * self.U / q)
            u1 = self.U * u0 + side * 0.5 * q / math.sqrt(math.pi) * torch.exp(-(self.U / q) ** 2)
        self.u = self._line(self.U, u0, u1)
        self.v = self._line(self.V, one, self.V)
        self.z = [one, self.K * self.h, self.K * (self.K + 2.0) * self.h ** 2,
                  self.K * (self.K + 2.0) * (self.K + 4.0) * self.h ** 3]

    def _line(self, mean, m0, m1):
        m = [m0, m1]
        for k in range(8):
            m.append(mean * m[k + 1] + (k + 1) * self.h * m[k])
        return m

    def mean(self, p):
        return sum(c * self.u[a] * self.v[b] * self.z[k] for (a, b, k), c in p.items())

    def psi(self, p, lift=0):
        """<u^lift psi P> as a stack of four."""
        e = _add(_scale(0.5, _shift(p, 2)), _scale(0.5, _shift(p, 0, 2)),
                 _scale(0.5, {(a, b, k + 1): c for (a, b, k), c in p.items()}))
        return torch.stack([self.mean(_shift(q, lift)) for q in (p, _shift(p, 1), _shift(p, 0, 1), e)])

    def matrix(self):
        one = torch.ones_like(self.U)
        unit = [_psi([one if q == r else 0.0 * one for q in range(4)]) for r in range(4)]
        return torch.stack([self.psi(p) for p in unit], dim=1).permute(2, 0, 1)   # (n, 4, 4)


def _slopes(m, rows, with_At):
    """Polynomials of the slopes of a state from its derivative rows (5, 4, n)."""
    lu = torch.linalg.lu_factor(m.matrix())

    def solve(b):
        return torch.linalg.lu_solve(*lu, b.T[..., None])[..., 0].T

    d = rows / m.rho
    a1, a2 = _psi(solve(d[0])), _psi(solve(d[1]))
    A = _psi(solve(-m.psi(_add(_shift(a1, 1), _shift(a2, 0, 1)))))
    s = {"a1": a1, "a2": a2, "A": A}
    for name, row, p, q in (("a11", 2, a1, a1), ("a12", 3, a1, a2), ("a22", 4, a2, a2)):
        s[name] = _psi(solve(d[row] - m.psi(_times(p, q))))
    lead = _add(_shift(a1, 1), _shift(a2, 0, 1), A)
    s["A1"] = _psi(solve(-m.psi(_add(_times(a1, lead), _shift(s["a11"], 1), _shift(s["a12"], 0, 1)))))
    s["A2"] = _psi(solve(-m.psi(_add(_times(a2, lead), _shift(s["a12"], 1), _shift(s["a22"], 0, 1)))))
    if with_At:
        s["At"] = _psi(solve(-m.psi(_add(_times(A, lead), _shift(s["A1"], 1), _shift(s["A2"], 0, 1)))))
    return s


def _time_integrals(dt, tau):
    """Integrals over [0, dt] of c1..c8 of Eq. (13) and of t^2 c7."""
    x = dt / tau
    small = x < 1.0
    xs = torch.where(small, x, torch.zeros_like(x))
    t, c = [torch.zeros_like(x) for _ in range(3)], [torch.zeros_like(x) for _ in range(3)]
    for k in range(24):                                  # series about x = 0
        f = (-1.0) ** k * xs ** k / float(math.factorial(k))
        for n in range(3):
            t[n] = t[n] + f * xs ** (n + 1) / (n + k + 1)
        if k >= 2:
            c[0] = c[0] + f
        if k >= 3:
            c[1] = c[1] + (k - 2) * f
            c[2] = c[2] - f
    e = torch.exp(-x)
    t0 = -torch.expm1(-x)
    t1 = t0 - x * e
    t2 = 2.0 * t1 - x * x * e
    t = [torch.where(small, p, q) for p, q in zip(t, (t0, t1, t2))]
    c = [torch.where(small, p, q) for p, q in zip(c, (x - t0, t1 + t0 - x, 0.5 * x * x - x + t0))]
    return [tau * c[0], tau ** 2 * c[1], tau ** 2 * c[2], -tau ** 3 * (t[2] + 2.0 * t[1]),
            tau ** 3 * (x ** 3 / 3.0 - x * x), -tau ** 3 * (0.5 * x * x + t[1]), tau * t[0], -tau ** 2 * t[1],
            tau ** 3 * t[2]]


def _point_flux(L, R, dt, mu=0.0, prandtl=1.0):
    """Time-integrated flux for face-frame rows L, R (6, 4, n) -> (4, n)."""
    half = (_Maxwell(L[0], 1), _Maxwell(R[0], -1))
    one = {(0, 0, 0): torch.ones_like(L[0, 0])}
    w0 = sum(m.rho * m.psi(one) for m in half)
    Z = _Maxwell(w0)
    jump = torch.abs(half[0].p - half[1].p) / torch.abs(half[0].p + half[1].p)
    tau = (mu / Z.p if mu > 0.0 else 0.01 * dt) + dt * jump
    C = _time_integrals(dt, tau)

    def quad(s):
        uv = _add(_shift(_add(_times(s["a1"], s["a1"]), s["a11"]), 2),
                  _scale(2.0, _shift(_add(_times(s["a1"], s["a2"]), s["a12"]), 1, 1)),
                  _shift(_add(_times(s["a2"], s["a2"]), s["a22"]), 0, 2))
        cross = _add(_shift(_add(_times(s["A"], s["a1"]), s["A1"]), 1),
                     _shift(_add(_times(s["A"], s["a2"]), s["A2"]), 0, 1))
        return _add(_shift(s["a1"], 1), _shift(s["a2"], 0, 1)), uv, cross

    s = _slopes(Z, 0.5 * (L[1:] + R[1:]), True)
    lin, uv, cross = quad(s)
    Q = _add(_scale(C[0], one), _scale(C[2], s["A"]), _scale(C[1], lin), _scale(0.5 * C[3], uv), _scale(C[5], cross),
             _scale(0.5 * C[4], _add(_times(s["A"], s["A"]), s["At"])))
    f, d = Z.rho * Z.psi(Q, 1), Z.rho * Z.psi(Q)
    for rows, m in zip((L, R), half):
        s = _slopes(_Maxwell(rows[0]), rows[1:], False)
        lin, uv, cross = quad(s)
        Q = _add(_scale(C[6], one), _scale(-tau * C[6], s["A"]), _scale(C[7] - tau * C[6], lin),
                 _scale(0.5 * C[8] - tau * C[7], uv), _scale(-tau * C[7], cross))
        f, d = f + m.rho * m.psi(Q, 1), d + m.rho * m.psi(Q)
    if prandtl != 1.0:
        U, V = Z.U, Z.V
        q2 = U * U + V * V
        heat = f[3] - U * f[1] - V * f[2] + (0.5 * q2 + U * U) * f[0] - U * d[3] + U * V * d[2] - 0.5 * U * q2 * d[0]
        f[3] = f[3] + (1.0 / prandtl - 1.0) * heat
    return f


# Second-order jets (value, d/dn, d/dt, d2/dn2, d2/dndt, d2/dt2) of the no-slip ghost.

def _jet_mul(a, b):
    return torch.stack([a[0] * b[0], a[1] * b[0] + a[0] * b[1], a[2] * b[0] + a[0] * b[2],
                        a[3] * b[0] + 2.0 * a[1] * b[1] + a[0] * b[3],
                        a[4] * b[0] + a[1] * b[2] + a[2] * b[1] + a[0] * b[4],
                        a[5] * b[0] + 2.0 * a[2] * b[2] + a[0] * b[5]])


def _jet_inv(b):
    q = 1.0 / b[0]
    q1, q2 = -b[1] * q * q, -b[2] * q * q
    return torch.stack([q, q1, q2, -(b[3] * q + 2.0 * b[1] * q1) * q, -(b[4] * q + b[1] * q2 + b[2] * q1) * q,
                        -(b[5] * q + 2.0 * b[2] * q2) * q])


def _mirror(sign_even):
    s = torch.tensor([1.0, -1.0, 1.0, 1.0, -1.0, 1.0], dtype=torch.float64)
    return (s if sign_even else -s)[:, None]


def _noslip_ghost(L, un_w, ut_w, t_w):
    inv = _jet_inv(L[:, 0])
    un, ut = _jet_mul(L[:, 1], inv), _jet_mul(L[:, 2], inv)
    p = (GAMMA - 1.0) * (L[:, 3] - 0.5 * (_jet_mul(L[:, 1], un) + _jet_mul(L[:, 2], ut)))
    T = _jet_mul(p, inv)
    even, odd = _mirror(True).to(L.device), _mirror(False).to(L.device)
    p, un, ut, T = even * p, odd * un, odd * ut, odd * T
    un[0] += 2.0 * un_w
    ut[0] += 2.0 * ut_w
    T[0] += 2.0 * t_w
    rho = _jet_mul(p, _jet_inv(T))
    mn, mt = _jet_mul(rho, un), _jet_mul(rho, ut)
    E = p / (GAMMA - 1.0) + 0.5 * (_jet_mul(mn, un) + _jet_mul(mt, ut))
    return torch.stack([rho, mn, mt, E], dim=1)


class _Scheme:
    """Geometry and one step of the scheme on one mesh."""

    def __init__(self, mesh, dev, mu=0.0, prandtl=1.0, limiter=0, limit_char=0, second_order=0):
        t = lambda a, d=torch.float64: torch.from_numpy(np.ascontiguousarray(a)).to(dev, d)  # noqa: E731
        self.mu, self.prandtl, self.limiter, self.char = mu, prandtl, limiter, limit_char
        p = t(mesh.nodes)[t(mesh.tris, torch.int64)]                       # (T, 3, 2)
        e = [torch.hypot(*(p[:, (k + 1) % 3] - p[:, k]).T) for k in range(3)]
        d1, d2 = p[:, 1] - p[:, 0], p[:, 2] - p[:, 0]
        self.area = 0.5 * torch.abs(d1[:, 0] * d2[:, 1] - d2[:, 0] * d1[:, 1])
        self.inrad = 2.0 * self.area / (e[0] + e[1] + e[2])
        self.h = torch.maximum(e[0] * e[1] * e[2] / (4.0 * self.area), torch.sqrt(self.area))
        self.c = p.mean(dim=1)
        dp = p - self.c[:, None]
        self.S = torch.stack([(dp[..., a] * dp[..., b]).sum(1) / 12.0 for a, b in ((0, 0), (0, 1), (1, 1))])
        f = t(mesh.faces, torch.int64)
        self.l, self.r, self.tag = f[:, 2], f[:, 3], f[:, 4]
        self.bnd = self.r < 0
        T = p.shape[0]
        self.k = torch.full((T,), 1 if second_order else 2, dtype=torch.int64, device=dev)
        self.k[self.l[self.bnd]] = 1
        a, b = t(mesh.nodes)[f[:, 0]], t(mesh.nodes)[f[:, 1]]
        self.len = torch.hypot(*(b - a).T)
        n = torch.stack([(b - a)[:, 1], -(b - a)[:, 0]]) / self.len
        out = ((0.5 * (a + b) - self.c[self.l]) * n.T).sum(1)
        self.n = torch.where(out < 0.0, -n, n)
        self.shift, self.bc = t(mesh.face_shift), t(mesh.bc_state).T
        rs = torch.where(self.bnd, self.l, self.r)
        self.gl, self.gr = [], []
        for s in (0.5 - 0.5 / math.sqrt(3.0), 0.5 + 0.5 / math.sqrt(3.0)):
            x = a + s * (b - a)
            self.gl.append(((x - self.c[self.l]) / self.h[self.l, None]).T)
            self.gr.append(((x - self.shift - self.c[rs]) / self.h[rs, None]).T)
        # directed pairs (i, j) of face neighbours, j's centroid in i's scaled frame
        two = ~self.bnd
        self.i = torch.cat([self.l[two], self.r[two]])
        self.j = torch.cat([self.r[two], self.l[two]])
        off = torch.cat([self.shift[two], -self.shift[two]])
        self.d = ((self.c[self.j] + off - self.c[self.i]) / self.h[self.i, None]).T
        dx, dy = self.d
        hi2 = self.h[self.i] ** 2
        m = [self.S[q][self.j] / hi2 - self.S[q][self.i] / hi2 for q in range(3)]
        zero, w = torch.zeros_like(dx), torch.full_like(dx, CLS_W)
        A = torch.stack([torch.stack([dx, dy, 0.5 * (dx * dx + m[0]), dx * dy + m[1], 0.5 * (dy * dy + m[2])]),
                         torch.stack([w, zero, w * dx, w * dy, zero]),
                         torch.stack([zero, w, zero, w * dx, w * dy])])       # (3, 5, E)
        A[:, 2:, self.k[self.i] == 1] = 0.0
        self.a0 = A[0]
        D = torch.zeros(25, T, dtype=torch.float64, device=dev)
        D.index_add_(1, self.i, torch.einsum("rae,rbe->abe", A, A).reshape(25, -1))
        D = D.T.reshape(T, 5, 5)
        pad = torch.zeros(T, 5, dtype=torch.float64, device=dev)
        pad[self.k == 1, 2:] = 1.0
        self.Dinv = torch.linalg.inv(D + torch.diag_embed(pad)).permute(1, 2, 0).contiguous()   # (5, 5, T)
        self.O = A[1:] * (CLS_W * self.h[self.i] / self.h[self.j])              # (2, 5, E): A^T B per gradient entry

    def reconstruct(self, w):
        """Coefficients (4, 5, T) of the per-cell least-squares system."""
        T = w.shape[1]
        du = w[:, self.j] - w[:, self.i]
        b = torch.zeros(4, 5, T, dtype=torch.float64, device=w.device)
        b.view(20, T).index_add_(1, self.i, (du[:, None] * self.a0).reshape(20, -1))
        u = torch.einsum("abt,vbt->vat", self.Dinv, b)
        best = math.inf
        for _ in range(400):
            g = u[:, :2, self.j]
            s = b.clone()
            s.view(20, T).index_add_(1, self.i, torch.einsum("gae,vge->vae", self.O, g).reshape(20, -1))
            new = torch.einsum("abt,vbt->vat", self.Dinv, s)
            change = float((new - u).norm() / new.norm().clamp_min(1e-300))
            u = new
            if change < 1e-14 and change > 0.7 * best:       # rounding is all that is left
                break
            best = min(best, change)
        return u

    def cell_values(self, w, u, c, x):
        """Values (4, n) of the cells c's polynomials at scaled offsets x (2, n)."""
        dx, dy = x
        m = self.S[:, c] / self.h[c] ** 2
        phi = torch.stack([dx, dy, 0.5 * (dx * dx - m[0]), dx * dy - m[1], 0.5 * (dy * dy - m[2])])
        return w[:, c] + (u[:, :, c] * phi).sum(1)

    def face_rows(self, w, u, c, x, n):
        """Face-frame rows (6, 4, n): value, d/dn, d/dt, d2/dn2, d2/dndt, d2/dt2."""
        dx, dy = x
        nx, ny = n
        ih = 1.0 / self.h[c]
        q = u[:, :, c]
        gx, gy = (q[:, 0] + q[:, 2] * dx + q[:, 3] * dy) * ih, (q[:, 1] + q[:, 3] * dx + q[:, 4] * dy) * ih
        xx, xy, yy = (q[:, s] * ih * ih for s in (2, 3, 4))
        rows = torch.stack([self.cell_values(w, u, c, x), nx * gx + ny * gy, nx * gy - ny * gx,
                            nx * nx * xx + 2.0 * nx * ny * xy + ny * ny * yy,
                            nx * ny * (yy - xx) + (nx * nx - ny * ny) * xy,
                            ny * ny * xx - 2.0 * nx * ny * xy + nx * nx * yy])
        mx, my = rows[:, 1].clone(), rows[:, 2].clone()
        rows[:, 1], rows[:, 2] = nx * mx + ny * my, nx * my - ny * mx
        return rows

    def ghosts(self, L, tag, bc, n):
        R = L.clone()                                            # outflow
        s = tag == inputs.TAG_DIRICHLET
        nx, ny = n
        R[:, :, s] = 0.0
        R[0][:, s] = torch.stack([bc[0], nx * bc[1] + ny * bc[2], nx * bc[2] - ny * bc[1], bc[3]])[:, s]
        s = tag == inputs.TAG_SLIP
        even, odd = _mirror(True).to(L.device), _mirror(False).to(L.device)
        for v in range(4):
            R[:, v, s] = (odd if v == 1 else even) * L[:, v, s]
        s = tag == inputs.TAG_NOSLIP
        if bool(s.any()):
            R[:, :, s] = _noslip_ghost(L[:, :, s], (nx * bc[0] + ny * bc[1])[s], (nx * bc[1] - ny * bc[0])[s], bc[2][s])
        return R

    def flux(self, w, u, dt, chunk=1 << 18):
        """Face fluxes (4, F) in the global frame."""
        F = self.l.shape[0]
        out = torch.zeros(4, F, dtype=torch.float64, device=w.device)
        for lo in range(0, F, chunk):
            f = slice(lo, min(F, lo + chunk))
            n, bnd = self.n[:, f], self.bnd[f]
            for g in range(2):
                L = self.face_rows(w, u, self.l[f], self.gl[g][:, f], n)
                rs = torch.where(bnd, self.l[f], self.r[f])
                R = self.face_rows(w, u, rs, self.gr[g][:, f], n)
                if bool(bnd.any()):
                    R[:, :, bnd] = self.ghosts(L[:, :, bnd], self.tag[f][bnd], self.bc[:, f][:, bnd], n[:, bnd])
                q = _point_flux(L, R, dt, self.mu, self.prandtl)
                out[:, f] += 0.5 * self.len[f] * torch.stack([q[0], n[0] * q[1] - n[1] * q[2],
                                                              n[1] * q[1] + n[0] * q[2], q[3]])
        return out

    def pressure(self, w):
        return (GAMMA - 1.0) * (w[3] - 0.5 * (w[1] ** 2 + w[2] ** 2) / w[0])

    def cfl_dt(self, w):
        speed = torch.hypot(w[1], w[2]) / w[0] + torch.sqrt(GAMMA * self.pressure(w) / w[0])
        return CFL * float((self.inrad / (speed + 2.0 * self.mu / (w[0] * self.inrad))).min())

    def physical(self, w, u):
        """Cells whose polynomial has rho > 0 and p > 0 at all their Gauss points."""
        ok = torch.ones(w.shape[1], dtype=torch.bool, device=w.device)
        two = ~self.bnd
        for c, gs, sel in ((self.l, self.gl, slice(None)), (self.r[two], self.gr, two)):
            for g in gs:
                v = self.cell_values(w, u, c, g[:, sel])
                ok[c[~((v[0] > 0.0) & (self.pressure(v) > 0.0))]] = False
        return ok

    def limit(self, w, u):
        """Detector (Eqs. (37)-(38)) and DWBAP limiter (Eqs. (34)-(36)): limited
        coefficients, flags (1 limited, 2 reset to the average)."""
        i, j, T = self.i, self.j, w.shape[1]
        acc = lambda x: torch.zeros(T, dtype=torch.float64, device=w.device).index_add_(0, i, x)  # noqa: E731
        J = acc(torch.ones_like(self.d[0]))
        ri = -self.d * (self.h[i] / self.h[j])                   # r_i in j's scaled frame
        at_i = self.cell_values(w, u, i, torch.zeros_like(self.d))
        at_j = self.cell_values(w, u, j, ri)
        scale = J * self.h ** (0.5 * (self.k + 1))
        smooth = torch.ones(T, dtype=torch.bool, device=w.device)
        for v in (0, 3):
            top = w[v].clone().index_reduce_(0, i, w[v][j], "amax")
            smooth &= acc(torch.abs(at_i[v] - at_j[v])) / (scale * top) < 1.0
        flagged = (J > 0) & ~(smooth & self.physical(w, u))
        lim, flags = u.clone(), torch.zeros(T, dtype=torch.int32, device=w.device)
        if self.limiter == 2:
            lim[:, :, flagged] = 0.0
            flags[flagged] = 2
            return lim, flags
        # weights from the distances to the interior faces' midpoints and the pressures' spread
        two = ~self.bnd
        mid = torch.cat([0.5 * (self.gl[0] + self.gl[1])[:, two], 0.5 * (self.gr[0] + self.gr[1])[:, two]], dim=1)
        order = torch.argsort(i, stable=True)
        first = torch.searchsorted(i[order], torch.arange(T, device=w.device))
        slot = torch.empty_like(i)
        slot[order] = torch.arange(i.shape[0], device=w.device) - first[i[order]]
        put = lambda x, fill: torch.full((3, T), fill, dtype=x.dtype, device=w.device).index_put_((slot, i), x)  # noqa: E731
        has = put(torch.ones_like(i, dtype=torch.bool), False)
        mx, my, ox, oy = put(mid[0], 0.0), put(mid[1], 0.0), put(self.d[0], 0.0), put(self.d[1], 0.0)
        pj = put(self.pressure(w)[j], 0.0)
        mean = pj.sum(0) / J
        chi = torch.sqrt((has * (pj - mean) ** 2).sum(0) / J) / mean
        power = -1.0 / (torch.sqrt(chi + 1e-8) + 0.05)
        dist = [self.h * (has * torch.hypot(px - mx, py - my)).sum(0) / J
                for px, py in [(0.0 * ox[0], 0.0 * oy[0])] + [(ox[q], oy[q]) for q in range(3)]]
        om = torch.stack([dist[0] ** power] + [torch.where(has[q], dist[1 + q] ** power, 0.0 * J) for q in range(3)])
        nb = put(j, 0)
        hj, kj = self.h[nb], self.k[nb]
        rix, riy = -ox * self.h / hj, -oy * self.h / hj
        for l in range(5):
            high = l >= 2
            sel = flagged & (self.k == 2) if high else flagged
            if not bool(sel.any()):
                continue
            unit = self.h ** 2 if high else self.h
            cand, wt = [u[:, l] / unit], [om[0]]
            for q in range(3):
                un = u[:, :, nb[q]]
                if high:
                    cand.append(un[:, l] / hj[q] ** 2)
                    wt.append(torch.where(kj[q] == 2, om[1 + q], 0.0 * J))
                else:
                    cand.append((un[:, l] + un[:, 2 + l] * rix[q] + un[:, 3 + l] * riy[q]) / hj[q])
                    wt.append(om[1 + q])
            cand, wt = torch.stack(cand)[:, :, sel], torch.stack(wt)[:, sel]
            wt = wt / wt.sum(0)
            if self.char:
                nx, ny = {0: (1.0, 0.0), 1: (0.0, 1.0), 2: (1.0, 0.0), 4: (0.0, 1.0)}.get(l, (math.sqrt(0.5),) * 2)
                right = self.eigenvectors(w[:, sel], nx, ny)                      # (n, 4, 4)
                cand = torch.linalg.solve(right[None], cand.permute(0, 2, 1)[..., None])[..., 0].permute(0, 2, 1)
            own = cand[0]
            safe = torch.where(own == 0.0, torch.ones_like(own), own)
            res = own * torch.tan((wt[:, None] * torch.atan(cand / safe)).sum(0))
            if self.char:
                res = torch.einsum("nab,bn->an", right, res)
            lim[:, l, sel] = unit[sel] * res
        flags[flagged] = 1
        bad = flagged & ~self.physical(w, lim)
        lim[:, :, bad] = 0.0
        flags[bad] = 2
        return lim, flags

    def eigenvectors(self, w, nx, ny):
        """Right eigenvectors (columns) of the Euler flux Jacobian along (nx, ny)."""
        u, v = w[1] / w[0], w[2] / w[0]
        p = self.pressure(w)
        c, H = torch.sqrt(GAMMA * p / w[0]), (w[3] + p) / w[0]
        one, qn = torch.ones_like(u), u * nx + v * ny
        cols = [[one, u - c * nx, v - c * ny, H - qn * c], [one, u, v, 0.5 * (u * u + v * v)],
                [0.0 * one, -ny * one, nx * one, -u * ny + v * nx], [one, u + c * nx, v + c * ny, H + qn * c]]
        return torch.stack([torch.stack(col) for col in cols], dim=1).permute(2, 0, 1)

    def step(self, w, dt):
        u = self.reconstruct(w)
        if self.limiter:
            u, _ = self.limit(w, u)
        F = self.flux(w, u, dt)
        two = ~self.bnd
        change = torch.zeros_like(w).index_add_(1, self.l, -F).index_add_(1, self.r[two], F[:, two])
        return w + change / self.area


def exact(case, seed):
    dev = torch.device("cuda" if torch.cuda.is_available() else "cpu")
    if case["kind"] == "points":
        wl, wr, dt = _point_rows(case, seed)
        return _point_flux(wl.to(dev).permute(1, 2, 0), wr.to(dev).permute(1, 2, 0), dt).T.contiguous()
    kw = _physics(case, seed)
    if case["kind"] == "batch":
        ws, ts = [], []
        for mesh, w0 in _batch_meshes(case, seed):
            w, t, _ = _march(_Scheme(mesh, dev, **kw), w0, case["steps"], dev)
            ws.append(w)
            ts.append(t)
        return {"w": torch.cat(ws, dim=1), "t": np.array(ts), "status": None, "steps": None}
    mesh, w0 = _FLOWS[case["flow"]](case["nx"], case["ny"], seed)
    sch = _Scheme(mesh, dev, **kw)
    if case["kind"] == "operators":
        w = torch.from_numpy(w0.copy()).to(dev)
        dt = sch.cfl_dt(w)
        out = {"dt": dt, "coef": sch.reconstruct(w)}
        u = out["coef"]
        if case.get("limiter"):
            u, out["flags"] = sch.limit(w, u)
            out["limited"] = u
        out["flux"] = sch.flux(w, u, dt)
        return out
    w, t, dts = _march(sch, w0, case["steps"], dev)
    if case["kind"] == "steps":
        return {"w": w, "dt": np.array(dts)}
    return {"w": w, "t": t, "steps": None}


def _march(sch, w0, steps, dev):
    w, t, dts = torch.from_numpy(w0.copy()).to(dev), 0.0, []
    for _ in range(steps):
        dts.append(sch.cfl_dt(w))
        t += dts[-1]
        w = sch.step(w, dts[-1])
    return w, t, dts
