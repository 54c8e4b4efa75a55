"""The work that users of this framework have it do, as cases that can be timed.

Every case goes through the public entry points of `paper_2410_21607_gb300.sem`
with the calls that a program makes: a Runge-Kutta step in either form, a single
tendency, the batched step, the refinement criterion with the wind diagnostics,
a remesh, and the network's inference and training.  Sizes are those of the
configurations, tests and benchmark of this repository or lie between them.

`exact` restates the method in float64 torch: the arithmetic is written out
here; only the mesh's own numbering (column map, hanging rows, leaves, heights)
and the inputs that `prepare` makes are taken over.
"""
import math

import numpy as np
import torch

from paper_2410_21607_gb300 import sem

DEV = "cuda"
LZ = 24.0e3
G, F0, RD, CP, P00, THS, NBV = 9.81, 5.0e-5, 287.0, 1004.0, 1.0e5, 300.0, 0.01
CV, GAMMA = CP - RD, CP / (CP - RD)
THRESHOLDS = (5.0, 10.0, 15.0)
SCALES = (1e-3, 10.0, 10.0, 1.0, 1.0)
CLASS_W = (0.6, 0.5, 4.0)
RUN_STEPS = 400   # steps of one run; the next run starts from the initial state again


# --------------------------------------------------------------------------- cases
def listed():
    """The cases; each comment says what it stands for."""
    return [
        # the benchmark run: the mixed form on the large uniform mesh, tuned once
        _step("step 64x64x16 N4", 64, 64, 16, 4, tuned=True),
        # the smallest run (config "6x6x4"): a step is a few launches
        _step("step 6x6x4 N4", 6, 6, 4, 4, width_km=100.0),
        # an adaptive run between two remeshes: three levels inside 150 km, 2:1 faces
        _step("step amr 32x32x8 N4", 32, 32, 8, 4, width_km=18.75, levels=3),
        # the paper's own equation set with its stress and absorbing layer
        _step("step paper terms 40x36x12 N4", 40, 36, 12, 4, eqset="NC", terms=True),
        # an order above the benchmark's on warped (non-affine) layers
        _step("step warped 30x26x10 N5", 30, 26, 10, 5, warp=True),
        # the float64 form, the reference that mixed runs are judged against
        _step("step fp64 32x32x16 N4", 32, 32, 16, 4, form="fp64"),
        # one float64 tendency on the small adaptive mesh (a caller's own time loop)
        _step("rhs fp64 amr 8x8x4 N4", 8, 8, 4, 4, width_km=75.0, levels=2, form="fp64", kind="rhs"),
        # many storms at once: uneven meshes and orders in one graph launch per step
        {"name": "batch 12 instances", "kind": "batch", "instances": 12, "most": 24, "mix": 4, "levels": 1},
        # the checks between remeshes and the run's wind record
        {"name": "monitor 64x64x16 N4", "kind": "monitor", "nx": 64, "ny": 64, "nz": 16, "N": 4, "width_km": 32.0,
         "levels": 0, "criterion": "speed"},
        # a remesh of the adaptive run: criterion, host plan, new mesh, transfer
        {"name": "remesh amr 32x32x8 N4", "kind": "remesh", "nx": 32, "ny": 32, "nz": 8, "N": 4, "width_km": 18.75,
         "levels": 3},
        # the learned schedule's inference on every element of the large mesh
        {"name": "predict 64x64x16 N4", "kind": "predict", "nx": 64, "ny": 64, "nz": 16, "N": 4, "width_km": 32.0,
         "levels": 0},
        # one training iteration of the flag network at its usual batch
        {"name": "train 65536 rows", "kind": "train", "rows": 65536},
    ]


def _step(name, nx, ny, nz, N, width_km=32.0, levels=0, form="mixed", eqset="C", terms=False, warp=False,
          tuned=False, kind="step"):
    c = {"kind": kind, "form": form, "set": eqset, "nx": nx, "ny": ny, "nz": nz, "N": N, "width_km": width_km,
         "levels": levels, "terms": terms, "warp": warp, "tuned": tuned}
    return dict(c, name=name) if name else c


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the same ranges."""
    kind = rng.choice(["mixed", "mixed", "mixed", "paper", "warped", "fp64", "rhs", "batch", "monitor", "remesh",
                       "predict", "train"])
    N = rng.choice([2, 3, 4, 4, 4, 5, 6])
    budget = {"mixed": 8.0e6, "paper": 4.0e6, "warped": 2.5e6, "fp64": 1.2e6, "rhs": 1.2e6, "monitor": 8.0e6,
              "remesh": 1.0e6, "predict": 8.0e6}.get(kind, 1e6)
    nz = rng.randint(2, 18)
    cols = min(_log_int(rng, 16, 4096), int(budget / (nz * (N + 1) ** 3)))
    nx = max(4, int(math.sqrt(cols) * rng.uniform(0.8, 1.25)))
    ny = max(4, cols // nx)
    width = rng.uniform(12.0, 60.0)
    if kind == "train":
        return {"kind": "train", "rows": _log_int(rng, 1500, 65536)}
    if kind == "batch":
        return {"kind": "batch", "instances": rng.randint(3, 14), "most": rng.choice([12, 16, 20, 24]),
                "mix": rng.randint(0, 10 ** 6), "levels": rng.randint(0, 1)}
    levels = rng.randint(1, 2) if kind == "remesh" or rng.random() < 0.4 else 0
    if levels:   # the refined storm region multiplies the columns
        nx, ny = max(5, int(nx * 0.55)), max(5, int(ny * 0.55))
    if kind == "mixed":
        return _step(None, nx, ny, nz, N, width, levels, terms=rng.random() < 0.3, tuned=rng.random() < 0.5)
    if kind == "paper":
        return _step(None, nx, ny, nz, N, width, levels, eqset="NC", terms=rng.random() < 0.5)
    if kind == "warped":
        return _step(None, nx, ny, nz, N, width, 0, eqset=rng.choice(["C", "C", "NC"]), warp=True)
    if kind in ("fp64", "rhs"):
        return _step(None, nx, ny, nz, N, width, levels, form="fp64", eqset=rng.choice(["C", "C", "NC"]),
                     kind="step" if kind == "fp64" else "rhs")
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "N": N, "width_km": width, "levels": levels}
    if kind == "monitor":
        c["criterion"] = rng.choice(["speed", "speed", "vorticity", "pv"])
    return c


# --------------------------------------------------------------------------- meshes and states
def _mesh(c, lvl_max=3):
    """The case's mesh: a base grid, refined `levels` times in whole columns
    inside a storm region (a quarter of the smaller side), 2:1 balanced."""
    Lx, Ly = c["nx"] * c["width_km"] * 1e3, c["ny"] * c["width_km"] * 1e3
    warp = (500.0, 2, 3) if c.get("warp") else None
    m = sem.sem_mesh_create(Lx, Ly, LZ, c["nx"], c["ny"], c["nz"], c["N"], lvl_max=lvl_max, warp=warp)
    for _ in range(c.get("levels", 0)):
        lv = sem.sem_mesh_leaves_host(m).astype(np.float64)
        h = 0.5 ** lv[:, 0]
        x = -0.5 * Lx + (lv[:, 1] + 0.5) * Lx / c["nx"] * h
        y = -0.5 * Ly + (lv[:, 2] + 0.5) * Ly / c["ny"] * h
        inside = np.hypot(x, y) < 0.25 * min(Lx, Ly)
        m = sem.sem_transfer_plan(m, np.repeat(inside.astype(np.int8), c["nz"]))
    return m


def _reference(z):
    """theta0, p0, rho0, (rho theta)0 and dtheta0/dz of the constant-N atmosphere."""
    th = THS * torch.exp(NBV * NBV * z / G)
    pi = 1.0 + G * G / (CP * THS * NBV * NBV) * (torch.exp(-NBV * NBV * z / G) - 1.0)
    p = P00 * pi ** (CP / RD)
    rho = P00 * pi ** (CV / RD) / (RD * th)
    return th, p, rho, rho * th, th * NBV * NBV / G


def _state(mesh, Lx, Ly, seed, eqset="C", storm=None):
    """A warm-core vortex in gradient-wind and hydrostatic balance (closed form:
    the pressure falls by Pc exp(-(r/L)^2) exp(-z^2 / 2 D^2)), off the centre, with
    a small vertical motion and 0.1 K of theta noise; all from the seed, or, with
    the storm's five numbers in 0..1 given, only the noise."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    r4 = storm or torch.rand(5, generator=g, device=DEV, dtype=torch.float64).tolist()
    vmax, L = 15.0 + 25.0 * r4[0], min(30e3 + 50e3 * r4[1], 0.12 * min(Lx, Ly))
    xyz = torch.empty((3, mesh.NG), dtype=torch.float64, device=DEV)
    sem.sem_mesh_coords(mesh, xyz)
    x, y, z = xyz[0] - (r4[2] - 0.5) * 0.1 * Lx, xyz[1] - (r4[3] - 0.5) * 0.1 * Ly, xyz[2]
    r2 = x * x + y * y
    D = 7000.0
    th0, p0, rho0, rt0, _ = _reference(z)
    Pc = 1.15 * vmax * vmax * math.e / 2.0
    shape = torch.exp(-r2 / (L * L)) * torch.exp(-z * z / (2 * D * D))
    rp = -Pc * shape * z / (D * D) / G                 # -(1/g) dp'/dz
    rho = rho0 + rp
    rt = P00 / RD * ((p0 - Pc * shape) / P00) ** (CV / CP)
    dpdr_r = 2.0 * Pc / (L * L) * shape                # (1/r) dp'/dr
    om = -0.5 * F0 + torch.sqrt(0.25 * F0 * F0 + dpdr_r / rho)   # v / r
    w = 0.2 * torch.sin(math.pi * z / LZ) * torch.sin(2 * math.pi * (x / Lx + r4[4])) * torch.cos(2 * math.pi * y / Ly)
    noise = 0.1 * (2.0 * torch.rand(mesh.NG, generator=g, device=DEV, dtype=torch.float64) - 1.0)
    if eqset == "NC":
        return torch.stack([rp, -om * y, om * x, w, rt / rho - th0 + noise])
    return torch.stack([rp, -rho * om * y, rho * om * x, rho * w, rt - rt0 + rho * noise])


def _params(c, **more):
    p = dict(precision=sem.SEM_PREC_FP64 if c.get("form", "mixed") == "fp64" else sem.SEM_PREC_MIXED,
             eqset=sem.SEM_EQ_NONCONSERVATIVE if c.get("set", "C") == "NC" else sem.SEM_EQ_CONSERVATIVE)
    if c.get("terms"):   # the paper's values
        p.update(smag_cs=0.21, sponge_gamma=1.0, sponge_depth=4000.0)
    return sem.sem_params_default(**p, **more)


def _basis(N):
    """LGL nodes, weights and the derivative matrix D[i][j] = h_j'(xi_i), float64 numpy."""
    P = np.polynomial.legendre.Legendre.basis(N)
    xi = np.concatenate([[-1.0], np.sort(np.real(P.deriv().roots())), [1.0]])
    for _ in range(3):   # polish the interior roots of P_N'
        d1, d2 = P.deriv()(xi[1:-1]), P.deriv(2)(xi[1:-1])
        xi[1:-1] -= d1 / d2
    w = 2.0 / (N * (N + 1) * P(xi) ** 2)
    D = np.zeros((N + 1, N + 1))
    for i in range(N + 1):
        for j in range(N + 1):
            if i != j:
                D[i, j] = P(xi[i]) / P(xi[j]) / (xi[i] - xi[j])
        D[i, i] = -D[i].sum()
    return xi, w, D


def _dt(c):
    """Acoustic Courant number 0.3 on the smallest LGL spacing."""
    xi = _basis(c["N"])[0]
    gap = 0.5 * (xi[1] - xi[0])
    return 0.3 * gap * min(c["width_km"] * 1e3 / (1 << c.get("levels", 0)), LZ / c["nz"]) / 347.0


def _instances(c):
    """The batch's uneven instances: base size, layers, order, level, width."""
    rng = np.random.default_rng(1000 + c["mix"])
    out = []
    for _ in range(c["instances"]):
        n = int(rng.integers(2, c["most"] // 4 + 1)) * 4
        out.append({"nx": n, "ny": n, "nz": max(n // 4, 2), "N": int(rng.integers(3, 7)),
                    "levels": int(rng.integers(0, c["levels"] + 1)), "width_km": float(rng.uniform(15.0, 40.0))})
    return out


def _buffers(mesh, q):
    """The float32 mirror and scratch that a mixed step works with."""
    q32 = torch.empty(q.shape, dtype=torch.float32, device=DEV)
    work = torch.zeros((10, mesh.NG), dtype=torch.float32, device=DEV)
    sem.sem_mirror(mesh, q, q32)
    return q32, work


def _box(c):
    return c["nx"] * c["width_km"] * 1e3, c["ny"] * c["width_km"] * 1e3


def prepare(case, seed):
    c, k = case, case["kind"]
    s = {"case": c, "left": RUN_STEPS}
    if k == "train":
        g = torch.Generator(device=DEV).manual_seed(int(seed))
        n = c["rows"]
        X = torch.randn((n, 136), generator=g, device=DEV)
        # rows are elements: the 27 samples of a field share the element's mean
        X[:, :135] = 0.3 * X[:, :135] + torch.randn((n, 5), generator=g, device=DEV).repeat_interleave(27, dim=1)
        X[:, 135] = torch.randint(0, 4, (n,), generator=g, device=DEV).float()
        speed = (X[:, 27:54] ** 2 + X[:, 54:81] ** 2).amax(dim=1) + 0.3 * torch.randn(n, generator=g, device=DEV)
        s["X"], s["y"] = X.contiguous(), ((speed > 1.0).to(torch.int8) + (speed > 4.0).to(torch.int8)).contiguous()
        s["net"] = sem.sem_mlp_create(int(seed) % 100003, n)
        return s
    if k == "batch":
        s["cases"] = _instances(c)
        s["meshes"] = [_mesh(i) for i in s["cases"]]
        s["q"] = [_state(m, *_box(i), seed + 7 * n) for n, (m, i) in enumerate(zip(s["meshes"], s["cases"]))]
        s["q0"] = [q.clone() for q in s["q"]]
        s["q32"], s["work"] = map(list, zip(*[_buffers(m, q) for m, q in zip(s["meshes"], s["q"])]))
        s["dt"], s["p"] = [_dt(i) for i in s["cases"]], _params({})
        s["batch"] = sem.sem_batch_create(s["meshes"])
        return s
    m = s["mesh"] = _mesh(c)
    # the size of a remesh's result follows from the winds: there the seed leaves the storm as it is
    q = s["q"] = _state(m, *_box(c), seed, c.get("set", "C"), (0.6, 0.6, 0.9, 0.7, 0.25) if k == "remesh" else None)
    if k == "step":
        s["p"], s["dt"], s["q0"] = _params(c), _dt(c), q.clone()
        if c["form"] == "mixed":
            s["q32"], s["work"] = _buffers(m, q)
            if c["tuned"]:
                sem.sem_autotune(m, s["p"], s["q32"], 3)
        else:
            s["w1"], s["w2"] = torch.empty_like(q), torch.empty_like(q)
    elif k == "rhs":
        s["p"], s["out"] = _params(c), torch.empty_like(q)
    elif k == "monitor":
        v = {"speed": sem.SEM_CRIT_SPEED, "vorticity": sem.SEM_CRIT_VORTICITY, "pv": sem.SEM_CRIT_PV}[c["criterion"]]
        thr = {"speed": THRESHOLDS, "vorticity": (1e-4, 3e-4, 1e-3), "pv": (2e-6, 4e-6, 8e-6)}[c["criterion"]]
        s["p"] = _params(c, thresholds=list(thr), lvl_max=3, criterion=[v] * 3)
        s["flags"] = torch.empty(m.Ne, dtype=torch.int8, device=DEV)
        s["cmax"] = torch.empty(m.Ne, dtype=torch.float64, device=DEV)
    elif k == "remesh":
        s["p"] = _params(c, thresholds=list(THRESHOLDS), lvl_max=3)
    elif k == "predict":
        s["net"] = sem.sem_mlp_create(11, 4096)
        s["feats"] = torch.empty((m.Ne, 136), dtype=torch.float32, device=DEV)
        s["prob"] = torch.empty((m.Ne, 3), dtype=torch.float32, device=DEV)
        s["flags"] = torch.empty(m.Ne, dtype=torch.int8, device=DEV)
    return s


def _next_run(s):
    """After RUN_STEPS steps the next run starts from the initial state."""
    s["left"] -= 1
    if s["left"] < 0:
        s["left"] = RUN_STEPS - 1
        many = isinstance(s["q"], list)
        for i in range(len(s["q"]) if many else 1):
            m, q, q0 = (s["meshes"][i], s["q"][i], s["q0"][i]) if many else (s["mesh"], s["q"], s["q0"])
            q.copy_(q0)
            if "q32" in s:
                sem.sem_mirror(m, q, s["q32"][i] if many else s["q32"])


def run(s):
    c, k = s["case"], s["case"]["kind"]
    if k == "step":
        _next_run(s)
        if c["form"] == "mixed":   # the new state as its float32 mirror, the precision of the step's arithmetic
            sem.sem_step_mixed(s["mesh"], s["p"], s["q"], s["q32"], s["work"], s["dt"])
            return {"q32": s["q32"]}
        sem.sem_step(s["mesh"], s["p"], s["q"], s["w1"], s["w2"], s["dt"])
        return {"q": s["q"]}
    if k == "rhs":
        return {"rhs": sem.sem_rhs(s["mesh"], s["p"], s["q"], s["out"])}
    if k == "batch":
        _next_run(s)
        sem.sem_batch_step_mixed(s["batch"], s["p"], s["q"], s["q32"], s["work"], s["dt"])
        return {"q32": s["q32"]}
    if k == "monitor":
        sem.sem_adapt_flags(s["mesh"], s["p"], s["q"], s["flags"], s["cmax"])
        d = sem.sem_diag(s["mesh"], s["p"], s["q"], 100.0e3)
        return {"flags": s["flags"], "cmax": s["cmax"], "wind": d["max_wind"], "mean_wind": d["max_mean_wind"]}
    if k == "remesh":
        flags = sem.sem_adapt_flags_host(s["mesh"], s["p"], s["q"])
        new = sem.sem_transfer_plan(s["mesh"], flags)
        q = torch.empty((5, new.NG), dtype=torch.float64, device=DEV)
        sem.sem_transfer(s["mesh"], new, s["q"], q)
        return {"flags": flags, "q": q}
    if k == "predict":
        sem.sem_mlp_features(s["mesh"], s["q"], SCALES, s["feats"])
        sem.sem_mlp_forward(s["net"], s["feats"], s["prob"])
        sem.sem_mlp_predict_flags(s["net"], s["feats"], s["flags"])
        return {"feats": s["feats"], "prob": s["prob"], "flags": s["flags"]}
    # train: gradients of the batch, then the update
    sem.sem_mlp_backward(s["net"], s["X"], s["y"], CLASS_W, want_loss=False)
    sem.sem_mlp_adam(s["net"], 1e-3)
    return {"grads": sem.sem_mlp_get_grads(s["net"])}


# --------------------------------------------------------------------------- work
def work(case):
    """Each input read once and each output written once; operations of the method."""
    c, k = case, case["kind"]
    if k == "train":
        n, par = c["rows"], 136 * 128 + 128 * 128 + 3 * 128 + 259
        return {"bytes": n * (136 * 4 + 1) + 4 * par * 7, "flops": 6.0 * n * (136 * 128 + 128 * 128 + 3 * 128)}
    if k == "batch":
        parts = [_step_work(i, _mesh(i), "mixed") for i in _instances(c)]
        return {"bytes": sum(p["bytes"] for p in parts), "flops": sum(p["flops"] for p in parts)}
    m = _mesh(c)
    NL = m.Ne * (m.N + 1) ** 3
    if k == "step":
        return _step_work(c, m, c["form"], c["terms"])
    if k == "rhs":
        one = _step_work(c, m, c["form"])
        return {"bytes": 80.0 * m.NG + 4.0 * m.Ncol * (m.N + 1) ** 2, "flops": one["flops"] / 3.0}
    if k == "monitor":
        f = 4 if c["criterion"] == "speed" else 5
        return {"bytes": 8.0 * f * m.NG + 9.0 * m.Ne, "flops": NL * (9.0 + (0.0 if f == 4 else 24.0 * (m.N + 1)))}
    if k == "remesh":   # about as many new nodes as old ones
        return {"bytes": 80.0 * m.NG + m.Ne, "flops": NL * 20.0 * (m.N + 1)}
    # predict: the samples are a part of the state's nodes at even orders
    nodes = min(1.0, (27.0 if m.N % 2 == 0 else (m.N + 1) ** 3) / (m.N + 1) ** 3)
    return {"bytes": 40.0 * m.NG * nodes + m.Ne * (136 * 4 + 3 * 4 + 1), "flops": 2.0 * 2 * m.Ne * 128 * (136 + 128 + 3)}


def _step_work(c, m, form, terms=False):
    NL = m.Ne * (m.N + 1) ** 3
    per = 30.0 * (m.N + 1) + 70.0 + (12.0 * (m.N + 1) + 40.0 if terms else 0.0)
    return {"bytes": (120.0 if form == "mixed" else 80.0) * m.NG + 4.0 * m.Ncol * (m.N + 1) ** 2, "flops": 3.0 * NL * per}


# --------------------------------------------------------------------------- exact values
class _Ref:
    """The discretisation in float64 torch on one mesh's numbering.  Local values
    are [..., column, b, a, layer, c] (a along x, b along y, c along z)."""

    def __init__(self, m, Lx, Ly, nx, ny):
        self.m, self.N, self.n1, self.nz, self.NZ, self.NH = m, m.N, m.N + 1, m.nz, int(m.NZ), int(m.NH)
        t = lambda a: torch.as_tensor(np.asarray(a), device=DEV)  # noqa: E731
        hmap, hh, hw = sem.sem_mesh_hmap_host(m)
        self.leaves = sem.sem_mesh_leaves_host(m)
        self.line = t(np.where(hmap >= 0, hmap, self.NH - 1 - hmap).astype(np.int64))
        self.hh, self.hw = t(hh.astype(np.int64)), t(hw)
        xi, w, D = _basis(self.N)
        self.xi, self.w, self.D = t(xi), t(w), t(D)
        lv = t(self.leaves[:, 0].astype(np.float64))
        five = (-1, 1, 1, 1, 1)
        self.hx, self.hy = (Lx / nx * 0.5 ** lv).reshape(five), (Ly / ny * 0.5 ** lv).reshape(five)
        self.Lx, self.Ly = Lx, Ly
        xyz = t(sem.sem_mesh_coords_host(m))
        self.x, self.y = xyz[0], xyz[1]
        self.z = self.local(xyz[2:3])[0]
        self.zx, self.zy, self.zz = self.d(self.z, 0), self.d(self.z, 1), self.d(self.z, 2)
        n = self.n1
        self.w3 = self.w.view(n, 1, 1, 1) * self.w.view(1, n, 1, 1) * self.w.view(1, 1, 1, n)
        self.wJ = self.w3 * self.hx * self.hy * 0.25 * self.zz
        self.mass = self.assemble(self.wJ[None])[0]

    def local(self, q):
        F = q.shape[0]
        q = q.reshape(F, self.NH, self.NZ)
        if len(self.hh):
            q = torch.cat([q, sum(self.hw[:, i, None] * q[:, self.hh[:, i]] for i in range(self.n1))], dim=1)
        q = q[:, self.line]                                     # [F, col, Nq, NZ]
        out = torch.stack([q[..., c:c + self.N * (self.nz - 1) + 1:self.N] for c in range(self.n1)], dim=-1)
        return out.reshape(F, -1, self.n1, self.n1, self.nz, self.n1)

    def assemble(self, r):
        F = r.shape[0]
        r = r.reshape(F, -1, self.nz, self.n1)                  # [F, lines, layer, c]
        col = torch.zeros((F, r.shape[1], self.NZ), dtype=r.dtype, device=DEV)
        for c in range(self.n1):
            col[..., c:c + self.N * (self.nz - 1) + 1:self.N] += r[..., c]
        out = torch.zeros((F, self.NH + len(self.hh), self.NZ), dtype=r.dtype, device=DEV)
        out.index_add_(1, self.line.reshape(-1), col)
        g = out[:, :self.NH].contiguous()
        for i in range(self.n1 if len(self.hh) else 0):
            g.index_add_(1, self.hh[:, i], self.hw[:, i, None] * out[:, self.NH:])
        return g.reshape(F, -1)

    def d(self, f, way):
        """Derivative along a reference direction (0: x, 1: y, 2: z)."""
        return torch.tensordot(f, self.D, dims=([(-3, -4, -1)[way]], [1])).movedim(-1, (-3, -4, -1)[way])

    def dt(self, f, way):
        return torch.tensordot(f, self.D, dims=([(-3, -4, -1)[way]], [0])).movedim(-1, (-3, -4, -1)[way])

    def grad(self, f):
        dz = self.d(f, 2) / self.zz
        return 2.0 / self.hx * (self.d(f, 0) - self.zx * dz), 2.0 / self.hy * (self.d(f, 1) - self.zy * dz), dz

    def weak(self, fx, fy, fz):
        a = self.w3 * 0.5 * self.hy * self.zz * fx
        b = self.w3 * 0.5 * self.hx * self.zz * fy
        e = self.w3 * (0.25 * self.hx * self.hy * fz - 0.5 * self.hy * self.zx * fx - 0.5 * self.hx * self.zy * fy)
        return self.dt(a, 0) + self.dt(b, 1) + self.dt(e, 2)

    def tendency(self, q, eqset, terms):
        L = self.local(q)
        th0, p0, rho0, rt0, dth0 = _reference(self.z)
        rp, rho, wJ = L[0], rho0 + L[0], self.wJ
        if eqset == "C":
            U, V, W, Tp = L[1], L[2], L[3], L[4]
            u, v, w = U / rho, V / rho, W / rho
            pp = p0 * torch.expm1(GAMMA * torch.log1p(Tp / rt0))
            rt = rt0 + Tp
            r = torch.stack([self.weak(U, V, W), self.weak(U * u + pp, U * v, U * w) + wJ * F0 * V,
                             self.weak(V * u, V * v + pp, V * w) - wJ * F0 * U,
                             self.weak(W * u, W * v, W * w + pp) - wJ * rp * G, self.weak(rt * u, rt * v, rt * w)])
        else:
            u, v, w, th = L[1], L[2], L[3], L[4]
            pp = p0 * torch.expm1(GAMMA * torch.log1p((rho0 * th + rp * (th0 + th)) / rt0))
            gp = self.grad(pp)
            adv = lambda f: sum(a * b for a, b in zip((u, v, w), self.grad(f)))  # noqa: E731
            r = torch.stack([self.weak(rho * u, rho * v, rho * w), wJ * (-adv(u) - gp[0] / rho + F0 * v),
                             wJ * (-adv(v) - gp[1] / rho - F0 * u), wJ * (-adv(w) - gp[2] / rho - rp / rho * G),
                             wJ * (-w * dth0 - adv(th))])
        if terms:
            gu, gv, gw = self.grad(u), self.grad(v), self.grad(w)
            sxy = 0.5 * (gu[1] + gv[0])
            nu = (0.21 * (self.hx + self.hy) / (2.0 * self.N)) ** 2 * torch.sqrt(
                2.0 * (gu[0] ** 2 + gv[1] ** 2 + 2.0 * sxy ** 2))
            k, zero = (rho if eqset == "C" else 1.0) * nu, torch.zeros_like(nu)
            r[1] += self.weak(-2.0 * k * gu[0], -2.0 * k * sxy, zero)
            r[2] += self.weak(-2.0 * k * sxy, -2.0 * k * gv[1], zero)
            r[3] += self.weak(-k * gw[0], -k * gw[1], zero)
            R = torch.clamp(torch.sin(0.5 * math.pi * (1.0 - (LZ - self.z) / 4000.0)) ** 2, max=1.0)
            r -= wJ * torch.where(self.z >= LZ - 4000.0, R, zero) * L
        T = self.assemble(r) / self.mass
        T.view(5, self.NH, self.NZ)[3, :, [0, self.NZ - 1]] = 0.0
        return T

    def step(self, q, dt, eqset, terms):
        f = lambda x: self.tendency(x, eqset, terms)  # noqa: E731
        q1 = q + dt * f(q)
        q2 = 0.75 * q + 0.25 * (q1 + dt * f(q1))
        return q / 3.0 + 2.0 / 3.0 * (q2 + dt * f(q2))

    def criterion(self, q, var):
        """Element maxima [Ne] of a criterion variable (conservative set)."""
        L = self.local(q)
        th0, p0, rho0, rt0, _ = _reference(self.z)
        rho = rho0 + L[0]
        if var == "speed":
            v = torch.sqrt(L[1] ** 2 + L[2] ** 2 + L[3] ** 2) / rho
        else:
            gu, gv, gw = self.grad(L[1] / rho), self.grad(L[2] / rho), self.grad(L[3] / rho)
            v = gv[0] - gu[1]
            if var == "pv":
                gt = self.grad((rt0 + L[4]) / rho)
                v = ((gw[1] - gv[2]) * gt[0] + (gu[2] - gw[0]) * gt[1] + (v + F0) * gt[2]) / rho
            v = v.abs()
        return v.amax(dim=(1, 2, 4)).reshape(-1)


def _lagrange(xi, x):
    """[len(x), len(xi)]: the nodal basis at x."""
    return np.array([[np.prod([(p - xi[m]) / (xi[j] - xi[m]) for m in range(len(xi)) if m != j])
                      for j in range(len(xi))] for p in x])


def _transferred(old, new, q):
    """Interpolation into refined columns, exact L2 projection into coarsened
    ones, then (Q^T W Q) q = Q^T W q_L by conjugate gradients."""
    xi = _basis(old.N)[0]
    gx, gw = np.polynomial.legendre.leggauss(old.N + 2)
    H = _lagrange(xi, gx)
    M = H.T @ (gw[:, None] * H)
    P = [_lagrange(xi, 0.5 * (xi + s)) for s in (-1.0, 1.0)]
    R = [np.linalg.solve(M, p.T @ M) for p in P]
    t = lambda a: torch.as_tensor(np.asarray(a), device=DEV)  # noqa: E731
    at = {tuple(x): i for i, x in enumerate(old.leaves.tolist())}
    L = old.local(q)
    out = torch.empty((5, len(new.leaves)) + tuple(L.shape[2:]), dtype=torch.float64, device=DEV)
    same, fine, coarse = [], {}, []
    for i, (l, a, b) in enumerate(new.leaves.tolist()):
        if (l, a, b) in at:
            same.append((i, at[l, a, b]))
        elif (l - 1, a >> 1, b >> 1) in at:
            fine.setdefault((a & 1, b & 1), []).append((i, at[l - 1, a >> 1, b >> 1]))
        else:
            coarse.append([i] + [at[l + 1, 2 * a + (s & 1), 2 * b + (s >> 1)] for s in range(4)])
    same = np.array(same).reshape(-1, 2)
    out[:, t(same[:, 0])] = L[:, t(same[:, 1])]
    both = lambda A, B, f: torch.einsum("im,jn,ocnmkz->ocjikz", t(A), t(B), f)  # noqa: E731
    for (a, b), pairs in fine.items():
        pairs = np.array(pairs)
        out[:, t(pairs[:, 0])] = both(P[a], P[b], L[:, t(pairs[:, 1])])
    if coarse:
        ix = np.array(coarse)
        out[:, t(ix[:, 0])] = 0.25 * sum(both(R[s & 1], R[s >> 1], L[:, t(ix[:, 1 + s])]) for s in range(4))
    rhs = new.assemble(new.wJ * out)
    A = lambda v: new.assemble(new.wJ * new.local(v))  # noqa: E731
    x = rhs / new.mass
    r = rhs - A(x)
    z = r / new.mass
    p, rz = z, (r * z).sum(dim=1, keepdim=True)
    for _ in range(200):
        if float(((r / new.mass) ** 2).sum().sqrt()) <= 1e-16 * float((x ** 2).sum().sqrt()):
            break
        Ap = A(p)
        den = (p * Ap).sum(dim=1, keepdim=True)
        alpha = rz / torch.where(den > 0, den, torch.ones_like(den))
        x, r = x + alpha * p, r - alpha * Ap
        z = r / new.mass
        rz2 = (r * z).sum(dim=1, keepdim=True)
        p, rz = z + rz2 / torch.where(rz > 0, rz, torch.ones_like(rz)) * p, rz2
    return x


def _bf16(x):
    return x.to(torch.float32).to(torch.bfloat16).to(torch.float64)


def _network(net):
    """The network's rounded weights and its biases, float64."""
    p = torch.as_tensor(sem.sem_mlp_get_params(net), device=DEV)
    out, at = [], 0
    for a, b in ((136, 128), (128, 128), (128, 3)):
        out.append(_bf16(p[at:at + a * b].reshape(a, b)))
        out.append(p[at + a * b:at + a * b + b].double())
        at += a * b + b
    return out


def _forward(X, par):
    """Inputs and hidden activations enter their products as bfloat16."""
    W1, b1, W2, b2, W3, b3 = par
    X = _bf16(X)
    H1 = _bf16(torch.relu(X @ W1 + b1))
    H2 = _bf16(torch.relu(H1 @ W2 + b2))
    return X, H1, H2, torch.softmax(H2 @ W3 + b3, dim=1)


def exact(case, seed):
    c, k = case, case["kind"]
    s = prepare(case, seed)
    if k == "train":
        par = _network(s["net"])
        X, H1, H2, prob = _forward(s["X"], par)
        y = s["y"].long()
        w = torch.tensor(CLASS_W, device=DEV).double()[y]
        one = torch.nn.functional.one_hot(y, 3).double()
        d3 = (w / w.sum())[:, None] * (prob - one)
        d2 = (d3 @ par[4].T) * (H2 > 0)
        d1 = (d2 @ par[2].T) * (H1 > 0)
        g = [X.T @ d1, d1.sum(0), H1.T @ d2, d2.sum(0), H2.T @ d3, d3.sum(0)]
        return {"grads": torch.cat([v.reshape(-1) for v in g])}
    if k == "batch":
        q = [_Ref(m, *_box(i), i["nx"], i["ny"]).step(x, dt, "C", False)
             for m, i, x, dt in zip(s["meshes"], s["cases"], s["q"], s["dt"])]
        return {"q32": q}
    R = _Ref(s["mesh"], *_box(c), c["nx"], c["ny"])
    if k == "step":
        q = R.step(s["q"], s["dt"], c["set"], c["terms"])
        return {"q32" if c["form"] == "mixed" else "q": q}
    if k == "rhs":
        return {"rhs": R.tendency(s["q"], c["set"], c["terms"])}
    if k == "monitor":
        q = s["q"]
        z = R.m.NZ
        near = ((R.x.abs() <= 100.0e3 + 1e-6) & (R.y.abs() <= 100.0e3 + 1e-6)).reshape(-1, z)
        rho = _reference(torch.as_tensor(sem.sem_mesh_coords_host(R.m)[2], device=DEV))[2] + q[0]
        v = (torch.sqrt(q[1] ** 2 + q[2] ** 2) / rho).reshape(-1, z)
        w = torch.where(near, R.mass.reshape(-1, z), torch.zeros_like(v))
        return {"flags": None, "cmax": R.criterion(q, c["criterion"]),
                "wind": float(torch.where(near, v, torch.zeros_like(v)).max()),
                "mean_wind": float(((w * v).sum(0) / w.sum(0)).max())}
    if k == "remesh":
        v = R.criterion(s["q"], "speed")
        lv = torch.as_tensor(np.repeat(R.leaves[:, 0], R.nz).astype(np.int64), device=DEV)
        thr = torch.tensor(THRESHOLDS, device=DEV).double()
        up = (lv < 3) & (v > thr[lv.clamp(max=2)])
        down = (lv > 0) & (v <= thr[(lv - 1).clamp(min=0)]) & ~up
        new = sem.sem_transfer_plan(s["mesh"], (up.to(torch.int8) - down.to(torch.int8)).cpu().numpy())
        return {"flags": None, "q": _transferred(R, _Ref(new, *_box(c), c["nx"], c["ny"]), s["q"])}
    # predict: the elements' polynomials at {-1, 0, 1}^3, then the network on them
    H = torch.as_tensor(_lagrange(_basis(R.N)[0], (-1.0, 0.0, 1.0)), device=DEV)
    T = torch.einsum("am,bn,cz,oenmkz->oekcba", H, H, H, R.local(s["q"]))
    T = T.reshape(5, -1, 27) / torch.tensor(SCALES, device=DEV).double()[:, None, None]
    lv = torch.as_tensor(np.repeat(R.leaves[:, 0], R.nz).astype(np.float64), device=DEV)
    X = torch.cat([T.movedim(0, 1).reshape(-1, 135), lv[:, None]], dim=1)
    return {"feats": X, "prob": _forward(X.float(), _network(s["net"]))[3], "flags": None}
