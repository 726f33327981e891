"""The work that users of this library have it do, as cases that can be timed and checked.

A case is one pass through the public entry points of paper_2105_01722_gb300.gdg
on a state that a program holds anyway: a context (or batch, or network) and its
fields on the device.  Kinds:

  march    gdg_step on a constant-coefficient Cartesian mesh, 1-D to 3-D
           (optionally followed by the energy reading of a monitored run)
  rate     gdg_rhs on such a mesh, for a caller with a time integrator of its own
  element  gdg_step on a mapped mesh with variable c^2: element PCG in FP64,
           FP32 PCG refined in FP64, or precomputed element inverses
  batch    gdg_batch_step: many small independent problems advanced together
  train    one minibatch of the learned initial guess: gradients and Adam update

exact() restates the method in plain FP64 torch: Galerkin-difference basis,
quadrature, fluxes, direct element solves, classic RK4.
"""
import math

import numpy as np
import torch

from paper_2105_01722_gb300 import gdg

FLUX = {"central": gdg.FLUX_CENTRAL, "upwind": gdg.FLUX_UPWIND, "alternating": gdg.FLUX_ALTERNATING}
# RK4 step over the cell width: inside the stability limit of every flux in 2-D
CFL = {1: 0.2, 3: 0.15, 5: 0.12, 7: 0.1}
BATCH_ROWS = 4096      # training rows the minibatches are drawn from


def listed():
    return [
        # the 1-D standing wave of the convergence studies, advanced between two outputs:
        # 144 unknowns a field, so nothing but latency and launches
        march("line_16", 16, steps=16, p=3, flux="central"),
        # a small odd plane mesh watched by its energy after every few steps
        march("plane_21x13_energy", 21, 13, steps=4, N=7, p=7, per="xy", energy=True),
        # the headline workload: 64 x 64 elements, p = 5, upwind, between two outputs
        march("plane_64", 64, 64, steps=32),
        # a plane mesh too large to stay on chip, ragged, low order, conservative flux, periodic in x
        march("plane_251x187", 251, 187, steps=4, N=9, p=3, flux="central", per="x"),
        # one time derivative for a caller's own integrator, alternating flux
        dict(march("rate_97x70", 97, 70, steps=0, flux="alternating", per="y"), kind="rate"),
        # the 3-D workload
        march("cube_32", 32, 32, 32, steps=1),
        # a small mapped problem with exact element solves: launches count
        element("mapped_inverse_12", 12, 12, "inverse", steps=8, p=3, flux="central"),
        # mapped elements with variable c^2, p = 5: the fastest form, advanced between two outputs
        element("mapped_inverse_128", 128, 128, "inverse", steps=4),
        # the iterative forms: plain FP64 PCG, and FP32 PCG refined in FP64
        element("mapped_pcg_128", 128, 128, "pcg"),
        element("mapped_mixed_128x120", 128, 120, "mixed", p=3),
        # an ensemble of small problems, constant and variable c^2 in turn, each too small for the GPU alone
        {"name": "batch_24", "kind": "batch", "count": 24, "low": 8, "high": 24, "solver": "mixed", "steps": 4, "pick": 5},
        # the inner loop of the learned guess's training
        {"name": "train_256", "kind": "train", "batch": 256},
    ]


def march(name, nx, ny=1, nz=1, steps=8, N=8, p=5, flux="upwind", per="", energy=False):
    return {"name": name, "kind": "march", "nx": nx, "ny": ny, "nz": nz, "steps": steps, "N": N, "p": p, "flux": flux,
            "per": per, "energy": energy}


def element(name, nx, ny, solver, steps=1, N=8, p=5, flux="upwind", per=""):
    return {"name": name, "kind": "element", "nx": nx, "ny": ny, "solver": solver, "steps": steps, "N": N, "p": p,
            "flux": flux, "per": per}


def draw(rng):
    kind = rng.choice(["line", "plane", "plane", "plane", "rate", "cube", "element", "element", "element", "batch", "train"])

    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    if kind == "train":
        return {"kind": "train", "batch": log(32, 1024)}
    if kind == "batch":
        low = rng.randint(6, 10)
        return {"kind": "batch", "count": rng.randint(8, 24), "low": low, "high": rng.randint(low + 4, 24),
                "solver": rng.choice(["pcg", "mixed", "inverse"]), "steps": rng.randint(1, 6), "pick": rng.randint(0, 999)}
    N = rng.choice([6, 7, 8, 8, 8, 9])
    c = {"N": N, "p": rng.choice([p for p in (1, 3, 3, 5, 5, 7) if p <= N]), "flux": rng.choice(["central", "upwind", "upwind", "alternating"])}
    if kind == "line":
        return {"kind": "march", "nx": log(8, 3000), "ny": 1, "nz": 1, **c, "per": rng.choice(["", "x"]), "steps": log(1, 32),
                "energy": False}
    if kind == "cube":
        n = log(4, 24)
        size = [max(2, n + rng.randint(-3, 4)) for _ in range(3)]
        return {"kind": "march", "nx": size[0], "ny": size[1], "nz": size[2], **c, "per": rng.choice(["", "x", "yz"]),
                "steps": rng.randint(1, 2), "energy": False}
    if kind == "element":
        nx = log(8, 100)
        ny = max(4, min(110, int(nx * rng.uniform(0.5, 1.5))))
        solver = rng.choice(["pcg", "mixed", "inverse"])
        return {"kind": "element", "nx": nx, "ny": ny, "solver": solver, **c, "p": max(3, c["p"]),
                "per": rng.choice(["", "", "x"]), "steps": {"pcg": 1, "mixed": rng.randint(1, 2), "inverse": rng.randint(1, 4)}[solver]}
    nx = log(10, 200)
    ny = max(5, min(200, int(nx * rng.uniform(0.5, 1.5))))
    plane = {"kind": "march", "nx": nx, "ny": ny, "nz": 1, **c, "per": rng.choice(["", "x", "y", "xy"]), "steps": log(1, 16),
             "energy": rng.random() < 0.25}
    return plane if kind == "plane" else dict(plane, kind="rate", steps=0, energy=False)


# ------------------------------------------------------------- inputs -------


def reference_nodes(n, N):
    """Per direction the GD node coordinates in [0, 1], laid out [ez, ey, ex, k, j, i]."""
    d = len(n)
    out = []
    for a in range(d):
        x = (np.arange(n[a])[:, None] + np.arange(N + 1)[None, :] / N) / n[a]
        shape = [1] * (2 * d)
        shape[d - 1 - a], shape[2 * d - 1 - a] = n[a], N + 1
        out.append(x.reshape(shape))
    return out


def fields(coords, seed):
    """A displacement and a velocity: a few standing modes and a pulse, from the seed."""
    rng = np.random.default_rng(seed)
    coords = [torch.as_tensor(x, device="cuda") for x in coords]
    out = []
    for _ in range(2):
        f = 0.0
        for _ in range(3):
            mode = float(rng.normal())
            for x in coords:
                mode = mode * torch.sin(int(rng.integers(1, 4)) * 2 * math.pi * x)
            f = f + mode
        r2, width = 0.0, float(rng.uniform(0.06, 0.2))
        for x in coords:
            r2 = r2 + ((x - float(rng.uniform(0.3, 0.7))) / width) ** 2
        out.append(f + torch.exp(-r2))
    return [f.contiguous().reshape(-1) for f in out]


def mapped(n, N, seed):
    """Nodes of the sine-mapped unit square and c^2 at them (host arrays, as gdg_create takes them)."""
    xi, eta = np.broadcast_arrays(*reference_nodes(n, N))
    x = xi + 0.05 * np.sin(2 * np.pi * xi) * np.sin(2 * np.pi * eta)
    phase = np.random.default_rng(seed + 77).uniform(0, 2 * np.pi)
    c2 = 1.0 + 0.5 * np.sin(2 * np.pi * x + phase) * np.cos(2 * np.pi * eta)
    return x, np.ascontiguousarray(eta), c2


def unmapped(n, N, seed):
    x, y = (np.ascontiguousarray(a) for a in np.broadcast_arrays(*reference_nodes(n, N)))
    rng = np.random.default_rng(seed + 77)
    s = sum(rng.uniform(-0.3, 0.3) * np.cos(2 * np.pi * a * x + rng.uniform(0, 6)) * np.cos(2 * np.pi * b * y + rng.uniform(0, 6))
            for a in range(2) for b in range(2))
    return x, y, 2.0 ** s


def mesh(case):
    """Elements, box and boundary kinds of a march, rate or element case."""
    n = tuple(case[k] for k in ("nx", "ny", "nz") if k in case)
    while len(n) > 1 and n[-1] == 1:
        n = n[:-1]
    hi = (1.0,) * len(n) if case["kind"] == "element" else tuple(m / n[0] for m in n)   # square cells
    bc = tuple(gdg.BC_PERIODIC if a in case["per"] else gdg.BC_DIRICHLET for a in "xyz"[: len(n)])
    return n, hi, bc


def time_step(case):
    n = max(case["nx"], case["ny"]) if case["kind"] == "element" else case["nx"]
    c = math.sqrt(1.5) if case["kind"] == "element" else math.sqrt(C2)
    return CFL[case["p"]] / (n * case["N"]) / c / (1.25 if case.get("nz", 1) > 1 else 1.0)


C2 = 1.3     # c^2 of the constant-coefficient cases
FORM = {"pcg": {}, "mixed": {"precision": gdg.MIXED}, "inverse": {"solver": gdg.SOLVE_INVERSE}}


def members(case, seed):
    """The problems of a batch case: (elements per direction, p, variable c^2?, dt, seed of its own)."""
    rng = np.random.default_rng(1000 + case["pick"])
    out = []
    for i in range(case["count"]):
        n, p = int(rng.integers(case["low"], case["high"] + 1)), int(rng.choice([3, 5, 7]))
        out.append((n, p, bool(i % 2), CFL[p] / (n * 8) / math.sqrt(2.5), seed * 100 + i))
    return out


def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        return prepare_train(case, seed)
    if kind == "batch":
        problems, us, vs, dts = [], [], [], []
        for n, p, variable, dt, own in members(case, seed):
            if variable:
                x, y, c2 = unmapped((n, n), 8, own)
                problems.append(gdg.make_problem(2, (n, n), 8, p, coef=gdg.COEF_NODAL, x_nodes=x, y_nodes=y, c2_nodes=c2,
                                                 pcg_rtol=1e-10, pcg_maxit=100, **FORM[case["solver"]]))
            else:
                problems.append(gdg.make_problem(2, (n, n), 8, p, c2=C2))
            u, v = fields(reference_nodes((n, n), 8), own)
            us.append(u)
            vs.append(v)
            dts.append(dt)
        return {"case": case, "batch": gdg.Batch(problems), "u": us, "v": vs, "dt": dts}
    n, hi, bc = mesh(case)
    if kind == "element":
        x, y, c2 = mapped(n, case["N"], seed)
        problem = gdg.make_problem(2, n, case["N"], case["p"], bc=bc, flux=FLUX[case["flux"]], coef=gdg.COEF_NODAL, x_nodes=x,
                                   y_nodes=y, c2_nodes=c2, pcg_rtol=1e-10, pcg_maxit=100, **FORM[case["solver"]])
    else:
        problem = gdg.make_problem(len(n), n, case["N"], case["p"], hi=hi, bc=bc, flux=FLUX[case["flux"]], c2=C2)
    u, v = fields(reference_nodes(n, case["N"]), seed)
    state = {"case": case, "ctx": gdg.Context(problem), "u": u, "v": v, "t": 0.0, "dt": time_step(case)}
    if kind == "rate":
        state.update(du=torch.empty_like(u), dv=torch.empty_like(v))
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "train":
        return run_train(state)
    u, v = state["u"], state["v"]
    if case["kind"] == "batch":
        state["batch"].step(u, v, state["dt"], case["steps"])
        return {"u": u, "v": v}
    if case["kind"] == "rate":
        state["ctx"].rhs(u, v, state["du"], state["dv"])
        return {"du": state["du"], "dv": state["dv"]}
    state["ctx"].step(u, v, state["t"], state["dt"], case["steps"])
    state["t"] += case["steps"] * state["dt"]
    out = {"u": u, "v": v}
    if case.get("energy"):
        out["energy"] = state["ctx"].energy(u, v)
    return out


# ----------------------------------------------------------- training -------


def training_state(case, seed):
    """Rows, and a network in the middle of its training: parameters, Adam moments, the minibatch's rows."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    c2 = 1.0 + 0.3 * torch.randn(BATCH_ROWS, gdg.MLP_OUT, device="cuda", generator=g)
    r = torch.randn(BATCH_ROWS, gdg.MLP_OUT, device="cuda", generator=g)
    X = torch.cat([c2, r / r.norm(dim=1, keepdim=True)], 1).contiguous()
    T = (0.3 * r / r.norm(dim=1, keepdim=True) + 0.02 * torch.randn(BATCH_ROWS, gdg.MLP_OUT, device="cuda", generator=g)).contiguous()
    parts = []
    for a, b in ((gdg.MLP_IN, gdg.MLP_HID), (gdg.MLP_HID, gdg.MLP_HID), (gdg.MLP_HID, gdg.MLP_OUT)):
        parts += [(2 * torch.rand(b * a, device="cuda", generator=g) - 1) * math.sqrt(6.0 / (a + b)),
                  0.05 * torch.randn(b, device="cuda", generator=g)]
    params = torch.cat(parts)
    m = 1e-3 * torch.randn(params.numel(), device="cuda", generator=g)
    v = (1e-3 * (1.0 + torch.rand(params.numel(), device="cuda", generator=g))) ** 2
    rows = torch.randperm(BATCH_ROWS, device="cuda", generator=g)[: case["batch"]].to(torch.int32)
    return X, T, params, m, v, rows


LR, STEPS_DONE = 2e-5, 400     # late in a decayed schedule


def prepare_train(case, seed):
    X, T, params, m, v, rows = training_state(case, seed)
    net = gdg.Mlp(params)
    net.m.copy_(m)
    net.v.copy_(v)
    net.step_count = STEPS_DONE
    return {"case": case, "net": net, "X": X, "T": T, "rows": rows}


def run_train(state):
    net = state["net"]
    loss = net.backward(state["X"], state["T"], state["rows"])
    net.adam(LR)
    return {"loss": loss, "grad": net.grad, "params": net.params, "m": net.m, "v": net.v, "weights": net.wbf16.view(torch.bfloat16)}


def exact_train(case, seed):
    X, T, params, m, v, rows = training_state(case, seed)
    sizes = ((gdg.MLP_HID, gdg.MLP_IN), (gdg.MLP_HID, gdg.MLP_HID), (gdg.MLP_OUT, gdg.MLP_HID))
    W, b, at = [], [], 0
    for o, i in sizes:     # the kernels multiply by BF16 weights, the biases stay FP32
        W.append(params[at : at + o * i].to(torch.bfloat16).double().view(o, i).requires_grad_())
        b.append(params[at + o * i : at + o * i + o].double().requires_grad_())
        at += o * i + o
    x, t = X[rows.long()].double(), T[rows.long()].double()
    h = torch.tanh(x @ W[0].T + b[0])
    h = torch.tanh(h @ W[1].T + b[1])
    loss = ((h @ W[2].T + b[2] - t) ** 2).sum() / len(rows)
    loss.backward()
    grad = torch.cat([g.grad.reshape(-1) for pair in zip(W, b) for g in pair])
    step = STEPS_DONE + 1
    m = 0.9 * m.double() + 0.1 * grad
    v = 0.999 * v.double() + 0.001 * grad**2
    params = params.double() - LR * (m / (1 - 0.9**step)) / (torch.sqrt(v / (1 - 0.999**step)) + 1e-8)
    return {"loss": loss.detach().reshape(1), "grad": grad, "params": params, "m": m, "v": v, "weights": None}


# --------------------------------------------------------------- work -------


def work(case):
    kind = case["kind"]
    if kind == "train":
        macs = gdg.MLP_IN * gdg.MLP_HID + gdg.MLP_HID**2 + gdg.MLP_HID * gdg.MLP_OUT
        back = 2 * macs - gdg.MLP_IN * gdg.MLP_HID          # no gradient for the inputs
        rows = case["batch"] * (gdg.MLP_IN + gdg.MLP_OUT + 1) * 4
        return {"bytes": rows + gdg.MLP_NPARAM * 4 * 7 + gdg.MLP_NWEIGHT * 4, "flops": 2.0 * case["batch"] * (macs + back)}
    if kind == "batch":
        total = {"bytes": 0.0, "flops": 0.0}
        for n, p, variable, _, _ in members(case, 0):
            one = {"kind": "element" if variable else "march", "nx": n, "ny": n, "nz": 1, "N": 8, "p": p, "steps": case["steps"],
                   "solver": case["solver"], "per": ""}
            for k, w in work(one).items():
                total[k] += w
        return total
    n, _, _ = mesh(case)
    ne, n1, stages = math.prod(n), case["N"] + 1, 4 * case["steps"] if case["steps"] else 1
    na = n1 ** len(n)
    state = 4.0 * 8 * ne * na                               # both fields, in and out
    if kind in ("march", "rate"):
        # traces, fluxes, lifts, diagonal solves and the stage update, per unknown of a field pair
        per = {1: 30.0, 2: 40.0, 3: 34.0 + 66.0 / n1}[len(n)]
        back = 8.0 * len(n) * n1 * ne * na                  # to the modified basis and back, both fields
        return {"bytes": state, "flops": per * ne * na * stages + back}
    faces = 144.0 * n1 * n1 + 16 * na                       # face operators, lifts, stage update
    matrix = 2.0 * na * na                                  # one product with an element matrix
    if case["solver"] == "inverse":
        return {"bytes": state + 8.0 * ne * ((12 * n1 + na) * na + 72 * n1 * n1), "flops": ne * stages * (faces + 2.0 * (12 * n1 + na) * na)}
    # iterations to 1e-10 of the two element systems on these meshes: about 9 and 4.5 in FP64 (one product and one
    # preconditioner each), two refinement residuals each in the mixed form
    solves = 13.5 * (matrix + 8.0 * n1**3) if case["solver"] == "pcg" else 4 * matrix
    return {"bytes": state + 8.0 * ne * (na * (na + 1) + 72 * n1 * n1), "flops": ne * stages * (faces + matrix + solves)}


# ------------------------------------------------- the method in 64 bits ----


def basis(p, N):
    """1-D Galerkin-difference basis on [0, 1]: values B and slopes D at the composite Gauss points (weights w),
    and the one-sided slopes at both ends."""
    def on_cell(k, r):
        s = min(max(k - (p + 1) // 2 + 1, 0), N - p)
        x = np.arange(s, s + p + 1) / N
        val, der = np.zeros(N + 1), np.zeros(N + 1)
        for m in range(p + 1):
            others = np.delete(np.arange(p + 1), m)
            val[s + m] = np.prod((r - x[others]) / (x[m] - x[others]))
            der[s + m] = sum(np.prod((r - x[np.setdiff1d(others, [q])]) / (x[m] - x[np.setdiff1d(others, [q])])) / (x[m] - x[q])
                             for q in others)
        return val, der

    gx, gw = np.polynomial.legendre.leggauss(p + 1)
    rows = [on_cell(k, (k + 0.5 * (g + 1)) / N) for k in range(N) for g in gx]
    B, D = (np.array([r[i] for r in rows]) for i in range(2))
    return B, D, np.tile(0.5 * gw / N, N), on_cell(0, 0.0)[1], on_cell(N - 1, 1.0)[1]


def cuda(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def rk4(rate, y, dt, steps):
    add = lambda a, b, c: tuple(p + c * q for p, q in zip(a, b))  # noqa: E731
    for _ in range(steps):
        k1 = rate(y)
        k2 = rate(add(y, k1, dt / 2))
        k3 = rate(add(y, k2, dt / 2))
        k4 = rate(add(y, k3, dt))
        y = tuple(a + dt / 6 * (p + 2 * q + 2 * r + s) for a, p, q, r, s in zip(y, k1, k2, k3, k4))
    return y


def fluxes(kind, side, vi, di, vo, do, beta, tau, wall):
    """v* - v_in and q* of one face; vo, do hold the mirror state where `wall`."""
    if kind != "alternating":
        return 0.5 * (vo - vi) - beta * (di + do), 0.5 * (di - do) - tau * (vi - vo)
    zero = torch.zeros_like(vi)
    g, q = (vo - vi, di) if side == 0 else (zero, -do)
    return torch.where(wall, -vi, g), torch.where(wall, di, q)


class Modal:
    """Constant c^2 on a Cartesian box, in the basis that diagonalises mass and stiffness per direction."""

    def __init__(self, n, N, p, hi, per, flux, c2):
        self.n, self.n1, self.d, self.per, self.flux, self.c2 = n, N + 1, len(n), per, flux, c2
        B, D, w, sL, sR = basis(p, N)
        M, S = B.T @ (w[:, None] * B), D.T @ (w[:, None] * D)
        Li = np.linalg.inv(np.linalg.cholesky(M))
        lam, Y = np.linalg.eigh(Li @ S @ Li.T)
        Psi = Li.T @ Y
        Psi[:, 0], lam[0] = 1.0 / math.sqrt(M.sum()), 0.0
        self.beta, self.tau = (0.5 * math.sqrt(c2), 0.5 / math.sqrt(c2)) if flux == "upwind" else (0.0, 0.0)
        self.to, self.back, self.e, self.g = [], [], [], []
        shape = [1] * (2 * self.d)
        self.lam = torch.zeros(shape, dtype=torch.float64, device="cuda")
        for a in range(self.d):
            H = hi[a] / n[a]
            P = Psi / math.sqrt(H)
            self.to.append(cuda(P.T @ (H * M)))
            self.back.append(cuda(P))
            self.e.append((cuda(P[0]), cuda(P[-1])))
            self.g.append((cuda(-sL @ P / H), cuda(sR @ P / H)))
            s = list(shape)
            s[2 * self.d - 1 - a] = self.n1
            self.lam = self.lam + cuda(lam / H**2).reshape(s)
        self.inv = torch.where(self.lam > 0, 1.0 / self.lam.clamp_min(1e-300), torch.zeros_like(self.lam))

    def transform(self, f, mats):
        f = f.reshape(*reversed(self.n), *([self.n1] * self.d))
        for a in range(self.d):
            ax = 2 * self.d - 1 - a
            f = torch.tensordot(f, mats[a], dims=([ax], [1])).movedim(-1, ax)
        return f

    def rate(self, y):
        U, V = y
        ru, rv = torch.zeros_like(U), -self.c2 * self.lam * U
        for a in range(self.d):
            ax, ex = 2 * self.d - 1 - a, self.d - 1 - a
            v = [torch.tensordot(V, self.e[a][s], dims=([ax], [0])) for s in (0, 1)]
            d = [torch.tensordot(U, self.g[a][s], dims=([ax], [0])) for s in (0, 1)]
            for s in (0, 1):
                vo, do = (f[1 - s].roll(1 - 2 * s, ex) for f in (v, d))
                wall = torch.zeros([self.n[a] if i == ex else 1 for i in range(v[s].dim())], dtype=torch.bool, device="cuda")
                if "xyz"[a] not in self.per:
                    wall.select(ex, 0 if s == 0 else self.n[a] - 1).fill_(True)
                vo, do = torch.where(wall, -v[s], vo), torch.where(wall, -d[s], do)
                g, q = fluxes(self.flux, s, v[s], d[s], vo, do, self.beta, self.tau, wall)
                shape = [1] * (2 * self.d)
                shape[ax] = self.n1
                ru += g.unsqueeze(ax) * self.g[a][s].reshape(shape)
                rv += self.c2 * q.unsqueeze(ax) * self.e[a][s].reshape(shape)
        return V + self.inv * ru, rv

    def energy(self, y):
        return float(0.5 * ((y[1] ** 2).sum() + self.c2 * (self.lam * y[0] ** 2).sum()))


class Elements:
    """Variable c^2 on mapped elements: quadrature assembly and direct element solves."""

    def __init__(self, n, N, p, x, y, c2, per, flux):
        self.n, n1, self.flux = n, N + 1, flux
        self.n1 = n1
        B, D, w, sL, sR = (cuda(a) for a in basis(p, N))
        self.B, self.D, self.slope = B, D, (sL, sR)
        x, y, c2 = (cuda(a).reshape(-1, n1, n1) for a in (x, y, c2))
        ne, na = x.shape[0], n1 * n1
        Phi, Gr, Gs, W = torch.kron(B, B), torch.kron(B, D), torch.kron(D, B), torch.kron(w, w)
        self.M, self.A = (torch.empty(ne, na, na, dtype=torch.float64, device="cuda") for _ in range(2))
        for i in range(0, ne, 64):
            X, Y, C = (f[i : i + 64].reshape(-1, na) for f in (x, y, c2))
            xr, xs, yr, ys, c = X @ Gr.T, X @ Gs.T, Y @ Gr.T, Y @ Gs.T, C @ Phi.T
            det = xr * ys - xs * yr
            M = (Phi.T * (W * det)[:, None, :]) @ Phi
            k = W * c / det
            mixed = (Gr.T * (-k * (xr * xs + yr * ys))[:, None, :]) @ Gs
            S = (Gr.T * (k * (xs**2 + ys**2))[:, None, :]) @ Gr + (Gs.T * (k * (xr**2 + yr**2))[:, None, :]) @ Gs + mixed + mixed.mT
            one = M.sum(2) / (W * det).sum(1, keepdim=True)
            self.M[i : i + 64], self.A[i : i + 64] = M, S + one[:, :, None] * one[:, None, :]
            if i == 0:
                self.w = torch.empty(ne, na, dtype=torch.float64, device="cuda")
            self.w[i : i + 64] = one
        self.LM, self.LA = torch.linalg.cholesky(self.M), torch.linalg.cholesky(self.A)
        ex, ey = torch.arange(ne, device="cuda") % n[0], torch.arange(ne, device="cuda") // n[0]
        self.faces = []
        for f in range(4):     # x-, x+, y-, y+
            a, s = f // 2, f % 2
            slope, edge = self.slope[s], (0 if s == 0 else n1 - 1)
            lines = []
            for g in (x, y):
                normal = torch.tensordot(g, slope, dims=([2 if a == 0 else 1], [0])) @ B.T
                along = (g[:, :, edge] if a == 0 else g[:, edge, :]) @ D.T
                lines.append((normal, along) if a == 0 else (along, normal))
            (xr, xs), (yr, ys) = lines
            T = torch.sqrt(xs**2 + ys**2) if a == 0 else torch.sqrt(xr**2 + yr**2)
            nx_, ny_ = (ys / T, -xs / T) if a == 0 else (-yr / T, xr / T)
            if s == 0:
                nx_, ny_ = -nx_, -ny_
            det = xr * ys - xs * yr
            cf = (c2[:, :, edge] if a == 0 else c2[:, edge, :]) @ B.T
            e2 = (ex if a == 0 else ey) + (2 * s - 1)
            wall = (e2 < 0) | (e2 >= n[a])
            if "xy"[a] in per:
                wall = torch.zeros_like(wall)
            e2 = e2 % n[a]
            other = ey * n[0] + e2 if a == 0 else e2 * n[0] + ex
            c = torch.sqrt(cf)
            up = 1.0 if flux == "upwind" else 0.0
            self.faces.append((a, s, slope, edge, (ys * nx_ - xs * ny_) / det, (xr * ny_ - yr * nx_) / det, cf * T * w, 0.5 * c * up,
                               0.5 / c * up, wall[:, None], other))

    def rate(self, y):
        n1 = self.n1
        U, V = (f.reshape(-1, n1, n1) for f in y)
        v, d = [], []
        for a, s, slope, edge, fr, fs, *_ in self.faces:
            v.append((V[:, :, edge] if a == 0 else V[:, edge, :]) @ self.B.T)
            normal = torch.tensordot(U, slope, dims=([2 if a == 0 else 1], [0])) @ self.B.T
            along = (U[:, :, edge] if a == 0 else U[:, edge, :]) @ self.D.T
            d.append(fr * normal + fs * along if a == 0 else fr * along + fs * normal)
        flat = U.reshape(-1, n1 * n1, 1)
        SU = self.A @ flat - self.w[:, :, None] * (self.w[:, None, :] @ flat)
        ru, rv = torch.zeros_like(U), -SU.reshape(U.shape)
        for f, (a, s, slope, edge, fr, fs, cw, beta, tau, wall, other) in enumerate(self.faces):
            vo, do = torch.where(wall, -v[f], v[f ^ 1][other]), torch.where(wall, -d[f], d[f ^ 1][other])
            g, q = fluxes(self.flux, s, v[f], d[f], vo, do, beta, tau, wall)
            normal, along = ((cw * fr * g), (cw * fs * g)) if a == 0 else ((cw * fs * g), (cw * fr * g))
            if a == 0:
                ru += (normal @ self.B)[:, :, None] * slope
                ru[:, :, edge] += along @ self.D
                rv[:, :, edge] += (cw * q) @ self.B
            else:
                ru += (normal @ self.B)[:, None, :] * slope[:, None]
                ru[:, edge, :] += along @ self.D
                rv[:, edge, :] += (cw * q) @ self.B

        def solve(L, b):
            z = torch.linalg.solve_triangular(L, b.reshape(-1, n1 * n1, 1), upper=False)
            return torch.linalg.solve_triangular(L.mT, z, upper=True)

        return y[1] + solve(self.LA, ru).reshape(-1), solve(self.LM, rv).reshape(-1)


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return exact_train(case, seed)
    if kind == "batch":
        out = {"u": [], "v": []}
        for n, p, variable, dt, own in members(case, seed):
            u, v = march_exact((n, n), p, 8, dt, case["steps"], own, variable)
            out["u"].append(u)
            out["v"].append(v)
        return out
    n, hi, _ = mesh(case)
    y = tuple(fields(reference_nodes(n, case["N"]), seed))
    if kind == "element":
        op = Elements(n, case["N"], case["p"], *mapped(n, case["N"], seed), case["per"], case["flux"])
        u, v = rk4(op.rate, y, time_step(case), case["steps"])
        return {"u": u, "v": v}
    op = Modal(n, case["N"], case["p"], hi, case["per"], case["flux"], C2)
    y = tuple(op.transform(f, op.to) for f in y)
    if kind == "rate":
        du, dv = (op.transform(f, op.back).reshape(-1) for f in op.rate(y))
        return {"du": du, "dv": dv}
    y = rk4(op.rate, y, time_step(case), case["steps"])
    u, v = (op.transform(f, op.back).reshape(-1) for f in y)
    return {"u": u, "v": v, "energy": op.energy(y)} if case.get("energy") else {"u": u, "v": v}


def march_exact(n, p, N, dt, steps, seed, variable):
    """One problem of a batch."""
    y = tuple(fields(reference_nodes(n, N), seed))
    if variable:
        op = Elements(n, N, p, *unmapped(n, N, seed), "", "upwind")
        return rk4(op.rate, y, dt, steps)
    op = Modal(n, N, p, (1.0, 1.0), "", "upwind", C2)
    y = rk4(op.rate, tuple(op.transform(f, op.to) for f in y), dt, steps)
    return tuple(op.transform(f, op.back).reshape(-1) for f in y)
