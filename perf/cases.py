"""The work a user of this library has it do, as cases that can be timed and checked: whole solves
(multigrid in its three precisions, line-preconditioned CG, the batched solver, the cubed-sphere
panel), single kernels of the method, and the learned stage's network in inference and training.

A case is a dict of plain values. listed() gives the fixed ones, draw(rng) one more of the same
ranges; prepare(case, seed) makes operators, workspace and inputs on the GPU, run(state) is one pass
through the public entry points, work(case) the bytes and operations such a pass cannot do without,
and exact(case, seed) the same outputs from plain torch in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1402_3545_gb300 import tpmg

RHO = 0.8       # relaxation of the library's default parameters
OMEGA2 = 1e-2   # omega^2 of the benchmark problems

# Every case names its kind and sizes; "lam" is lambda^2 (0: the column-varying field of the mid-size
# benchmark), "cfl" a horizontal CFL number that sets omega = cfl h / 2 instead of OMEGA2.
CASES = [
    # the plain method's small configuration: a whole solve of 0.26 M cells, bound by latency and launches
    dict(name="mg_small_f64", kind="solve", method="mg", prec="f64", nx=64, ny=64, nz=64, levels=4, lam=1e3,
         cfl=0.0, tol=1e-6),
    # the benchmark's headline: 512^2 x 128, lambda^2 varying by column, native FP64 multigrid to 1e-6
    dict(name="mg_mid_f64", kind="solve", method="mg", prec="f64", nx=512, ny=512, nz=128, levels=7, lam=0.0,
         cfl=0.0, tol=1e-6),
    # the same problem in the library's default precision (double-word)
    dict(name="mg_mid_dw", kind="solve", method="mg", prec="dw", nx=512, ny=512, nz=128, levels=7, lam=0.0,
         cfl=0.0, tol=1e-6),
    # the largest plain problem of the benchmark: 134 M cells, FP32 V-cycles inside double-word refinement
    dict(name="mg_large_mixed", kind="solve", method="mg", prec="mixed", nx=1024, ny=1024, nz=128, levels=8,
         lam=1e4, cfl=0.0, tol=1e-10),
    # the method's other solver on the paper-shaped problem (omega = 4.2 h), to the paper's 1e-5
    dict(name="cg_paper_dw", kind="solve", method="cg", prec="dw", nx=512, ny=512, nz=128, levels=5, lam=1e3,
         cfl=8.4, tol=1e-5),
    # many problems of uneven size in one persistent launch
    dict(name="mg_batched", kind="batched", nprob=12, pseed=0, tol=1e-9),
    # the paper's own operator: one gnomonic cubed-sphere panel, V(1,1), rho = 2/3, to 1e-5
    dict(name="mg_panel_f64", kind="panel", prec="f64", nx=512, ny=512, nz=128, levels=5, tol=1e-5),
    # one smoothing step of the mixed solver's inner cycle, per-column lambda^2
    dict(name="smooth_f32", kind="smooth", prec="f32", nx=512, ny=512, nz=128, lam=0.0, norm=False),
    # a smoothing step with its residual norm on a grid that fits no tile
    dict(name="smooth_ragged_f64", kind="smooth", prec="f64", nx=300, ny=150, nz=60, lam=0.0, norm=True),
    # the transfers between two levels: residual + restriction + first coarse step, and prolongation
    dict(name="transfer_f32", kind="transfer", prec="f32", nx=1024, ny=512, nz=64, lam=1e3),
    # the learned stage applied: a forward pass of the network (its application grid is 2048^2 x 64)
    dict(name="nn_forward", kind="forward", cin=2, nx=1024, ny=512, nz=64),
    # a training step's gradient on the training crop: forward, residual loss and backward
    dict(name="nn_train", kind="train", cin=2, nx=256, ny=256, nz=64),
]


def listed():
    return [dict(c) for c in CASES]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ones' ranges. Solver grids are b 2^(L-1) cells across with 8 <= b <=
    15 (odd coarsest grids among them), unit kernels take any size, the network its multiples of 64."""
    kind = rng.choice(["solve", "solve", "solve", "batched", "panel", "smooth", "smooth", "transfer", "forward", "train"])
    lam = rng.choice([0.0, 10.0 ** rng.uniform(2.0, 4.0)])
    if kind == "solve":
        method, prec = rng.choice([("mg", "f64"), ("mg", "dw"), ("mg", "mixed"), ("cg", "f64"), ("cg", "dw")])
        cap = {"f64": 1 << 24 if method == "cg" else 1 << 25, "dw": 1 << 25, "mixed": 1 << 27}[prec]
        while True:
            L = rng.randint(3, 7)
            nx, ny = (rng.randint(8, 15) << (L - 1) for _ in range(2))
            nz = _log_int(rng, 16, 160)
            if nx <= 2 * ny and ny <= 2 * nx and nx * ny * nz <= cap:
                break
        return dict(kind=kind, method=method, prec=prec, nx=nx, ny=ny, nz=nz, levels=L, lam=lam,
                    cfl=8.4 if method == "cg" else 0.0,
                    tol=1e-5 if method == "cg" else 1e-10 if prec == "mixed" else 1e-6)
    if kind == "batched":
        return dict(kind=kind, nprob=rng.randint(2, 10), pseed=rng.randint(1, 10 ** 6), tol=1e-9)
    if kind == "panel":
        L = rng.randint(3, 6)
        b, prec = rng.randint(8, 15) << (L - 1), rng.choice(["f64", "mixed"])
        return dict(kind=kind, prec=prec, nx=b, ny=b, nz=_log_int(rng, 16, 128), levels=L,
                    tol=1e-10 if prec == "mixed" else 1e-5)
    if kind in ("smooth", "transfer"):
        prec = rng.choice(["f64", "f32", "dw"])
        while True:
            m = rng.choice([1, 32, 64, 128]) if kind == "smooth" else 2 * rng.choice([1, 32])
            nx, ny = (max(m, _log_int(rng, 40, 1000) // m * m) for _ in range(2))
            nz = min(_log_int(rng, 8, 200), (1 << 25) // (nx * ny))
            # FP32 works on levels whose column blocks are as well conditioned as the finest ones of the
            # benchmark problems (lambda^2 (h / hz)^2 about 100)
            if prec != "f32" or (lam or 1e3) * (nz / max(nx, ny)) ** 2 <= 100.0:
                break
        case = dict(kind=kind, prec=prec, nx=nx, ny=ny, nz=nz, lam=lam)
        return dict(case, norm=rng.random() < 0.25) if kind == "smooth" else case
    while True:
        nx, ny, nz = 64 * rng.randint(1, 16), 2 * _log_int(rng, 16, 512), _log_int(rng, 8, 64)
        if 1 << 16 <= nx * ny * nz <= (1 << 25 if kind == "forward" else 1 << 22):
            return dict(kind=kind, cin=rng.choice([1, 2]), nx=nx, ny=ny, nz=nz)


# ---------------------------------------------------------------- problems
def _problem(case):
    """(omega2, hx, hy, hz, lambda^2 scalar or (ny, nx) field): square cells on the unit box."""
    nx, ny = case["nx"], case["ny"]
    h = 1.0 / max(nx, ny)
    lam = case.get("lam", 1e3)
    if lam == 0.0:
        x, y = (np.arange(nx) + 0.5) / nx, (np.arange(ny) + 0.5) / ny
        lam = 1e3 * (1.0 + 0.5 * np.sin(2 * np.pi * x)[None, :] * np.cos(2 * np.pi * y)[:, None])
    w = OMEGA2 if case.get("cfl", 0.0) == 0.0 else (0.5 * case["cfl"] * h) ** 2
    return w, h, h, 1.0 / case["nz"], lam


def _batch(case):
    """The batched workload's problems: sizes uniform in {64, ..., 512}^2 x {32, 64, 128}, lambda^2
    log-uniform in [1e2, 1e4]; one problem's case each."""
    rng = np.random.default_rng(case["pseed"])
    out = []
    for _ in range(case["nprob"]):
        nx, ny = (int(rng.choice([64, 128, 256, 512])) for _ in range(2))
        nz, lam, L, a, b = int(rng.choice([32, 64, 128])), float(10.0 ** rng.uniform(2.0, 4.0)), 1, nx, ny
        while a % 2 == 0 and b % 2 == 0 and max(a, b) > 8:
            a, b, L = a // 2, b // 2, L + 1
        out.append(dict(nx=nx, ny=ny, nz=nz, levels=L, lam=lam))
    return out


def _panel_numbers(case):
    """omega2, lambda2, H of the paper's configuration on an nx x ny panel (nu_CFL = 8.4)."""
    h = 0.5 * np.pi / case["nx"]
    return (0.5 * 8.4 * h) ** 2, 1.0, 10.0 / 6371.0


def _net_params(cin, seed):
    """He-normal weights, small biases: a network as training starts from."""
    rng = np.random.default_rng(seed)
    parts = []
    for ci, co in ((cin, 16), (16, 16), (16, 16), (16, 1)):
        parts += [rng.standard_normal(co * ci * 27) * math.sqrt(2.0 / (27 * ci)), 0.05 * rng.standard_normal(co)]
    return np.concatenate(parts).astype(np.float32)


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _normal(g, shape, dtype=torch.float64):
    return torch.randn(shape, generator=g, device="cuda", dtype=dtype)


def _rhs(g, shape):
    f = _normal(g, shape)
    return f.sub_(f.mean())


def _shape(case):
    return (case["nz"], case["ny"], case["nx"])


def _unit_fields(case, seed):
    """u and f as a smoothing step meets them: f of unit size, u such that A u is of f's size."""
    w, hx, _, hz, lam = _problem(case)
    scale = 1.0 / (1.0 + 4.0 * w / hx ** 2 + 2.0 * w * float(np.mean(lam)) / hz ** 2)
    g = _gen(seed)
    dt = torch.float32 if case["prec"] == "f32" else torch.float64
    u, f = _normal(g, _shape(case)).mul_(scale).to(dt), _normal(g, _shape(case)).to(dt)
    w0 = _normal(g, _shape(case)).mul_(scale).to(dt) if case["kind"] == "transfer" else None
    return u, f, w0


def _net_input(case, seed):
    """Channel 0 a residual of unit mean square, channel 1 (two-channel networks) log10(lambda^2) - 3."""
    x = torch.empty(_shape(case) + (case["cin"],), device="cuda", dtype=torch.float32)
    x[..., 0] = _normal(_gen(seed), _shape(case), torch.float32)
    if case["cin"] == 2:
        x[..., 1] = math.log10(_crop_lam(seed)) - 3.0
    return x


def _crop_lam(seed):
    return float(10.0 ** np.random.default_rng(seed + 7).uniform(2.0, 4.0))


def _params(case, **kw):
    return tpmg.default_params(prec=case["prec"], tol=case["tol"], zero_guess=1, max_iter=400, **kw)


# ---------------------------------------------------------------- prepare and run
def prepare(case, seed):
    kind = case["kind"]
    s = {"case": case}
    if kind in ("solve", "smooth", "transfer"):
        op = tpmg.Operator(case["nx"], case["ny"], case["nz"], *_problem(case),
                           nlevels=case.get("levels", 1 if kind == "smooth" else 2))
        s["op"] = op
        tpmg.op_reserve(op.op, tpmg.PREC[case["prec"]])
        if kind == "solve":
            s["f"] = _rhs(_gen(seed), _shape(case))
            s["u"] = torch.empty_like(s["f"])
            s["prm"] = _params(case)
        else:
            s["u"], s["f"], s["w"] = _unit_fields(case, seed)
            s["out"] = torch.empty_like(s["u"])
            s["norm"] = torch.zeros(1, dtype=torch.float64, device="cuda")
            if kind == "transfer":
                s["fc"] = torch.empty(op.level_shape(1), dtype=s["u"].dtype, device="cuda")
                s["uc"] = torch.empty_like(s["fc"])
    elif kind == "batched":
        g = _gen(seed)
        probs = _batch(case)
        s["ops"] = [tpmg.Operator(p["nx"], p["ny"], p["nz"], *_problem(p), nlevels=p["levels"]) for p in probs]
        for op in s["ops"]:
            tpmg.op_reserve(op.op, tpmg.MIXED)
        s["handles"] = [op.op for op in s["ops"]]
        s["f"] = [_rhs(g, _shape(p)) for p in probs]
        s["u"] = [torch.empty_like(f) for f in s["f"]]
        s["prm"] = tpmg.default_params(prec="mixed", tol=case["tol"], zero_guess=1, max_iter=200)
    elif kind == "panel":
        w, lam, H = _panel_numbers(case)
        s["op"] = tpmg.PanelOperator(case["nx"], case["ny"], case["nz"], w, lam, H, nlevels=case["levels"])
        s["f"] = _normal(_gen(seed), _shape(case))
        s["u"] = torch.empty_like(s["f"])
        s["prm"] = _params(case, nu_pre=1, nu_post=1, rho=2.0 / 3.0)
    else:
        s["net"] = tpmg.Network(case["cin"], _net_params(case["cin"], seed))
        s["x"] = _net_input(case, seed)
        if kind == "train":
            # a crop of the application grid: h = 1/2048, hz = 1/64
            s["op"] = tpmg.Operator(case["nx"], case["ny"], case["nz"], OMEGA2, 1 / 2048, 1 / 2048, 1 / 64,
                                    _crop_lam(seed), nlevels=1)
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "solve":
        solve = tpmg.mg_solve if case["method"] == "mg" else tpmg.cg_solve
        res = solve(s["op"].op, s["prm"], s["f"], s["u"], s["u"].numel())
        return {"u": s["u"], "iters": res["iters"]}
    if kind == "batched":
        res = tpmg.mg_solve_batched(s["handles"], s["prm"], s["f"], s["u"])
        return {"u": s["u"], "iters": [p["iters"] for p in res["problems"]]}
    if kind == "panel":
        res = tpmg.mg_solve(s["op"].op, s["prm"], s["f"], s["u"], s["u"].numel())
        return {"u": s["u"], "iters": res["iters"]}
    if kind == "smooth":
        tpmg.smooth(s["op"].op, 1, tpmg.PREC[case["prec"]], RHO, s["u"], s["f"], s["out"], s["u"].numel(),
                    norm_out=s["norm"] if case["norm"] else None)
        return {"u": s["out"], "norm": s["norm"]} if case["norm"] else {"u": s["out"]}
    if kind == "transfer":
        op, p, n, nc = s["op"].op, tpmg.PREC[case["prec"]], s["u"].numel(), s["uc"].numel()
        tpmg.residual_restrict_smooth(op, 1, p, RHO, s["u"], s["f"], s["fc"], s["uc"], n, nc)
        tpmg.prolongate(op, 2, p, s["uc"], s["w"], nc, n)
        return {"fc": s["fc"], "uc": s["uc"], "w": s["w"]}
    if kind == "forward":
        return s["net"].forward(s["x"], _shape(case))
    loss, grad = s["net"].loss_grad_residual(s["op"].op, s["x"], s["x"].numel() // case["cin"])
    return {"loss": loss, "grad": grad}


# ---------------------------------------------------------------- work
def work(case):
    """Bytes: each input read once, each output written once. Operations (a multiply-add is 2): of one
    smoothing step 19 per cell (stencil residual 11, line solve 6, update 2), of a V(2,2) cycle five such
    steps' worth on the finest level with 4/3 for the coarser ones, of a CG iteration 28; solves with
    the iteration counts usual for these problems."""
    kind = case["kind"]
    if kind == "batched":
        n = sum(p["nx"] * p["ny"] * p["nz"] for p in _batch(case))
        return {"bytes": 16 * n, "flops": n * 12 * 5 * 19 * 4 / 3}
    n = case["nx"] * case["ny"] * case["nz"]
    if kind == "solve":
        per = 55 * 28 if case["method"] == "cg" else (13 if case["prec"] == "mixed" else 6) * 5 * 19 * 4 / 3
        return {"bytes": 16 * n, "flops": n * per}
    if kind == "panel":
        return {"bytes": 16 * n, "flops": n * 11 * 3 * 22 * 4 / 3}
    b = 4 if case.get("prec") == "f32" else 8
    if kind == "smooth":
        return {"bytes": 3 * b * n, "flops": n * (21 if case["norm"] else 19)}
    if kind == "transfer":
        return {"bytes": 4.5 * b * n, "flops": n * (11 + 1 + 6 / 4 + 5)}
    macs = 27 * (16 * case["cin"] + 2 * 256 + 16)
    if kind == "forward":
        return {"bytes": 4 * n * (case["cin"] + 1), "flops": 2.0 * macs * n}
    return {"bytes": 4 * n * case["cin"], "flops": 6.0 * macs * n}


# ---------------------------------------------------------------- the same in 64 bits, plain torch
def _dct(nz):
    """Orthonormal DCT-II modes (nz, nz) of the Neumann column and the eigenvalues 4 sin^2(pi m / 2 nz)."""
    k = torch.arange(nz, dtype=torch.float64, device="cuda")
    q = torch.cos(math.pi * (k[:, None] + 0.5) * k[None, :] / nz) * math.sqrt(2.0 / nz)
    q[:, 0] = math.sqrt(1.0 / nz)
    return q, 4.0 * torch.sin(math.pi * k / (2 * nz)) ** 2


class _Box:
    """The flat box's levels (index 0 the finest): A, M^{-1} and the transfers."""

    def __init__(self, case, problem, levels):
        w, hx, hy, hz, lam = problem
        v = torch.as_tensor(np.broadcast_to(np.asarray(lam, dtype=np.float64), (case["ny"], case["nx"])).copy(),
                            device="cuda") * w / (hz * hz)
        cx, cy = w / (hx * hx), w / (hy * hy)
        self.lv = []
        for _ in range(levels):
            self.lv.append((cx, cy, v))
            ny, nx = v.shape
            if len(self.lv) < levels:
                v = v.reshape(ny // 2, 2, nx // 2, 2).mean((1, 3))
                cx, cy = cx / 4.0, cy / 4.0
        self.q, self.mu = _dct(case["nz"])

    def apply(self, l, u):
        cx, cy, v = self.lv[l]
        y = u * (1.0 + 2.0 * cx + 2.0 * cy)
        y -= cx * (u.roll(1, 2) + u.roll(-1, 2))
        y -= cy * (u.roll(1, 1) + u.roll(-1, 1))
        d = v * (u[1:] - u[:-1])
        y[:-1] -= d
        y[1:] += d
        return y

    def lines(self, l, b):
        cx, cy, v = self.lv[l]
        t = (self.q.T @ b.reshape(b.shape[0], -1)).reshape(b.shape)
        t /= (1.0 + 2.0 * cx + 2.0 * cy) + self.mu[:, None, None] * v
        return (self.q @ t.reshape(b.shape[0], -1)).reshape(b.shape)

    def restrict(self, r):
        nz, ny, nx = r.shape
        return r.reshape(nz, ny // 2, 2, nx // 2, 2).mean((2, 4))

    def prolong(self, c):
        for dim in (1, 2):
            c = torch.stack((0.75 * c + 0.25 * c.roll(1, dim), 0.75 * c + 0.25 * c.roll(-1, dim)), dim + 1).flatten(dim, dim + 1)
        return c


class _Panel:
    """The same for the gnomonic cubed-sphere panel with its Dirichlet boundary (Eq. (14) of the paper)."""

    def __init__(self, case):
        w, lam, H = _panel_numbers(case)
        nz = case["nz"]
        hz = H / nz
        rf = 1.0 + H * np.arange(nz + 1) / nz
        self.a = torch.as_tensor((rf[1:] ** 3 - rf[:-1] ** 3) / (3.0 * hz), device="cuda")
        self.s = torch.as_tensor(w * lam * rf[1:-1] ** 2 / hz ** 2, device="cuda")  # coupling of planes k, k+1
        g = torch.diag(self.a)
        for k in range(nz - 1):
            g[k, k] += self.s[k]
            g[k + 1, k + 1] += self.s[k]
            g[k, k + 1] -= self.s[k]
            g[k + 1, k] -= self.s[k]
        self.mu, self.q = torch.linalg.eigh(g)
        self.lv = [self._geometry(case["nx"] >> l, case["ny"] >> l, w) for l in range(case["levels"])]

    @staticmethod
    def _geometry(nx, ny, w):
        def point(X, Y):
            X, Y = np.broadcast_arrays(X, Y)
            return np.stack([X, Y, np.ones_like(X)], -1) / np.sqrt(1.0 + X * X + Y * Y)[..., None]

        def arc(p, q):
            return np.arctan2(np.linalg.norm(np.cross(p, q), axis=-1), (p * q).sum(-1))

        xs, ys = (-1.0 + 2.0 * np.arange(m + 1) / m for m in (nx, ny))
        xc, yc = (-1.0 + 2.0 * (np.arange(-1, m + 1) + 0.5) / m for m in (nx, ny))
        F = np.arctan(xs[None, :] * ys[:, None] / np.sqrt(1.0 + xs[None, :] ** 2 + ys[:, None] ** 2))
        area = F[1:, 1:] - F[1:, :-1] - F[:-1, 1:] + F[:-1, :-1]
        corner, centre = point(xs[None, :], ys[:, None]), point(xc[None, :], yc[:, None])
        ax = w * arc(corner[:-1], corner[1:]) / arc(centre[1:-1, :-1], centre[1:-1, 1:])
        ay = w * arc(corner[:, :-1], corner[:, 1:]) / arc(centre[:-1, 1:-1], centre[1:, 1:-1])
        at = ax[:, :-1] + ax[:, 1:] + ay[:-1] + ay[1:]
        return tuple(torch.as_tensor(t, device="cuda") for t in (area, ax, ay, at))

    def apply(self, l, u):
        area, ax, ay, at = self.lv[l]
        y = u * (area * self.a[:, None, None] + at)
        y[:, :, 1:] -= ax[:, 1:-1] * u[:, :, :-1]
        y[:, :, :-1] -= ax[:, 1:-1] * u[:, :, 1:]
        y[:, 1:] -= ay[1:-1] * u[:, :-1]
        y[:, :-1] -= ay[1:-1] * u[:, 1:]
        d = area * self.s[:, None, None] * (u[1:] - u[:-1])
        y[:-1] -= d
        y[1:] += d
        return y

    def lines(self, l, b):
        area, _, _, at = self.lv[l]
        t = (self.q.T @ b.reshape(b.shape[0], -1)).reshape(b.shape)
        t /= self.mu[:, None, None] * area + at
        return (self.q @ t.reshape(b.shape[0], -1)).reshape(b.shape)

    def restrict(self, r):
        nz, ny, nx = r.shape
        return r.reshape(nz, ny // 2, 2, nx // 2, 2).sum((2, 4))

    def prolong(self, c):
        for dim in (1, 2):
            lo, hi = torch.zeros_like(c), torch.zeros_like(c)
            n = c.shape[dim]
            lo.narrow(dim, 1, n - 1).copy_(c.narrow(dim, 0, n - 1))
            hi.narrow(dim, 0, n - 1).copy_(c.narrow(dim, 1, n - 1))
            c = torch.stack((0.75 * c + 0.25 * lo, 0.75 * c + 0.25 * hi), dim + 1).flatten(dim, dim + 1)
        return c


def _mg(A, f, tol, pre=2, post=2, rho=RHO):
    """V(pre, post) cycles of Algorithm 1 from zero until the relative residual is below tol."""
    last = len(A.lv) - 1

    def smooth(l, u, b, times):
        for _ in range(times):
            u = u + rho * A.lines(l, b - A.apply(l, u))
        return u

    def cycle(l, u, b):
        if l == last:
            u = smooth(l, u, b, 1) if last == 0 else rho * A.lines(l, b)
            return smooth(l, u, b, 1)
        u = smooth(l, u, b, pre) if l == 0 else smooth(l, rho * A.lines(l, b), b, pre - 1)
        c = cycle(l + 1, None, A.restrict(b - A.apply(l, u)))
        return smooth(l, u + A.prolong(c), b, post)

    u, r0, it = torch.zeros_like(f), f.norm(), 0
    while it < 400:
        u, it = cycle(0, u, f), it + 1
        if (f - A.apply(0, u)).norm() / r0 < tol:
            break
    return u, it


def _cg(A, f, tol):
    u, r = torch.zeros_like(f), f.clone()
    z = A.lines(0, r)
    p, rz, r0, it = z.clone(), (r * z).sum(), f.norm(), 0
    while it < 400:
        q = A.apply(0, p)
        al = rz / (p * q).sum()
        u += al * p
        r -= al * q
        it += 1
        if r.norm() / r0 < tol:
            break
        z = A.lines(0, r)
        new = (r * z).sum()
        p, rz = z + (new / rz) * p, new
    return u, it


def _split(params, cin):
    """W (27, ci, co) with taps in (dz, dy, dx) order and b per layer, from the flat parameters."""
    out, o = [], 0
    for ci, co in ((cin, 16), (16, 16), (16, 16), (16, 1)):
        W = params[o:o + co * ci * 27].reshape(co, ci, 27).permute(2, 1, 0)
        out.append((W, params[o + co * ci * 27:o + co * ci * 27 + co]))
        o += co * ci * 27 + co
    return out


def _forward(layers, x):
    """The network on x (nz, ny, nx, ci): 3x3x3 taps, periodic in x and y, zero in z, ReLU between."""
    for n, (W, b) in enumerate(layers):
        nz, ny, nx, ci = x.shape
        x = torch.cat((x[:, :, -1:], x, x[:, :, :1]), 2)
        x = torch.cat((x[:, -1:], x, x[:, :1]), 1)
        x = torch.cat((torch.zeros_like(x[:1]), x, torch.zeros_like(x[:1])), 0)
        y = b.expand(nz * ny * nx, -1)
        for t in range(27):
            dz, dy, dx = t // 9, t // 3 % 3, t % 3
            y = y + x[dz:dz + nz, dy:dy + ny, dx:dx + nx].reshape(-1, ci) @ W[t]
        x = (torch.relu(y) if n < 3 else y).reshape(nz, ny, nx, -1)
    return x[..., 0]


def exact(case, seed):
    kind = case["kind"]
    with torch.enable_grad() if kind == "train" else torch.no_grad():
        if kind == "solve":
            A, f = _Box(case, _problem(case), case["levels"]), _rhs(_gen(seed), _shape(case))
            u, it = _mg(A, f, case["tol"]) if case["method"] == "mg" else _cg(A, f, case["tol"])
            return {"u": u, "iters": it}
        if kind == "batched":
            g, probs = _gen(seed), _batch(case)
            fs = [_rhs(g, _shape(p)) for p in probs]
            got = [_mg(_Box(p, _problem(p), p["levels"]), f, case["tol"]) for p, f in zip(probs, fs)]
            return {"u": [u for u, _ in got], "iters": [it for _, it in got]}
        if kind == "panel":
            u, it = _mg(_Panel(case), _normal(_gen(seed), _shape(case)), case["tol"], 1, 1, 2.0 / 3.0)
            return {"u": u, "iters": it}
        if kind in ("smooth", "transfer"):
            A = _Box(case, _problem(case), 1 if kind == "smooth" else 2)
            u, f, w = (t if t is None else t.double() for t in _unit_fields(case, seed))
            r = f - A.apply(0, u)
            if kind == "smooth":
                out = u + RHO * A.lines(0, r)
                return {"u": out, "norm": r.norm().reshape(1)} if case["norm"] else {"u": out}
            fc = A.restrict(r)
            uc = RHO * A.lines(1, fc)
            return {"fc": fc, "uc": uc, "w": w + A.prolong(uc)}
        prm = torch.as_tensor(_net_params(case["cin"], seed).astype(np.float64), device="cuda")
        x = _net_input(case, seed).double()
        if kind == "forward":
            return _forward(_split(prm, case["cin"]), x).reshape(-1)
        prm.requires_grad_(True)
        one = dict(case, levels=1)
        A = _Box(one, (OMEGA2, 1 / 2048, 1 / 2048, 1 / 64, _crop_lam(seed)), 1)
        cx, cy, v = A.lv[0]
        ends = torch.full((case["nz"],), 2.0, dtype=torch.float64, device="cuda")
        ends[0] -= 1.0
        ends[-1] -= 1.0
        diag = (1.0 + 2.0 * cx + 2.0 * cy) + ends[:, None, None] * v
        loss = (x[..., 0] - A.apply(0, _forward(_split(prm, case["cin"]), x) / diag)).square().mean()
        loss.backward()
        return {"loss": loss.detach().reshape(1), "grad": prm.grad}
