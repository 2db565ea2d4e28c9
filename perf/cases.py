"""The calls whose time matters to a user of this library, over the range of their sizes.

A fit spends its time in damped Gauss-Newton steps, and a step in five calls that a program can
also make by itself: the residual rows (every line-search trial is one), their Jacobian, the
adjoint gradient (what an autograd optimiser calls), the Gram product of a row block, and the
damped solve.  Each of those is measured alone, small, ordinary and large, and the whole step on
the smallest and on the headline profile of this repository.

Problems are the ones of `paper_2509_14185_gb300.inputs` (Xavier-initialised networks, log-spaced
and uniform points), with other widths and point counts where a case says so.  The Gram and the
solve take matrices with the structure of a network's Jacobian (`jacobian_like`).  The damping of
the solves and steps lies between 1e-2 and 10: at the start value 1e-6 a first step is so badly
conditioned that its direction is fixed by rounding alone, which nothing could be compared with.

`exact` is plain torch in 64 bits: torch.func derivatives of the residuals written out here, dense
products and a dense solve.
"""
import math

import torch

from paper_2509_14185_gb300 import gn, inputs

DEV = "cuda"
F64 = torch.float64
EQ = {"burgers": inputs.BURGERS, "ccf": inputs.CCF, "ipm": inputs.IPM, "boussinesq": inputs.BOUSSINESQ}
DIM = {"burgers": 1, "ccf": 1, "ipm": 2, "boussinesq": 2}
NEQ = {"burgers": 1, "ccf": 1, "ipm": 2, "boussinesq": 3}
PRECISION = {"fp64": gn.GN_PREC_FP64, "split": gn.GN_PREC_SPLIT_BF16, "split_all": gn.GN_PREC_SPLIT_ALL}


def listed():
    return [
        # a line-search trial of a small 1D fit: launches and latency
        dict(name="residual_burgers_1k", kind="residual", eq="burgers", width=32, depth=2, n=1024, nb=0),
        # a line-search trial (or a validation pass) of the 2D workload with a wall
        dict(name="residual_ipm_64k", kind="residual", eq="ipm", width=64, depth=4, n=65536, nb=4096),
        # forward and backward through the autograd function, weighted points, odd sizes
        dict(name="gradient_boussinesq_9k", kind="gradient", eq="boussinesq", width=48, depth=3, n=9001, nb=513,
             weighted=True),
        # the rows of a step on the headline profile, with its Hilbert contraction
        dict(name="jacobian_ccf_16k", kind="jacobian", eq="ccf", width=64, depth=3, n=16384, nb=0,
             precision="split_all", row0=0, rows=16385),
        # one block of a Jacobian that is streamed in row blocks; it starts inside a point
        dict(name="jacobian_ipm_block", kind="jacobian", eq="ipm", width=64, depth=4, n=65536, nb=4096,
             precision="split_all", row0=20001, rows=32768),
        # the Gram of the headline profile
        dict(name="gram_split_16k", kind="gram", width=64, depth=3, rows=16385, blocks=1, precision="split"),
        # a Gram accumulated over two row blocks, a fit of the batched sweep, ragged sizes
        dict(name="gram_split_5k_blocks", kind="gram", width=48, depth=3, rows=5003, blocks=2, precision="split"),
        # the default precision on a small fit
        dict(name="gram_fp64_1k", kind="gram", width=32, depth=2, rows=1025, blocks=1, precision="fp64"),
        dict(name="solve_fp64_1k", kind="solve", width=32, depth=2, rows=1025, precision="fp64", gamma=1e-2),
        # the damped solve of the headline profile
        dict(name="solve_split_8k", kind="solve", width=64, depth=3, rows=4097, precision="split_all", gamma=1e-2),
        # whole steps through the captured graph: the smallest profile and the headline one
        dict(name="step_ccf_1k", kind="step", eq="ccf", width=32, depth=2, n=1024, nb=0, precision="split_all",
             gamma=1.0),
        dict(name="step_ccf_16k", kind="step", eq="ccf", width=64, depth=3, n=16384, nb=0, precision="split_all",
             gamma=1.0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["residual", "gradient", "jacobian", "gram", "solve", "step"])
    if kind in ("residual", "gradient", "jacobian"):
        eq = rng.choice(sorted(EQ))
        c = dict(kind=kind, eq=eq, width=_log_int(rng, 12, 96), depth=rng.randint(2, 4))
        p = inputs.param_count(_widths(c))
        top = 16384 if eq == "ccf" else 65536
        if kind != "residual":   # no more work than the listed ones: 2e8 Jacobian entries
            top = min(top, int(2e8 / (p * NEQ[eq])))
        c["n"] = _log_int(rng, 300, max(600, top))
        c["nb"] = _log_int(rng, 10, max(20, c["n"] // 16)) if DIM[eq] == 2 else 0
        if kind == "jacobian":
            c["precision"] = rng.choice(["fp64", "split_all"]) if c["n"] * p < 2e7 else "split_all"
            total = c["n"] * NEQ[eq] + c["nb"] + 1
            c["row0"] = rng.choice([0, rng.randrange(total // 2)])
            c["rows"] = total - c["row0"]
        elif rng.random() < 0.5:
            c["weighted"] = True
        return c
    if kind == "step":
        return dict(kind=kind, eq=rng.choice(["burgers", "ccf"]), width=_log_int(rng, 14, 56), depth=2,
                    n=_log_int(rng, 300, 8000), nb=0, precision="split_all", gamma=10.0 ** rng.uniform(-0.3, 1.0))
    c = dict(kind=kind, width=_log_int(rng, 12, 64), depth=rng.randint(2, 3))
    p = inputs.param_count(_widths(c)) + 1
    if kind == "gram":
        c["rows"] = _log_int(rng, 300, 16385)
        c["blocks"] = rng.choice([1, 1, 2])
        c["precision"] = "fp64" if c["rows"] * p * p < 1e10 and rng.random() < 0.4 else "split"
    else:
        c["rows"] = min(4097, _log_int(rng, 300, 8000))
        c["precision"] = "fp64" if p < 2000 and rng.random() < 0.4 else "split_all"
        c["gamma"] = 10.0 ** rng.uniform(-2.0, 0.0)
    return c


# ---- inputs -----------------------------------------------------------------------------------


def _widths(c):
    eq = c.get("eq", "burgers")
    return [DIM[eq]] + [c["width"]] * c["depth"] + [{"ipm": 2, "boussinesq": 3}.get(eq, 1)]


def _workload(c, seed):
    eq, n = c["eq"], c["n"]
    if DIM[eq] == 1:
        y = inputs.points_1d(n // 4, n - n // 4, 1e-3, 1e4 if eq == "ccf" else 1e3, seed, uniform_lo=1e-3)
        yb = torch.zeros(1, 0).numpy()
        lam = 0.6057 if eq == "ccf" else 0.5
    else:
        y = inputs.points_2d_polar(n, 1, 1e-3, 1e3, seed, random_radius=True)
        yb = inputs.wall_points(c["nb"], 1e-3, 1e3, seed + 1, random=True)
        lam = 1.0 / 0.9723 if eq == "ipm" else 1.0 / 1.0863 + 1.0
    norm, target = inputs.NORM_POINT[EQ[eq]]
    rho = 0.25 + 3.75 * inputs.uniform(seed + 2, n) if c.get("weighted") else None
    widths = _widths(c)
    return inputs.Workload(name=eq, equation=EQ[eq], widths=widths, y=y, y_bnd=yb, lam=lam,
                           theta=inputs.xavier_init(widths, seed), y_norm=norm, c_norm=target, rho=rho)


def _dev(x):
    return torch.as_tensor(x, dtype=F64, device=DEV)


def jacobian_like(c, seed, rows):
    """(J, r) of `rows` points as a network's backward pass gives them: per layer the outer product
    of an adjoint and an activation (smooth in the point, scales over three decades), its bias
    column, the lambda column, weights sqrt(2/N), and a normalisation row of weight sqrt(2)."""
    g = torch.Generator().manual_seed(seed)
    widths = _widths(c)

    def rand(*s):
        return torch.rand(*s, generator=g, dtype=F64).to(DEV)

    x = torch.cat([torch.linspace(0.0, 1.0, rows - rows // 4, dtype=F64, device=DEV), rand(rows // 4)])[:, None]
    J = torch.empty(rows, inputs.param_count(widths) + 1, dtype=F64, device=DEV)
    off = 0
    for i, o in zip(widths[:-1], widths[1:]):
        h = torch.tanh((6.0 * rand(1, i) - 3.0) * x + 2.0 * rand(1, i) - 1.0)
        a = 10.0 ** (3.0 * rand(1, o) - 3.0) * torch.sin((9.0 * rand(1, o)) * x + 6.3 * rand(1, o)) * torch.exp(-2.0 * x)
        torch.mul(a[:, :, None], h[:, None, :], out=J[:, off:off + i * o].view(rows, o, i))
        off += i * o
        J[:, off:off + o] = a
        off += o
    J[:, off] = torch.cos(5.0 * x[:, 0]) * torch.exp(-x[:, 0])
    r = (torch.sin(7.0 * x[:, 0]) + 0.1 * rand(rows)) * torch.exp(-x[:, 0])
    w = torch.full((rows,), math.sqrt(2.0 / rows), dtype=F64, device=DEV)
    w[-1] = math.sqrt(2.0)
    J *= w[:, None]
    r *= w
    return J, r


def prepare(case, seed):
    kind = case["kind"]
    s = dict(kind=kind)
    if kind in ("gram", "solve"):
        # the handle of a fit of that network; its own points do not enter these two calls
        w = _workload(dict(case, eq="burgers", n=256, nb=0), seed)
        s["prob"] = gn.GNProblem.from_workload(w, precision=PRECISION[case["precision"]], n_slices=6)
        J, r = jacobian_like(case, seed, case["rows"])
        p = J.shape[1]
        s["g"] = torch.zeros(p, dtype=F64, device=DEV)
        if kind == "gram":
            cut = case["rows"] // case["blocks"]
            s["blocks"] = [(J[:cut], r[:cut])] + ([(J[cut:], r[cut:])] if case["blocks"] == 2 else [])
            s["G"] = torch.zeros(p, p, dtype=F64, device=DEV)
            s["precision"] = PRECISION[case["precision"]]
        else:
            s["G"], s["g"] = J.T @ J, J.T @ r
            s["delta"] = torch.zeros(p, dtype=F64, device=DEV)
            s["gamma"] = case["gamma"]
        return s
    w = _workload(case, seed)
    kw = dict(precision=PRECISION[case.get("precision", "fp64")], n_slices=6)
    if kind == "jacobian":
        kw["row_block"] = case["rows"]
    s["prob"] = gn.GNProblem.from_workload(w, **kw)
    s["theta"], s["lam"] = _dev(w.theta), w.lam
    if kind == "residual":
        s["r"] = s["prob"].new_vec(s["prob"].n_rows)
    elif kind == "gradient":
        s["theta"].requires_grad_()
        s["lam"] = torch.tensor(w.lam, dtype=F64, device=DEV, requires_grad=True)
    elif kind == "jacobian":
        s["J"] = torch.zeros(case["rows"], s["prob"].P + 1, dtype=F64, device=DEV)
        s["row0"], s["rows"] = case["row0"], case["rows"]
    else:
        s["start"], s["gamma"] = s["theta"].clone(), case["gamma"]
    return s


def run(s):
    kind, p = s["kind"], s["prob"]
    if kind == "residual":
        status, loss = p.gn_residual(s["theta"], s["lam"], s["r"])
        return {"r": s["r"], "loss": loss, "status": status}
    if kind == "gradient":
        r = gn.residual_fn(s["theta"], s["lam"], p)
        gt, gl = torch.autograd.grad(0.5 * (r * r).sum(), (s["theta"], s["lam"]))
        return {"r": r.detach(), "grad_theta": gt, "grad_lam": gl}
    if kind == "jacobian":
        p.gn_jacobian(s["theta"], s["lam"], s["J"], s["row0"], s["rows"])
        return {"J": s["J"]}
    if kind == "gram":
        for k, (J, r) in enumerate(s["blocks"]):
            p.gn_gram(J, J.shape[0], r, s["G"], s["g"], precision=s["precision"], accumulate=k > 0)
        return {"G": s["G"].tril_(), "g": s["g"]}   # above the diagonal G holds parts of tiles
    if kind == "solve":
        status, gamma, retries = p.gn_damped_solve(s["G"], s["g"], s["gamma"], s["delta"])
        return {"delta": s["delta"], "gamma": gamma, "status": status, "retries": retries}
    s["theta"].copy_(s["start"])
    status, lam, gamma, info = p.gn_step_graph(s["theta"], s["lam"], s["gamma"])
    return {"theta": s["theta"], "lam": lam, "gamma": gamma, "before": info["loss_before"],
            "after": info["loss_after"], "alpha": info["alpha"], "status": status, "trials": info["n_trials"]}


# ---- what a pass cannot do without ------------------------------------------------------------


def _pass_work(c, mode, rows=None):
    """Jets through the network (2 or 6 components forward; one more order where the lambda column
    needs it), then per row the adjoint and the row's entries, all as multiply-adds."""
    widths, d, ne = _widths(c), DIM[c["eq"]], NEQ[c["eq"]]
    p = inputs.param_count(widths)
    pw = sum(i * o for i, o in zip(widths[:-1], widths[1:]))
    cr, cf = (2, 3) if d == 1 else (6, 9)
    total = c["n"] * ne + c["nb"] + 1
    rows = total if rows is None else rows
    pts = (c["n"] + c["nb"] + 1) * rows / total
    flops = 2.0 * pts * (cr if mode == "residual" else cf) * pw
    if mode != "residual":
        flops += 2.0 * (pts if mode == "gradient" else rows) * cr * (pw + p)
    if c["eq"] == "ccf":
        flops += 2.0 * c["n"] * 512 * (p + 1 if mode == "jacobian" else 2 if mode == "gradient" else 1)
    out = rows * (p + 1) if mode == "jacobian" else total + (p + 1 if mode == "gradient" else 0)
    return 8.0 * (d * pts + p + out), flops


def work(case):
    kind = case["kind"]
    if kind in ("residual", "gradient", "jacobian"):
        b, f = _pass_work(case, kind, case.get("rows"))
        return {"bytes": b, "flops": f}
    p = inputs.param_count(_widths(case)) + 1
    if kind == "gram":
        return {"bytes": 8.0 * (case["rows"] * (p + 1) + p * (p + 1) / 2 + p),
                "flops": 1.0 * case["rows"] * p * (p + 3)}
    solve = p ** 3 / 3.0 + 2.0 * p * p
    if kind == "solve":
        return {"bytes": 8.0 * (p * (p + 1) / 2 + 2 * p), "flops": solve}
    _, jac = _pass_work(case, "jacobian")
    _, res = _pass_work(case, "residual")
    rows = case["n"] + 1
    return {"bytes": 8.0 * (2 * p + DIM[case["eq"]] * case["n"]), "flops": jac + res + rows * p * (p + 3.0) + solve}


# ---- the same values in plain torch -----------------------------------------------------------


class _Plain:
    """The residual rows of a workload, from the equations alone."""

    def __init__(self, c, seed):
        self.w = w = _workload(c, seed)
        self.eq, self.d, self.ne = c["eq"], DIM[c["eq"]], NEQ[c["eq"]]
        self.y, self.yb = _dev(w.y).T, _dev(w.y_bnd).T
        self.yn = _dev(w.y_norm[:self.d])[None]
        n = c["n"]
        rho = torch.ones(n, dtype=F64, device=DEV) if w.rho is None else _dev(w.rho)
        self.weight = torch.sqrt(2.0 * rho / (n * self.ne))
        self.n, self.nb = n, c["nb"]
        if self.eq == "ccf":
            m = w.hilbert_m
            psi = -math.pi + (torch.arange(m, dtype=F64, device=DEV) + 0.5) * (2.0 * math.pi / m)
            s = torch.tan(0.5 * psi)
            x = self.y[:, 0]
            cot = 1.0 / torch.tan(0.5 * (2.0 * torch.atan(x)[:, None] - psi[None, :]))
            k = (x[:, None] / m) * (cot - s[None, :])
            self.kf = k[:, m // 2:] - k[:, :m // 2].flip(1)   # the integrand is odd
            self.diag = -(x / m) * cot.sum(1)
            self.nodes = s[m // 2:, None]
        self.widths = w.widths

    def net(self, theta, z):
        off = 0
        for l, (i, o) in enumerate(zip(self.widths[:-1], self.widths[1:])):
            z = theta[off:off + i * o].view(o, i) @ z + theta[off + i * o:off + i * o + o]
            off += i * o + o
            if l < len(self.widths) - 2:
                z = torch.tanh(z)
        return z

    def fields(self, theta, lam, y):
        u = 1.0 + (y * y).sum()
        a = 1.0 / (1.0 + lam)
        q = torch.exp(-0.5 * a * torch.log(u))
        z = q[None] if self.d == 1 else torch.stack([q, y[1] / torch.sqrt(u)])
        out = self.net(theta, z)
        spec = {"burgers": [(lam, 1, -0.5)], "ccf": [(lam, 2, -1.0)],
                "ipm": [(lam, 0, 0.0), (1 + 2 * lam, 1, -0.5)],
                "boussinesq": [(-1.0, 1, -0.5), (lam - 1, 0, 0.0), (1 + 2 * lam, 1, -0.5)]}[self.eq]
        return torch.stack([y[0] ** m * torch.exp((e + 0.5 * k * a) * torch.log(u)) * out[f]
                            for f, (k, m, e) in enumerate(spec)])

    def g(self, theta, lam, y):   # CCF: Theta / y
        u = 1.0 + y[0] * y[0]
        a = 1.0 / (1.0 + lam)
        q = torch.exp(-0.5 * a * torch.log(u))
        return y[0] * torch.exp((-1.0 + 0.5 * lam * a) * torch.log(u)) * self.net(theta, q[None])[0]

    def interior(self, theta, lam, y, ug, dg):
        """R_k at one point; ug, dg: the Hilbert sum over the nodes and the diagonal coefficient."""
        f = lambda v: self.fields(theta, lam, v)   # noqa: E731
        if self.d == 1:
            v, t = torch.func.jvp(f, (y,), (torch.ones_like(y),))
            vel = v[0] if self.eq == "burgers" else ug + dg * self.g(theta, lam, y)
            return (-lam * v[0] + ((1 + lam) * y[0] + vel) * t[0])[None]
        v = f(y)
        e = torch.eye(2, dtype=F64, device=y.device)
        first = [torch.func.jvp(f, (y,), (e[k],))[1] for k in range(2)]
        lap = sum(torch.func.jvp(lambda x, k=k: torch.func.jvp(f, (x,), (e[k],))[1], (y,), (e[k],))[1][-1]
                  for k in range(2))
        v1, v2 = (1 + lam) * y[0] + first[1][-1], (1 + lam) * y[1] - first[0][-1]
        adv = v1 * first[0] + v2 * first[1]
        if self.eq == "ipm":
            return torch.stack([-lam * v[0] + adv[0], lap - first[0][0]])
        return torch.stack([v[0] + adv[0] - first[0][1], (1 - lam) * v[1] + adv[1], lap + v[0]])

    def norm(self, theta, lam):
        f = lambda v: self.fields(theta, lam, v)[0]   # noqa: E731
        if self.eq == "boussinesq":
            e = torch.eye(2, dtype=F64, device=DEV)[0]
            val = torch.func.jvp(f, (self.yn[0],), (e,))[1]
        else:
            val = f(self.yn[0])
        return math.sqrt(2.0) * (val - self.w.c_norm)

    def wall(self, theta, lam, y):
        return math.sqrt(2.0 / max(1, self.nb)) * self.fields(theta, lam, y)[-1]

    def hilbert(self, theta, lam):
        if self.eq != "ccf":
            z = torch.zeros(self.n, dtype=F64, device=DEV)
            return z, z
        gn_ = torch.func.vmap(lambda s: self.g(theta, lam, s))(self.nodes)
        return self.kf @ gn_, self.diag

    def rows(self, theta, lam, chunk=16384):
        ug, dg = self.hilbert(theta, lam)
        f = torch.func.vmap(lambda y, u, c: self.interior(theta, lam, y, u, c))
        out = [(f(self.y[k:k + chunk], ug[k:k + chunk], dg[k:k + chunk]) * self.weight[k:k + chunk, None]).reshape(-1)
               for k in range(0, self.n, chunk)]
        if self.nb:
            out.append(torch.func.vmap(lambda y: self.wall(theta, lam, y))(self.yb))
        return torch.cat(out + [self.norm(theta, lam)[None]])

    def jacobian(self, theta, lam, row0, rows):
        def block(f, *args):   # d f / d (theta, lam) of every point, (points, outputs, P + 1)
            j = torch.func.vmap(torch.func.jacrev(f, argnums=(0, 1)), in_dims=(None, None) + (0,) * len(args))
            jt, jl = j(theta, lam, *args)
            return torch.cat([jt, jl[..., None]], -1)

        ug, dg = self.hilbert(theta, lam)
        J = torch.zeros(rows, theta.numel() + 1, dtype=F64, device=DEV)
        if self.eq == "ccf":
            gn_rows = block(lambda t, l, y: self.g(t, l, y)[None], self.nodes)[:, 0]
        p0, p1 = row0 // self.ne, min(self.n, -(-(row0 + rows) // self.ne))
        step = 512
        for k in range(p0, p1, step):
            e = min(p1, k + step)
            b = block(self.interior, self.y[k:e], ug[k:e], dg[k:e])
            if self.eq == "ccf":
                du = torch.func.vmap(torch.func.jacrev(self.interior, argnums=3), in_dims=(None, None, 0, 0, 0))(
                    theta, lam, self.y[k:e], ug[k:e], dg[k:e])[:, 0]
                b[:, 0] += du[:, None] * (self.kf[k:e] @ gn_rows)
            b = (b * self.weight[k:e, None, None]).reshape(-1, b.shape[-1])
            lo, hi = max(row0, k * self.ne), min(row0 + rows, e * self.ne)
            J[lo - row0:hi - row0] = b[lo - k * self.ne:hi - k * self.ne]
        w0 = self.n * self.ne
        for k in range(max(0, row0 - w0), min(self.nb, row0 + rows - w0), step):
            e = min(self.nb, row0 + rows - w0, k + step)
            J[w0 + k - row0:w0 + e - row0] = block(lambda t, l, y: self.wall(t, l, y)[None], self.yb[k:e])[:, 0]
        if row0 + rows == w0 + self.nb + 1:
            jt, jl = torch.func.jacrev(self.norm, argnums=(0, 1))(theta, lam)
            J[-1, :-1], J[-1, -1] = jt, jl
        return J


def exact(case, seed):
    kind = case["kind"]
    if kind in ("gram", "solve"):
        J, r = jacobian_like(case, seed, case["rows"])
        G, g = J.T @ J, J.T @ r
        if kind == "gram":
            return {"G": G.tril(), "g": g}
        del J
        G.diagonal().add_(case["gamma"])
        x = torch.cholesky_solve(g[:, None], torch.linalg.cholesky(G))[:, 0]
        return {"delta": x, "gamma": case["gamma"], "status": None, "retries": None}
    q = _Plain(case, seed)
    theta, lam = _dev(q.w.theta), torch.tensor(q.w.lam, dtype=F64, device=DEV)
    if kind == "residual":
        r = q.rows(theta, lam)
        return {"r": r, "loss": float(0.5 * (r * r).sum()), "status": None}
    if kind == "gradient":
        theta.requires_grad_()
        lam.requires_grad_()
        r = q.rows(theta, lam)
        gt, gl = torch.autograd.grad(0.5 * (r * r).sum(), (theta, lam))
        return {"r": r.detach(), "grad_theta": gt, "grad_lam": gl}
    if kind == "jacobian":
        return {"J": q.jacobian(theta, lam, case["row0"], case["rows"])}
    # a damped step: Armijo backtracking from a full step, then the Levenberg-Marquardt rule
    r = q.rows(theta, lam)
    J = q.jacobian(theta, lam, 0, r.numel())
    G, g, gamma = J.T @ J, J.T @ r, case["gamma"]
    A = G.clone()
    A.diagonal().add_(gamma)
    delta = torch.cholesky_solve(g[:, None], torch.linalg.cholesky(A))[:, 0]
    h0, gd, dgd = float(0.5 * (r * r).sum()), float(g @ delta), float(delta @ (G @ delta))
    alpha = 1.0
    for _ in range(8):
        t, l = theta - alpha * delta[:-1], lam - alpha * delta[-1]
        h = float(0.5 * (q.rows(t, l) ** 2).sum())
        if h <= h0 - 1e-4 * alpha * gd:
            rho = (h0 - h) / (alpha * gd - 0.5 * alpha * alpha * dgd)
            gamma *= 1.5 if rho < 0.25 else 2.0 / 3.0 if rho > 0.75 else 1.0
            return {"theta": t, "lam": float(l), "gamma": gamma, "before": h0, "after": h, "alpha": alpha,
                    "status": None, "trials": None}
        alpha *= 0.5
    return None
