"""Performance cases: the work a user of this library has it do, through its
public entry points (paper_1912_04501_gb300.bie), and what that work gives in
64 bits, evaluated with plain torch.

A case is a dict of plain values:
    kind       apply   one operator application (the GMRES matvec)
               solve   a mobility solve from zero, then the body velocities
               step    a configuration restored and advanced three Euler steps
               contact two nearly touching ellipses moved, solved, extracted
               net     the warm-start network's loss and gradient
    bodies, nodes, ragged, phi, skew, images, precision, cells, gap: see _cells

The single-precision application (precision "mixed") promises single-
precision pair sums, so its result is handed on as float32, as a caller that
feeds it to the network or to an inner iteration does; everything else comes
back in the type the library gives.  Solves run to a 1e-12 residual (the
tolerance the repository's own comparisons of two solves use), so that the
density is determined to far below what is compared.
"""
import functools
import math

import numpy as np
import torch

from paper_1912_04501_gb300 import bie, learn, workloads

PRECISION = {"mixed": bie.BIE_MIXED, "df64": bie.BIE_DF64, "fp64": bie.BIE_FP64}
DT = 1e-3          # time step of the 25- and 400-ellipse workloads
STEPS = 3          # two start-up steps, then one with recycled directions
SOLVE_TOL = 1e-12


def listed():
    def apply_case(name, bodies, nodes, precision="mixed", ragged=False, phi=0.3, skew=0.0, images=9, cells=1):
        return dict(name=name, kind="apply", bodies=bodies, nodes=nodes, ragged=ragged, phi=phi, skew=skew,
                    images=images, precision=precision, cells=cells)
    return [
        # the one-ellipse validation cell: the smallest call, all launches and latency
        apply_case("apply-mixed-1", 1, 128, phi=0.0628),
        # the inner iteration of the 25-ellipse suspension (the paper's standard size)
        apply_case("apply-mixed-25", 25, 256),
        # a polydisperse sheared cell whose node counts follow the perimeters
        apply_case("apply-mixed-100-ragged", 100, 160, ragged=True, skew=0.3),
        # the inner iteration of the largest single-cell suspension (102400 nodes)
        apply_case("apply-mixed-400", 400, 256),
        # an ensemble of 64 independent cells of uneven size in one context
        apply_case("apply-mixed-batch-64", 50, 160, ragged=True, cells=64),
        # the paper's own periodizer (four images per node in the doubled cell)
        apply_case("apply-mixed-doubled-100", 100, 160, ragged=True, skew=-0.2, images=4),
        # the refinement residual of the largest suspension
        apply_case("apply-df64-400", 400, 256, precision="df64"),
        # the plain double-precision method, the comparison every solve is judged by
        apply_case("apply-fp64-25", 25, 256, precision="fp64"),
        # one quasi-static mobility solve
        dict(name="solve-25", kind="solve", bodies=25, nodes=256, ragged=False, phi=0.3, skew=0.0),
        # time stepping from a stored configuration, warm start and network included
        dict(name="step-25", kind="step", bodies=25, nodes=256, ragged=False, phi=0.3, skew=0.0),
        # the near-contact study: a new configuration of two ellipses 2e-3 apart
        dict(name="contact-2e-3", kind="contact", nodes=512, gap=2e-3),
        # one training batch of the warm-start network (loss and gradient)
        dict(name="net-gradient", kind="net", rows=102400),
    ]


def draw(rng):
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    kind = rng.choice(["apply"] * 6 + ["solve", "step", "contact", "net"])
    if kind == "net":
        return dict(kind="net", rows=log_int(300, 102400))
    if kind == "contact":
        return dict(kind="contact", nodes=2 * log_int(96, 256), gap=math.exp(rng.uniform(math.log(2e-3), math.log(5e-2))))
    phi, skew = rng.uniform(0.1, 0.3), rng.uniform(-0.45, 0.45)
    if kind in ("solve", "step"):
        return dict(kind=kind, bodies=log_int(2, 30), nodes=2 * rng.randint(48, 128), ragged=rng.random() < 0.5,
                    phi=phi, skew=skew)
    precision = rng.choice(["mixed", "mixed", "mixed", "df64", "fp64"])
    images = 4 if rng.random() < 0.2 else 9
    cells = log_int(2, 64) if images == 9 and precision == "mixed" and rng.random() < 0.25 else 1
    if cells > 1:
        bodies = rng.randint(5, 50)
    else:
        # the doubled cell takes bodies smaller than about half a cell
        bodies = log_int(16 if images == 4 else 1, 40 if precision == "fp64" else 400)
    return dict(kind="apply", bodies=bodies, nodes=2 * rng.randint(48, 128), ragged=rng.random() < 0.5, phi=phi,
                skew=skew, images=images, precision=precision, cells=cells)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _perimeter(b):
    return math.pi * (3 * (b["a"] + b["b"]) - math.sqrt((3 * b["a"] + b["b"]) * (b["a"] + 3 * b["b"])))


@functools.lru_cache(maxsize=None)
def _packing(bodies, nodes, ragged, phi, skew, which):
    """A seeded suspension of ellipses of aspect ratio 1..3 (fewer bodies are
    larger, so they keep wider gaps); ragged: sizes vary and each body gets
    nodes in proportion to its perimeter, an even number in 3/5 .. 8/5 of `nodes`."""
    gap = 1e-2 if bodies <= 60 else 2e-3
    cell = workloads.random_cell(bodies, phi, (1.0, 3.0 if bodies > 1 else 2.0), gap, nodes, 1000 + which,
                                 e2=(skew, 1.0), equal_area=not ragged, max_tries=2000000)
    if ragged:
        mean = np.mean([_perimeter(b) for b in cell["bodies"]])
        for b in cell["bodies"]:
            b["n"] = 2 * int(min(0.8 * nodes, max(0.3 * nodes, round(0.5 * nodes * _perimeter(b) / mean))))
    return cell


def _moved(cell, rng):
    """The suspension translated by a random vector (a new configuration with
    the same gaps), its bodies turned over to their cell and relisted."""
    e1, e2, c = (np.asarray(cell[k], float) for k in ("e1", "e2", "centre"))
    E = np.column_stack([e1, e2])
    shift = E @ rng.uniform(-0.5, 0.5, 2)
    bodies = []
    for i in rng.permutation(len(cell["bodies"])):
        b = dict(cell["bodies"][i])
        st = np.linalg.solve(E, np.asarray(b["xc"]) + shift - c)
        b["xc"] = (c + E @ (st - np.floor(st + 0.5))).tolist()
        bodies.append(b)
    return dict(cell, bodies=bodies)


def _cells(case, rng):
    """The unit cells of a case: one, or a batch of `cells` with 5..`bodies`
    bodies and area fractions 0.1..`phi` (16 packings, each moved anew)."""
    n = case.get("cells", 1)
    out = []
    for k in range(n):
        if n == 1:
            bodies, phi = case["bodies"], case["phi"]
        else:
            r = np.random.default_rng(77 + k % 16)
            bodies, phi = int(r.integers(5, case["bodies"] + 1)), round(float(r.uniform(0.1, max(0.1, case["phi"]))), 3)
        cell = _packing(bodies, case["nodes"], case["ragged"], phi, case["skew"], k % 16)
        M, m = (128, 32) if case.get("images", 9) == 4 else (48, 24)
        out.append(dict(_moved(cell, rng), solver=dict(n_proxy=M, proxy_radius=1.5, n_coll=m, gmres_tol=SOLVE_TOL)))
    return out


def _density(cells, rng):
    """A density as the solver meets it: a few smooth modes on every body and a
    little that is rough."""
    parts = []
    for cell in cells:
        for b in cell["bodies"]:
            t = 2 * np.pi * np.arange(b["n"]) / b["n"]
            k = np.arange(1, 9)
            amp = rng.standard_normal((2, 8, 2)) / k[None, :, None]
            parts.append(np.cos(np.outer(t, k)) @ amp[0] + np.sin(np.outer(t, k)) @ amp[1]
                         + 0.05 * rng.standard_normal((b["n"], 2)) + rng.standard_normal(2))
    return np.concatenate(parts).ravel()


def _contact(case, rng):
    """Two ellipses `gap` apart, translated together and turned a little."""
    cell = workloads.two_ellipses(case["gap"], case["nodes"])
    e2 = [float(rng.uniform(-0.1, 0.1)), 1.0]
    move = rng.uniform(-0.03, 0.03, 2)
    xc = np.array([b["xc"] for b in cell["bodies"]]) + move
    half, th = 0.5 * (xc[0] + xc[1]), float(rng.uniform(-0.3, 0.3))
    R = np.array([[math.cos(th), -math.sin(th)], [math.sin(th), math.cos(th)]])
    return cell, e2, (xc - half) @ R.T + half, np.full(2, th)


def _net_batch(case, rng):
    F, H, n = bie.BIE_NET_FEATURES, bie.BIE_NET_HIDDEN, case["rows"]
    p = (rng.standard_normal(H * F + H + H * H + H + 2 * H + 2) * 0.2).astype(np.float32)
    X = rng.standard_normal((n, F)).astype(np.float32)
    T = rng.standard_normal((n, 2)).astype(np.float32)
    W = rng.uniform(0.5, 1.5, n).astype(np.float32)
    return p, X, T, W


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind = case["kind"]
    if kind == "net":
        p, *batch = _net_batch(case, rng)
        net = bie.Net()
        net.set_params(p)
        return dict(case=case, net=net, batch=[torch.from_numpy(a).cuda() for a in batch])
    if kind == "contact":
        cell, e2, xc, th = _contact(case, rng)
        ctx = bie.Context(cell, precision=bie.BIE_MIXED, precond=1, gmres_tol=SOLVE_TOL)
        return dict(case=case, ctx=ctx, e2=e2, xc=xc, theta=th)
    cells = _cells(case, rng)
    state = dict(case=case, cells=cells)
    if kind == "apply":
        state["ctx"] = bie.Context(cells if case["cells"] > 1 else cells[0], precision=PRECISION[case["precision"]],
                                   n_images=case["images"])
        state["sigma"] = torch.from_numpy(_density(cells, rng)).cuda()
        state["out"] = torch.empty_like(state["sigma"])
    elif kind == "solve":
        state["ctx"] = bie.Context(cells[0], precision=bie.BIE_MIXED)
    else:
        state["net"] = learn.default_net()
        state["ctx"] = bie.Context(cells[0], precision=bie.BIE_MIXED, warm_start=2)
        state["ctx"].set_warm_net(state["net"])
        state["xc"] = np.array([b["xc"] for b in cells[0]["bodies"]])
        state["theta"] = np.array([b["theta"] for b in cells[0]["bodies"]])
    return state


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "net":
        loss, grad = state["net"].loss_grad(*state["batch"])
        return [loss, grad]
    ctx = state["ctx"]
    if kind == "apply":
        y = ctx.apply(state["sigma"], state["out"], precision=PRECISION[case["precision"]])
        return y.float() if case["precision"] == "mixed" else y
    if kind == "step":
        ctx.set_state(0.0, state["cells"][0]["e2"], state["xc"], state["theta"])
        mu, _ = ctx.step(DT, STEPS)
        st = ctx.get_state()
        return [mu, st["xc"], st["theta"], st["sigma"]]
    if kind == "contact":
        ctx.set_state(0.0, state["e2"], state["xc"], state["theta"])
    sigma, _ = ctx.solve()
    v, omega, mu = ctx.velocities(sigma)
    return [sigma, v, omega, mu]


def _counts(case):
    """(nodes per cell, proxies, collocation points) of a case's cells."""
    cells = _cells(case, np.random.default_rng(0))
    return [sum(b["n"] for b in c["bodies"]) for c in cells], cells[0]["solver"]["n_proxy"], cells[0]["solver"]["n_coll"]


def work(case):
    """An application reads the density and the geometry (position, normal,
    weight, curvature) and writes the result.  Its arithmetic: every node's
    strength spreads to, and its traction is gathered from, a field that a
    few dozen coefficients describe locally, plus its neighbours' pair terms:
    40 coefficients of 16 operations each way, 256 pairs of 18.  A solve is
    about 70 applications, a step after the first two about 30."""
    if case["kind"] == "net":
        F, H = bie.BIE_NET_FEATURES, bie.BIE_NET_HIDDEN
        return dict(bytes=4.0 * case["rows"] * (F + 3), flops=6.0 * case["rows"] * (F * H + H * H + 2 * H))
    if case["kind"] == "contact":
        n = 2 * case["nodes"]
        return dict(bytes=60 * 80.0 * n, flops=60 * n * (2 * 16 * 40 + 18.0 * 256))
    ns, _, _ = _counts(case)
    per = 1
    if case["kind"] == "solve":
        per = 70
    elif case["kind"] == "step":
        per = 170
    return dict(bytes=per * 80.0 * sum(ns), flops=per * sum(ns) * (2 * 16 * 40 + 18.0 * 256))


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _t(a):
    return torch.as_tensor(np.asarray(a), dtype=torch.float64, device=_dev())


def _gauss(m):
    s, _ = np.polynomial.legendre.leggauss(m)
    return 0.5 * s


def _stokeslet(r, f, mu):
    """(1 / 4 pi mu) (-log|r| f + r (r.f) / r^2); last axis 2."""
    r2 = (r * r).sum(-1, keepdim=True)
    return (-0.5 * torch.log(r2) * f + r * (r * f).sum(-1, keepdim=True) / r2) / (4 * math.pi * mu)


def _traction(r, n, f):
    r2 = (r * r).sum(-1, keepdim=True)
    return -(r * n).sum(-1, keepdim=True) * (r * f).sum(-1, keepdim=True) * r / (math.pi * r2 * r2)


class _Exact:
    """The discretised periodic operator of one cell in 64 bits: boundary
    nodes of the ellipses, image sum, wall discrepancy, proxy fit, close
    evaluation by the interpolated density on a fine grid of the exact curve."""

    def __init__(self, cell, images=9):
        self.mu, self.gamma = cell["mu"], cell["gamma"]
        self.e1, self.e2, self.C = _t(cell["e1"]), _t(cell["e2"]), _t(cell["centre"])
        self.bodies, self.images = cell["bodies"], images
        xs, ns, ws, ks, own = [], [], [], [], []
        for b, bd in enumerate(self.bodies):
            x, d = self._curve(bd, bd["n"])
            sp = d.norm(dim=1)
            xs.append(x)
            ns.append(torch.stack([d[:, 1], -d[:, 0]], 1) / sp[:, None])
            ws.append(2 * math.pi / bd["n"] * sp)
            ks.append(bd["a"] * bd["b"] / sp ** 3)
            own.append(torch.full((bd["n"],), b, device=_dev()))
        self.x, self.n, self.w, self.kap = torch.cat(xs), torch.cat(ns), torch.cat(ws), torch.cat(ks)
        self.own = torch.cat(own)
        self.N, self.nb = len(self.w), len(self.bodies)
        self.off = np.cumsum([0] + [b["n"] for b in self.bodies])
        self.xc = _t([b["xc"] for b in self.bodies])
        # image multiples per node: all nine, or the four inside the doubled cell
        E = torch.stack([self.e1, self.e2], 1)
        st = torch.linalg.solve(E, (self.x - self.C).T).T
        if images == 4:
            m0 = torch.ceil(-1.0 - st)
            self.mn = [m0 + torch.tensor([i, j], device=_dev(), dtype=torch.float64) for j in (0, 1) for i in (0, 1)]
            self.m0 = m0
            self.xt = self.x - torch.floor(st + 0.5) @ E.T
        else:
            self.mn = [torch.tensor([[i, j]], device=_dev(), dtype=torch.float64) for j in (-1, 0, 1) for i in (-1, 0, 1)]
            self.xt = self.x
        self.E = E
        self._proxies(cell["solver"])
        self._close()

    @staticmethod
    def _curve(bd, n):
        t = torch.arange(n, dtype=torch.float64, device=_dev()) * (2 * math.pi / n)
        c, s = math.cos(bd["theta"]), math.sin(bd["theta"])
        R = _t([[c, -s], [s, c]])
        p = torch.stack([bd["a"] * torch.cos(t), bd["b"] * torch.sin(t)], 1)
        d = torch.stack([-bd["a"] * torch.sin(t), bd["b"] * torch.cos(t)], 1)
        return p @ R.T + _t(bd["xc"]), d @ R.T

    def _walls(self):
        s = _t(_gauss(self.m))[:, None]
        L = self.C - 0.5 * self.e1 + s * self.e2
        D = self.C - 0.5 * self.e2 + s * self.e1
        nl = torch.stack([self.e2[1], -self.e2[0]]) / self.e2.norm()
        nd = torch.stack([self.e1[1], -self.e1[0]]) / self.e1.norm()
        nl = nl if nl @ self.e1 < 0 else -nl
        nd = nd if nd @ self.e2 < 0 else -nd
        return [(L, nl, self.e1, self.e2), (D, nd, self.e2, self.e1)]

    def _proxies(self, sv):
        M, self.m = sv["n_proxy"], sv["n_coll"]
        if self.images == 4:
            s = ((torch.arange(M // 4, device=_dev(), dtype=torch.float64) + 0.5) / (M // 4) * 2 - 1)[:, None]
            self.yp = torch.cat([self.C + side * a + s * b for side in (-1, 1)
                                 for a, b in ((self.e1, self.e2), (self.e2, self.e1))])
        else:
            a = 2 * math.pi * torch.arange(M, device=_dev(), dtype=torch.float64) / M
            self.yp = self.C + sv["proxy_radius"] * torch.stack([torch.cos(a), torch.sin(a)], 1)
        cols = []
        for f in (_t([1.0, 0.0]), _t([0.0, 1.0])):
            rows = []
            for X, nu, a, _ in self._walls():
                r1, r0 = X[:, None] + a - self.yp[None], X[:, None] - self.yp[None]
                for g in (_stokeslet(r1, f, self.mu) - _stokeslet(r0, f, self.mu),
                          _traction(r1, nu, f) - _traction(r0, nu, f)):
                    rows += [g[..., 0], g[..., 1]]
            cols.append(torch.cat(rows))
        Q = torch.cat(cols, 1)
        lam = 1e-8 * Q.norm()
        A = torch.cat([Q, lam * torch.eye(Q.shape[1], device=_dev(), dtype=torch.float64)]).cpu().numpy()
        q, r = np.linalg.qr(A)
        self.P = _t(np.linalg.solve(r, q[: Q.shape[0]].T))

    def strengths(self, q):
        """Proxy strengths that cancel the wall discrepancy of the image sum."""
        F, rows = q.sum(0), []
        for k, (X, nu, a, b) in enumerate(self._walls()):
            S = torch.zeros(self.m, 2, device=_dev(), dtype=torch.float64)
            T = torch.zeros_like(S)
            if self.images == 4:
                j, i = (1, 0) if k == 0 else (0, 1)  # b and a multiples of a node
                terms = [(sg, self.m0[:, i:i + 1] + (-1 if sg > 0 else 1), self.m0[:, j:j + 1] + d)
                         for sg in (1, -1) for d in (0, 1)]
            else:
                terms = [(sg, -2.0 if sg > 0 else 1.0, d) for sg in (1, -1) for d in (-1.0, 0.0, 1.0)]
            for sg, ca, cb in terms:
                y = self.x + ca * a + cb * b
                for l in range(self.m):
                    r = X[l] - y
                    S[l] += sg * _stokeslet(r, q, self.mu).sum(0)
                    T[l] += sg * _traction(r, nu, q).sum(0)
            T = F / (2 * b.norm()) - T
            rows += [-S[:, 0], -S[:, 1], T[:, 0], T[:, 1]]
        return (self.P @ torch.cat(rows)).reshape(2, -1).T

    def _close(self):
        """Blocks of the close pairs, grouped by the source body's node count."""
        shifts = [(i * self.e1 + j * self.e2) for j in (-1, 0, 1) for i in (-1, 0, 1)]
        groups = {}
        for b, bd in enumerate(self.bodies):
            n, sl = bd["n"], slice(self.off[b], self.off[b + 1])
            h = float(self.w[sl].sum()) / n
            hmax = float(self.w[sl].max())
            dense = self._curve(bd, 16 * n)[0]
            for k, s in enumerate(shifts):
                dc = (self.x - self.xc[b] - s).norm(dim=1) - max(bd["a"], bd["b"])
                if k == 4:
                    dc[sl] = 1e9
                idx = torch.nonzero(dc < 10 * h)[:, 0]
                if not len(idx):
                    continue
                dn = torch.cdist(self.x[idx] - s, self.x[sl], compute_mode="donot_use_mm_for_euclid_dist").min(1).values
                idx = idx[dn < 10 * h]
                if not len(idx):
                    continue
                d = torch.cdist(self.x[idx] - s, dense, compute_mode="donot_use_mm_for_euclid_dist").min(1).values
                rho = 2 ** torch.ceil(torch.log2(0.5 + 6.4 * hmax / (0.95 * d))).clamp(min=1).long()
                for r in torch.unique(rho).tolist():
                    groups.setdefault(n, []).append(self._blocks(b, s, idx[rho == r], r))
        self.groups = [(n, torch.cat([g[0] for g in v]), torch.cat([g[1] for g in v]), torch.cat([g[2] for g in v]))
                       for n, v in groups.items()]

    def _blocks(self, b, s, idx, rho):
        bd = self.bodies[b]
        n = bd["n"]

        def kernel(y, w):
            r = self.x[idx][:, None] - y[None] - s
            r2 = (r * r).sum(-1)
            c = -(r * self.n[idx][:, None]).sum(-1) * w / (math.pi * r2 * r2)
            return torch.stack([c * r[..., 0] ** 2, c * r[..., 0] * r[..., 1], c * r[..., 1] ** 2], 1)
        y, d = self._curve(bd, rho * n)
        g = torch.fft.rfft(kernel(y, d.norm(dim=1) * (2 * math.pi / (rho * n))), dim=-1)
        fine = torch.fft.irfft(g[..., : n // 2 + 1], n=n, dim=-1)
        sl = slice(self.off[b], self.off[b + 1])
        return idx, torch.full_like(idx, int(self.off[b])), fine - kernel(self.x[sl], self.w[sl])

    def near(self, q):
        """Image sum of the traction kernel at every target (on-curve pair left out)."""
        T = torch.empty_like(self.x)
        step = max(1, (1 << 25) // self.N)
        for i in range(0, self.N, step):
            X, nn = self.xt[i:i + step], self.n[i:i + step]
            tx = ty = 0
            for mn in self.mn:
                y = self.x + mn @ self.E.T
                dx, dy = X[:, :1] - y[None, :, 0], X[:, 1:] - y[None, :, 1]
                r2 = dx * dx
                r2.addcmul_(dy, dy).clamp_(min=1e-28)
                c = dx * nn[:, :1]
                c.addcmul_(dy, nn[:, 1:])
                rq = dx * q[None, :, 0]
                rq.addcmul_(dy, q[None, :, 1])
                c.mul_(rq)
                c.div_(r2.mul_(r2))
                tx = tx + (c * dx).sum(1)
                ty = ty + (c * dy).sum(1)
            T[i:i + step] = torch.stack([tx, ty], 1) / -math.pi
        return T

    def apply(self, sigma):
        s = sigma.reshape(-1, 2)
        q = s * self.w[:, None]
        T = self.near(q)
        tau = torch.stack([-self.n[:, 1], self.n[:, 0]], 1)
        T += -(self.kap / (2 * math.pi))[:, None] * tau * (tau * q).sum(1, keepdim=True)
        xi = self.strengths(q)
        for i in range(0, self.N, 1 << 15):
            j = slice(i, i + (1 << 15))
            T[j] += _traction(self.xt[j, None] - self.yp[None], self.n[j, None], xi[None]).sum(1)
        for n, idx, off, blk in self.groups:
            sb = s[off[:, None] + torch.arange(n, device=_dev())]
            T.index_add_(0, idx, torch.stack([(blk[:, 0] * sb[..., 0] + blk[:, 1] * sb[..., 1]).sum(1),
                                              (blk[:, 1] * sb[..., 0] + blk[:, 2] * sb[..., 1]).sum(1)], 1))
        alpha = -(T[0] @ self.n[0])
        d = self.x - self.xc[self.own]
        F = torch.zeros(self.nb, 2, device=_dev(), dtype=torch.float64).index_add_(0, self.own, q)
        tq = torch.zeros(self.nb, device=_dev(), dtype=torch.float64).index_add_(0, self.own, d[:, 0] * q[:, 1] - d[:, 1] * q[:, 0])
        perp = torch.stack([-d[:, 1], d[:, 0]], 1)
        return (0.5 * s + T + alpha * self.n + F[self.own] + perp * tq[self.own][:, None]).reshape(-1)

    def solve(self, tol=2e-14):
        """GMRES on -T(u0): restarted until the true residual stops falling."""
        b = (-self.mu * self.gamma * torch.stack([self.n[:, 1], self.n[:, 0]], 1)).reshape(-1)
        x, best = torch.zeros_like(b), math.inf
        for _ in range(3):
            r = b - self.apply(x) if best < math.inf else b.clone()
            beta = r.norm()
            if not beta < 0.1 * best or beta <= tol * b.norm():
                break
            best = float(beta)
            V, H = [r / beta], []
            for k in range(250):
                w = self.apply(V[-1])
                Vm = torch.stack(V)
                h = Vm @ w
                w = w - h @ Vm
                g = Vm @ w
                w = w - g @ Vm
                hn = w.norm()
                H.append(torch.cat([h + g, hn[None]]).cpu().numpy())
                Hm = np.zeros((k + 2, k + 1))
                for j, col in enumerate(H):
                    Hm[: len(col), j] = col
                e = np.zeros(k + 2)
                e[0] = float(beta)
                y, res, *_ = np.linalg.lstsq(Hm, e, rcond=None)
                if np.linalg.norm(e - Hm @ y) <= tol * float(b.norm()) or float(hn) == 0:
                    break
                V.append(w / hn)
            x = x + _t(y) @ torch.stack(V[: len(y)])
        return x

    def velocities(self, sigma):
        s = sigma.reshape(-1, 2)
        q = s * self.w[:, None]
        xi = self.strengths(q)

        def velocity(X, y, f):
            return _stokeslet(X[:, None] - y[None], f[None], self.mu).sum(1)

        def curl(X, y, f):
            r = X[:, None] - y[None]
            return ((r[..., 1] * f[None, :, 0] - r[..., 0] * f[None, :, 1]) / (r * r).sum(-1)).sum(1) / (2 * math.pi * self.mu)
        u = velocity(self.xc, self.yp, xi) - velocity(self.C[None], self.yp, xi)
        om = curl(self.xc, self.yp, xi)
        for mn in self.mn:
            y = self.x + mn @ self.E.T
            u, om = u + velocity(self.xc, y, q), om + curl(self.xc, y, q)
        v = u + torch.stack([self.gamma * self.xc[:, 1], torch.zeros_like(om)], 1)
        area = abs(self.e1[0] * self.e2[1] - self.e1[1] * self.e2[0])
        mu = self.mu - (s[:, 0] * (self.x - self.xc[self.own])[:, 1] * self.w).sum() / (self.gamma * area)
        return v, 0.5 * (om - self.gamma), float(mu)


def _exact_steps(cell):
    e1, s0 = np.asarray(cell["e1"]), cell["e2"]
    mus = []
    for k in range(STEPS):
        op = _Exact(cell)
        sigma = op.solve()
        v, om, mu = (a.cpu().numpy() if torch.is_tensor(a) else a for a in op.velocities(sigma))
        mus.append(mu)
        sx = s0[0] + cell["gamma"] * (k + 1) * DT * s0[1]
        ex = sx / e1[0]
        e2 = np.array([sx - e1[0] * math.copysign(math.floor(abs(ex) + 0.5), ex), s0[1]])
        E, c = np.column_stack([e1, e2]), np.asarray(cell["centre"])
        bodies = []
        for b, bd in enumerate(cell["bodies"]):
            X = np.asarray(bd["xc"]) + DT * v[b]
            st = np.linalg.solve(E, X - c)
            bodies.append(dict(bd, xc=X - E @ np.floor(st + 0.5), theta=bd["theta"] + DT * om[b]))
        cell = dict(cell, bodies=bodies, e2=e2)
    return [np.array(mus), np.array([b["xc"] for b in cell["bodies"]]),
            np.array([b["theta"] for b in cell["bodies"]]), sigma.cpu().numpy()]


def _exact_net(case, seed):
    F, H = bie.BIE_NET_FEATURES, bie.BIE_NET_HIDDEN
    p, X, T, W = (_t(a) for a in _net_batch(case, np.random.default_rng(seed)))
    p.requires_grad_(True)
    W1, b1, W2, b2, W3, b3 = torch.split(p, [H * F, H, H * H, H, 2 * H, 2])
    a1 = torch.tanh(X @ W1.reshape(H, F).T + b1)
    a2 = torch.tanh(a1 @ W2.reshape(H, H).T + b2)
    Y = a2 @ W3.reshape(2, H).T + b3
    loss = (W[:, None] * (Y - T) ** 2).sum() / W.sum()
    loss.backward()
    return [float(loss), p.grad.cpu().numpy()]


def exact(case, seed):
    kind = case["kind"]
    if kind == "net":
        return _exact_net(case, seed)
    rng = np.random.default_rng(seed)
    if kind == "contact":
        cell, e2, xc, th = _contact(case, rng)
        bodies = [dict(b, xc=x, theta=t) for b, x, t in zip(cell["bodies"], xc, th)]
        op = _Exact(dict(cell, e2=e2, bodies=bodies))
    else:
        cells = _cells(case, rng)
        if kind == "apply":
            sigma, out, at = _t(_density(cells, rng)), [], 0
            for cell in cells:
                op = _Exact(cell, case["images"])
                out.append(op.apply(sigma[at:at + 2 * op.N]))
                at += 2 * op.N
            return torch.cat(out)
        if kind == "step":
            return _exact_steps(cells[0])
        op = _Exact(cells[0])
    sigma = op.solve()
    v, om, mu = op.velocities(sigma)
    return [sigma.cpu().numpy(), v.cpu().numpy(), om.cpu().numpy(), mu]
