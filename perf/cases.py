"""What a user has this library compute, as cases whose time and accuracy can be
measured: node relaxations one at a time and batched, the fused pass, the
certificate, the regularizer's operations and the warm-start network's training
step, each through the package's own calls.

A relaxation runs under an iteration budget (``max_iters``), as a node solve in
a branch and bound does: its work is then the same for every input.  The
budgets end before the gap reaches the floor of FP32 data, where the best
iterate (the least Phi) is one of several that rounding cannot tell apart.
"""
import math

import numpy as np
import torch

import paper_2603_01306_gb300 as relax
from paper_2603_01306_gb300.warmstart import WarmStartNet

BOX = 2.0                      # M, the box of the synthetic settings
ETA = math.exp(3.0)            # restart factor
DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.float32, "fp8": torch.float32}
PRECISION = {"f64": 0, "f32": 0, "bf16": relax.RELAX_BF16, "fp8": relax.RELAX_FP8E4M3}


def listed():
    return [
        # the root relaxation of the large least-squares configuration
        dict(name="solve_ls_f32_20000x50000", kind="solve", loss="ls", store="f32", n=20000, p=50000, rho=0.9, k=50,
             lambda2=0.1, iters=40, node=False),
        # the root relaxation of the paper's sweep (n = p), logistic, middle size
        dict(name="solve_logistic_f32_4000x4000", kind="solve", loss="logistic", store="f32", n=4000, p=4000, rho=0.5,
             k=10, lambda2=1.0, iters=100, node=False),
        # a child node at the sweep's smallest size: fixings, and its parent's solution as the start
        dict(name="solve_ls_f32_1000x1000_node", kind="solve", loss="ls", store="f32", n=1000, p=1000, rho=0.5, k=10,
             lambda2=1.0, iters=24, node=True),
        # the small reference configuration, double precision throughout
        dict(name="solve_ls_f64_500x1000", kind="solve", loss="ls", store="f64", n=500, p=1000, rho=0.5, k=10,
             lambda2=1.0, iters=100, node=False),
        # the tall logistic configuration (a quarter of its rows) on BF16 and on FP8 storage of X
        dict(name="solve_logistic_bf16_25000x20000", kind="solve", loss="logistic", store="bf16", n=25000, p=20000,
             rho=0.5, k=30, lambda2=0.1, iters=40, node=False),
        dict(name="solve_logistic_fp8_25000x20000", kind="solve", loss="logistic", store="fp8", n=25000, p=20000,
             rho=0.5, k=30, lambda2=0.1, iters=40, node=False),
        # the batched configuration: 256 nodes of one tree that share X
        dict(name="batch_ls_f32_5000x10000_256", kind="batch", loss="ls", store="f32", n=5000, p=10000, rho=0.7, k=20,
             lambda2=0.5, iters=30, nodes=256, warm=False),
        # the children of one step of the batched branch and bound, from their parents' solutions
        dict(name="batch_ls_f32_2000x5000_48", kind="batch", loss="ls", store="f32", n=2000, p=5000, rho=0.8, k=15,
             lambda2=0.2, iters=32, nodes=48, warm=True),
        # the certified values of a batch's starts (the learned start's fallback test)
        dict(name="certify_ls_f32_2000x5000_96", kind="certify", loss="ls", store="f32", n=2000, p=5000, rho=0.8, k=15,
             lambda2=0.2, nodes=96),
        # one product pair through a design with odd sizes and rows that start off 16 bytes
        dict(name="xpass_logistic_f32_3001x7003", kind="xpass", loss="logistic", store="f32", n=3001, p=7003, rho=0.7,
             k=20, lambda2=0.5),
        # the regularizer's own micro-benchmark at its small end: prox, value and conjugate
        dict(name="regularizer_f32_1000", kind="regularizer", store="f32", p=1000, k=10, box=1.0, rho=1.0, node=True),
        # one minibatch of the warm-start network's training
        dict(name="mlp_train_16384", kind="mlp", rows=16384, bf16=True),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "batch", "batch", "certify", "xpass", "regularizer", "mlp"])
    if kind == "regularizer":
        return dict(kind=kind, store=rng.choice(["f32", "f64"]), p=_log(rng, 300, 102400), k=rng.choice([5, 10, 50]),
                    box=rng.choice([1.0, 2.0]), rho=rng.choice([0.1, 1.0]), node=rng.random() < 0.5)
    if kind == "mlp":
        return dict(kind=kind, rows=_log(rng, 1000, 65536), bf16=rng.random() < 0.75)
    c = dict(kind=kind, loss=rng.choice(["ls", "logistic"]), store="f32", rho=rng.choice([0.5, 0.7, 0.8, 0.9]),
             k=rng.choice([10, 15, 20, 30]), lambda2=rng.choice([0.1, 0.2, 0.5, 1.0]))
    if kind == "solve":
        c.update(store=rng.choice(["f32", "f32", "bf16", "fp8", "f64"]), node=rng.random() < 0.5)
        c.update(iters=rng.randint(12, 20) if c["node"] else rng.randint(20, 32))
        if c["store"] == "f64":
            return {**c, "n": _log(rng, 300, 3000), "p": _log(rng, 500, 5000)}
        n = _log(rng, 500, 30000)
        return {**c, "n": n, "p": _log(rng, 800, min(50000, 500_000_000 // n))}
    if kind == "batch":
        c.update(iters=rng.randint(12, 24), nodes=_log(rng, 6, 200), warm=rng.random() < 0.5)
    if kind == "certify":
        c.update(nodes=_log(rng, 8, 128))
    if kind == "xpass":
        c.update(store=rng.choice(["f32", "f32", "f64"]))
    return {**c, "n": _log(rng, 500, 5000), "p": _log(rng, 1000, 10000)}


# ------------------------------------------------------------------- inputs
def _design(n, p, rho, dtype, g, offset=0):
    """Rows ~ N(0, rho^|i-j|): x_j = rho x_{j-1} + sqrt(1 - rho^2) e_j, 128 columns
    at a time.  offset > 0: rows of a wider buffer that start off 16 bytes."""
    X = torch.empty((n, p + offset), dtype=dtype, device="cuda")[:, offset:]
    w = 128
    i = torch.arange(w, device="cuda", dtype=torch.float64)
    lag = i[None, :] - i[:, None]
    T = torch.where(lag >= 0, rho ** lag.clamp(min=0), torch.zeros_like(lag)).to(dtype) * math.sqrt(1 - rho * rho)
    carry = (rho ** (i + 1)).to(dtype)
    last = torch.randn(n, generator=g, device="cuda", dtype=dtype)
    for j in range(0, p, w):
        m = min(w, p - j)
        blk = torch.randn(n, w, generator=g, device="cuda", dtype=dtype) @ T
        blk += last[:, None] * carry[None, :]
        X[:, j:j + m] = blk[:, :m]
        last = X[:, j + m - 1].clone()
    return X


def _problem(case, seed):
    """X, y (k equally spaced unit coefficients, SNR 5) and the Lipschitz constant
    of the loss's gradient, which a program that solves many nodes or several k
    and lambda2 on one design computes once."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, p, k = case["n"], case["p"], case["k"]
    dtype = DTYPES[case["store"]]
    X = _design(n, p, case["rho"], dtype, g, offset=1 if case["kind"] == "xpass" else 0)
    sup = torch.tensor([(i * p) // k for i in range(k)], device="cuda")
    s = X[:, sup].double().sum(dim=1)
    e = torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    if case["loss"] == "ls":
        y = s + (s.square().sum() / (5 * n)).sqrt() * e
    else:
        y = torch.where(s + 0.5 * e >= 0, 1.0, -1.0)
    v = torch.ones(p, device="cuda", dtype=dtype) / math.sqrt(p)
    for _ in range(40):
        w = X.t() @ (X @ v)
        norm = float(w.norm())
        v = w / norm
    return X, y.to(dtype), (2.0 if case["loss"] == "ls" else 0.25) * 1.1 * norm, g


def _node(p, k, g, rows=None):
    """Fixings of random nodes: up to 40 coordinates fixed out, up to k - 1 fixed in."""
    out = torch.zeros((rows or 1, p), dtype=torch.int8, device="cuda")
    for r in range(rows or 1):
        n0, n1 = (int(v) for v in torch.randint(0, 1 << 20, (2,), generator=g, device="cuda"))
        at = torch.randperm(p, generator=g, device="cuda")
        n0, n1 = n0 % 41, n1 % k
        out[r, at[:n0]] = -1
        out[r, at[n0:n0 + n1]] = 1
    return out if rows else out[0]


def _starts(p, k, g, dtype, rows):
    """What parents' solutions look like: the true support, shrunk, and a tail of
    small coefficients."""
    b = torch.zeros((rows, p), dtype=dtype, device="cuda")
    sup = torch.tensor([(i * p) // k for i in range(k)], device="cuda")
    b[:, sup] = 0.4 + 0.4 * torch.rand(rows, k, generator=g, device="cuda", dtype=dtype)
    tail = torch.rand(rows, p, generator=g, device="cuda") < 3 * k / p
    return torch.where(tail & (b == 0), 0.02 * torch.randn(rows, p, generator=g, device="cuda", dtype=dtype), b)


def _handle(case, X, y, L):
    return relax.Handle(X, y, loss=case["loss"], k=case["k"], lambda2=case["lambda2"], M=BOX, lipschitz=L,
                        precision=PRECISION[case["store"]], max_iters=case.get("iters", 0))


def _inputs(case, seed):
    """The case's data on the GPU, from the seed alone."""
    kind = case["kind"]
    if kind == "regularizer":
        g = torch.Generator(device="cuda").manual_seed(seed)
        p, dtype = case["p"], DTYPES[case["store"]]
        v = torch.randn(p, generator=g, device="cuda", dtype=dtype)
        fix = _node(p, min(case["k"], 4), g) if case["node"] else None
        # a point of the regularizer's domain: sum |b_j| <= M (k - |J1|), |b_j| <= M, zero where fixed out
        b = torch.zeros(p, dtype=dtype, device="cuda")
        at = torch.randperm(p, generator=g, device="cuda")[:2 * case["k"]]
        b[at] = 0.2 * case["box"] * (2 * torch.rand(at.numel(), generator=g, device="cuda", dtype=dtype) - 1)
        return dict(v=v, fix=fix, b=b if fix is None else torch.where(fix < 0, torch.zeros_like(b), b))
    if kind == "mlp":
        g = torch.Generator(device="cuda").manual_seed(seed)
        rows = case["rows"]
        feat = torch.randn(rows, 5, generator=g, device="cuda")
        feat[:, 2] = torch.randint(-1, 2, (rows,), generator=g, device="cuda").float()
        target = feat[:, 0] + 0.1 * torch.tanh(feat[:, 1] * feat[:, 3]) + 0.05 * feat[:, 4]
        theta = torch.zeros(relax.MLP_NPARAM, device="cuda")
        theta[:4609] = torch.randn(4609, generator=g, device="cuda") * 0.18
        theta[4614:] = 1.0
        m = 1e-3 * torch.randn(relax.MLP_NTRAIN, generator=g, device="cuda")
        v = 1e-4 + 1e-4 * torch.rand(relax.MLP_NTRAIN, generator=g, device="cuda")
        return dict(feat=feat, base=feat[:, 0].contiguous(), target=target, theta=theta, m=m, v=v, t=100)
    X, y, L, g = _problem(case, seed)
    d = dict(X=X, y=y, L=L)
    p, k = case["p"], case["k"]
    if kind == "solve":
        d["fix"] = _node(p, k, g) if case["node"] else None
        d["warm"] = _starts(p, k, g, X.dtype, 1)[0] if case["node"] else None
    elif kind == "batch":
        d["fix"] = _node(p, k, g, case["nodes"])
        d["warm"] = _starts(p, k, g, X.dtype, case["nodes"]) if case["warm"] else None
    elif kind == "certify":
        d["fix"] = _node(p, k, g, case["nodes"])
        d["points"] = torch.where(d["fix"] < 0, 0.0, _starts(p, k, g, X.dtype, case["nodes"])).to(X.dtype)
    else:
        d["beta"] = _starts(p, k, g, X.dtype, 1)[0]
    return d


def prepare(case, seed):
    d = _inputs(case, seed)
    d["case"] = case
    if case["kind"] == "regularizer":
        d["out"] = torch.empty_like(d["v"])
        d["counts"] = torch.empty(2, dtype=torch.int32, device="cuda")
    elif case["kind"] == "mlp":
        net = WarmStartNet(bf16=case["bf16"], theta=d["theta"].double().cpu().numpy())
        net.m.copy_(d["m"])
        net.v.copy_(d["v"])
        net.t = d["t"]
        d["net"] = net
    else:
        d["h"] = _handle(case, d["X"], d["y"], d["L"])
    return d


# ---------------------------------------------------------------------- run
def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "solve":
        beta, res, _ = s["h"].solve(fixings=s["fix"], warm_start=s["warm"], gap_tol=1e-12)
        return {"beta": beta, "bounds": np.array([res.primal, res.dual_bound], dtype=_np(case))}
    if kind == "batch":
        beta, res, _ = s["h"].solve_batch(case["nodes"], fixings=s["fix"], warm_start=s["warm"], gap_tol=1e-12)
        return {"beta": beta, "bounds": np.array([[r.primal, r.dual_bound] for r in res], dtype=_np(case))}
    if kind == "certify":
        return {"values": s["h"].certify_batch(s["points"], s["fix"])}
    if kind == "xpass":
        z, g, loss = s["h"].xpass(s["beta"])
        return {"z": z, "g": g, "loss": list(loss)}
    if kind == "regularizer":
        k, M = case["k"], case["box"]
        relax.prox_persp(s["v"], s["out"], 0.5 * case["rho"], k, 1.0, M, fixings=s["fix"], counts_out=s["counts"])
        g = relax.gval_persp(s["b"], k, M, fixings=s["fix"])
        gs = relax.gstar_persp(s["v"], k, M, fixings=s["fix"])
        return {"prox": s["out"], "counts": s["counts"], "g": g, "gstar": gs}
    net = s["net"]
    relax.relax_mlp_grad(net.theta, s["feat"], s["base"], s["target"], net.grad, net.loss, bf16=net.bf16)
    net.t += 1
    relax.relax_mlp_adam(net.theta, net.grad, net.m, net.v, net.t, 1e-3)
    return {"theta": net.theta, "m": net.m, "v": net.v, "grad": net.grad, "loss": net.loss}


def _np(case):
    """Bounds in the precision of the data."""
    return np.float64 if case["store"] == "f64" else np.float32


def work(case):
    kind = case["kind"]
    if kind == "regularizer":
        es = 8 if case["store"] == "f64" else 4
        return {"bytes": case["p"] * (4 * es + (3 if case["node"] else 0)), "flops": 30 * case["p"]}
    if kind == "mlp":
        return {"bytes": case["rows"] * 28 + 5 * 4609 * 4, "flops": 6.0 * case["rows"] * 4480}
    n, p = case["n"], case["p"]
    es = {"f64": 8, "f32": 4, "bf16": 2, "fp8": 1}[case["store"]]
    grads = 1 if case["loss"] == "ls" else 2      # logistic: the gradient at beta^t and at the momentum point
    if kind == "solve":
        # each iteration reads X once; so does the certificate, at full precision
        it = case["iters"] + 1
        master = 8 if case["store"] == "f64" else 4
        return {"bytes": float(n) * p * (it * es + master), "flops": (2.0 + 2.0 * grads) * n * p * it}
    if kind == "batch":
        # X is read once per iteration for all nodes, and each node's vectors
        it = case["iters"] + 1
        return {"bytes": float(it) * (n * p * es + case["nodes"] * 8.0 * (4 * p + 3 * n)),
                "flops": (2.0 + 2.0 * grads) * n * p * it * case["nodes"]}
    if kind == "certify":
        return {"bytes": float(n) * p * es + case["nodes"] * p * 5.0, "flops": 4.0 * n * p * case["nodes"]}
    return {"bytes": float(n) * p * es + (n + 2 * p) * es, "flops": 4.0 * n * p}


# --------------------------------------------------- the same in 64 bits
def _rows64(X):
    """X in 64 bits, a slice of rows at a time."""
    step = max(1, 100_000_000 // X.shape[1])
    for i in range(0, X.shape[0], step):
        yield i, min(X.shape[0], i + step), X[i:i + step].double()


class _Exact:
    """The relaxation of every row of `fix` in 64 bits on the design X: F, g, g*,
    the prox, and FISTA with the duality-gap restart."""

    def __init__(self, X, y, loss, k, lam, L, fix, M=BOX):
        self.X, self.y, self.loss, self.lam, self.L, self.M = X, y.double(), loss, lam, L, M
        self.fix = fix
        self.free, self.on = fix == 0, fix > 0
        self.kbar = (k - self.on.sum(1)).double()[:, None]

    def mul(self, b, X=None):
        z = torch.empty((b.shape[0], self.y.numel()), dtype=torch.float64, device=b.device)
        for i, j, x in _rows64(self.X if X is None else X):
            z[:, i:j] = b @ x.t()
        return z

    def tmul(self, r, X=None):
        g = 0
        for i, j, x in _rows64(self.X if X is None else X):
            g = g + r[:, i:j] @ x
        return g

    def loss_terms(self, z):
        """F(z), the loss's part of Psi at zeta = -grad F(z), and grad F(z)."""
        if self.loss == "ls":
            d = z - self.y
            return d.square().sum(1), (-2 * d * self.y - d.square()).sum(1), 2 * d
        t = self.y * z
        u = torch.sigmoid(-t)
        ent = -(torch.xlogy(u, u) + torch.xlogy(1 - u, 1 - u))
        return torch.nn.functional.softplus(-t).sum(1), ent.sum(1), -self.y * u

    def g(self, b):
        a = torch.where(self.free, b.abs(), 0.0).sort(1, descending=True).values
        tail = a.flip(1).cumsum(1).flip(1)                       # sum of a from position t on
        t = torch.arange(a.shape[1], device=a.device, dtype=torch.float64)[None]
        level = tail / (self.kbar - t).clamp(min=1)
        top = (((level >= a) & (t < self.kbar)).double().argmax(1))[:, None]   # the first position under the level
        head = a.square().cumsum(1) - a.square()
        few = ((a > 0).sum(1, keepdim=True) <= self.kbar)
        pooled = head.gather(1, top) + tail.gather(1, top).square() / (self.kbar - top).clamp(min=1)
        val = torch.where(few, a.square().sum(1, keepdim=True), pooled)[:, 0]
        out = 0.5 * (val + torch.where(self.on, b, 0.0).square().sum(1))
        bad = ((self.fix < 0) & (b != 0)).any(1) | (b.abs() > self.M * (1 + 1e-6)).any(1)
        return torch.where(bad | (tail[:, 0] > self.M * self.kbar[:, 0] * (1 + 1e-6)), math.inf, out)

    def huber(self, a):
        a = a.abs()
        return torch.where(a <= self.M, 0.5 * a * a, self.M * a - 0.5 * self.M ** 2)

    def gstar(self, a):
        h = self.huber(a)
        top = torch.where(self.free, h, 0.0).sort(1, descending=True).values
        keep = torch.arange(a.shape[1], device=a.device)[None] < self.kbar
        return torch.where(self.on, h, 0.0).sum(1) + (top * keep).sum(1)

    def prox(self, v, rho):
        """The prox of rho g: one threshold c per row, by bisection over its
        magnitude and the closed form on its piece."""
        M, kb = self.M, self.kbar
        m = torch.where(self.free, v.abs(), 0.0)
        lo = torch.full_like(kb, 1e-30)
        hi = m.amax(1, keepdim=True).clamp(min=1e-29)
        for _ in range(90):
            c = (lo * hi).sqrt()
            over = ((m - c).clamp(min=0) / (c / rho).clamp(max=M)).clamp(max=1).sum(1, keepdim=True) >= kb
            lo, hi = torch.where(over, c, lo), torch.where(over, hi, c)
        c = hi
        T = torch.where(c <= rho * M, c * (1 + rho) / rho, c + M)
        top = (m >= T).sum(1, keepdim=True).double()
        mid = (m > c) & (m < T)
        n, sm = mid.sum(1, keepdim=True).double(), (m * mid).sum(1, keepdim=True)
        closed = torch.where(c <= rho * M, rho * sm / (kb - top + rho * n), (sm - M * (kb - top)) / n)
        c = torch.where((n > 0) & (closed > 0), closed, c)
        few = (m > 0).sum(1, keepdim=True) <= kb
        c = torch.where(few, 0.0, c)
        out = torch.minimum(torch.minimum(m - c, m / (1 + rho)), torch.full_like(m, M)).clamp(min=0)
        out = torch.where(self.on, (v.abs() / (1 + rho)).clamp(max=M), out)
        T = torch.where(c <= rho * M, c * (1 + rho) / rho, c + M)
        out = torch.where(self.fix < 0, 0.0, out)
        tops = torch.stack([(self.free & (out > 0) & (m >= T)).sum(1), (self.free & (out > 0)).sum(1)], 1)
        return out * v.sign(), tops.int()

    def dual(self, z, X=None):
        _, d, r = self.loss_terms(z)
        return d - 2 * self.lam * self.gstar(self.tmul(r, X) / (2 * self.lam))

    def solve(self, warm, iters, master):
        """beta_best and (Phi(beta_best), the better Psi) on the master X after
        `iters` steps on this X."""
        rows, p = self.fix.shape
        b = torch.zeros((rows, p), dtype=torch.float64, device=self.fix.device) if warm is None else warm.double()
        prev, z_prev = b, None
        col = lambda v: torch.full((rows, 1), v, dtype=torch.float64, device=b.device)
        tau, ref, phi_best, psi_best = col(1.0), col(math.inf), col(math.inf), col(-math.inf)
        best, zd = b, None
        for t in range(iters + 1):
            z = self.mul(b)
            f, d, r = self.loss_terms(z)
            G = self.tmul(r)
            phi = (f + 2 * self.lam * self.g(b))[:, None]
            psi = (d - 2 * self.lam * self.gstar(G / (2 * self.lam)))[:, None]
            best = torch.where(phi < phi_best, b, best)
            zd = z if zd is None else torch.where(psi > psi_best, z, zd)
            phi_best, psi_best = torch.minimum(phi, phi_best), torch.maximum(psi, psi_best)
            gap = phi - psi
            again = (gap <= ref / ETA) & torch.isfinite(ref) & (t >= 1)
            ref = torch.where(again | (~torch.isfinite(ref) & torch.isfinite(gap)), gap, ref)
            nxt = 0.5 * (1 + (1 + 4 * tau * tau).sqrt())
            mu = torch.where(again, 0.0, (tau - 1) / nxt) if t else col(0.0)
            tau = torch.where(again, 1.0, nxt) if t else tau
            if t == iters:
                break
            y = b + mu * (b - prev)
            zy = z if z_prev is None else (1 + mu) * z - mu * z_prev
            v = y - self.tmul(self.loss_terms(zy)[2]) / self.L
            prev, z_prev = b, z
            b, _ = self.prox(v, 2 * self.lam / self.L)
        zb = self.mul(best, master)
        primal = self.loss_terms(zb)[0] + 2 * self.lam * self.g(best)
        return best, torch.stack([primal, torch.maximum(self.dual(zd, master), self.dual(zb, master))], 1)


class _Stored:
    """X as the loop stores it: BF16, or FP8 with a scale per column."""

    def __init__(self, X, store):
        self.X, self.store, self.shape = X, store, X.shape
        if store == "fp8":
            self.scale = X.abs().amax(0) / torch.full((1,), 448.0, device=X.device)   # a division, not a reciprocal

    def __getitem__(self, rows):
        x = self.X[rows]
        if self.store == "bf16":
            return x.bfloat16()
        return (x / self.scale).to(torch.float8_e4m3fn).double() * self.scale.double()


def exact(case, seed):
    d = _inputs(case, seed)
    kind = case["kind"]
    if kind == "regularizer":
        p = case["p"]
        fix = (torch.zeros(p, dtype=torch.int8, device="cuda") if d["fix"] is None else d["fix"])[None]
        e = _Exact(None, torch.zeros(1, device="cuda"), "ls", case["k"], 1.0, 1.0, fix, M=case["box"])
        out, tops = e.prox(d["v"].double()[None], case["rho"])
        return {"prox": out[0], "counts": tops[0], "g": float(e.g(d["b"].double()[None])),
                "gstar": float(e.gstar(d["v"].double()[None]))}
    if kind == "mlp":
        return _exact_mlp(case, d)
    X, y = d["X"], d["y"]
    fix = d.get("fix")
    fix = torch.zeros((1, case["p"]), dtype=torch.int8, device="cuda") if fix is None else fix.reshape(-1, case["p"])
    loop = _Stored(X, case["store"]) if case["store"] in ("bf16", "fp8") else X
    e = _Exact(loop, y, case["loss"], case["k"], case["lambda2"], d["L"], fix)
    if kind in ("solve", "batch"):
        warm = d["warm"] if d["warm"] is None else d["warm"].reshape(-1, case["p"])
        beta, bounds = e.solve(warm, case["iters"], X)
        return {"beta": beta if kind == "batch" else beta[0],
                "bounds": (bounds if kind == "batch" else bounds[0]).cpu().numpy()}
    if kind == "certify":
        b = d["points"].double()
        z = e.mul(b)
        return {"values": torch.stack([e.loss_terms(z)[0] + 2 * e.lam * e.g(b), e.dual(z)], 1).cpu().numpy()}
    z = e.mul(d["beta"].double()[None])
    f, dual, r = e.loss_terms(z)
    return {"z": z[0], "g": e.tmul(r)[0], "loss": [float(f), float(dual)]}


def _exact_mlp(case, d):
    """Mean squared error of base + f(x) and its gradient by reverse differentiation,
    then one Adam step."""
    theta = d["theta"].double()
    w = (d["theta"][:4609].bfloat16() if case["bf16"] else d["theta"][:4609]).double().requires_grad_()
    W1, b1, W2, b2, w3, b3 = w.split([320, 64, 4096, 64, 64, 1])
    x = (d["feat"].double() - theta[4609:4614]) / theta[4614:]
    h = torch.relu(x @ W1.view(64, 5).t() + b1)
    h = torch.relu(h @ W2.view(64, 64).t() + b2)
    loss = (d["base"].double() + h @ w3 + b3 - d["target"].double()).square().mean()
    g, = torch.autograd.grad(loss, w)
    t = d["t"] + 1
    m = 0.9 * d["m"].double() + 0.1 * g
    v = 0.999 * d["v"].double() + 0.001 * g * g
    theta[:4609] -= 1e-3 * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-8)
    return {"theta": theta, "m": m, "v": v, "grad": torch.cat([g, torch.zeros(10, device="cuda")]),
            "loss": loss.detach().reshape(1)}
