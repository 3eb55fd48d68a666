"""g where coefficients equal the water level of Algorithm 1 to rounding: the
level's search has to end although such a coefficient falls on either side of it in
turn.  At the boundary of the domain this is the usual case: sum |b_j| = M kbar puts
the level at M, where the box has put the largest coefficients.

g is continuous there: 1e-12 relative (FP64), 1e-9 (FP32), as at ordinary points."""
import numpy as np
import pytest

from oracle import regularizer as R

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("p", [40, 300, 3000])
def test_coefficients_at_the_level(lib, p, dtype):
    rng = np.random.default_rng(p)
    for _ in range(60):
        k = int(rng.integers(3, 20))
        m = int(rng.integers(1, k))                     # coefficients at the level
        n = int(rng.integers(k + 1, min(p, 4 * k)))
        rest = rng.uniform(0, 1, n)
        w = rest.sum() / (k - m)
        if rest.max() >= w:
            rest *= 0.9 * w / rest.max()
            w = rest.sum() / (k - m)
        b = np.zeros(p)
        at = rng.permutation(p)[:n + m] if n + m <= p else rng.permutation(p)
        vals = np.concatenate([np.full(m, w), rest])[:at.size]
        b[at] = vals * rng.choice([-1.0, 1.0], at.size)
        b = b.astype(dtype)
        b64 = b.astype(np.float64)
        M = float(np.abs(b64).max())
        want = R.g_alg1(b64, None, k, M, domain_rtol=1e-6)
        got = lib.gval_persp(torch.tensor(b, device="cuda"), k, M)
        assert got == pytest.approx(want, rel=1e-12 if dtype == np.float64 else 1e-9)


def test_solve_at_the_domains_boundary(lib):
    # small boxes: every budget is full after a few steps; the certified primal is Phi of the point returned
    from oracle import solver
    rng = np.random.default_rng(3)
    for t in range(40):
        n, p, k = int(rng.integers(20, 120)), int(rng.integers(30, 300)), int(rng.integers(2, 20))
        X = rng.standard_normal((n, p)).astype(np.float32).astype(np.float64)
        y = (X[:, :k].sum(1) * 3 + rng.standard_normal(n)).astype(np.float32).astype(np.float64)
        M, lam = 10.0 ** rng.uniform(-2, 0), 10.0 ** rng.uniform(-3, 0)
        h = lib.Handle(torch.tensor(X.astype(np.float32), device="cuda"), torch.tensor(y.astype(np.float32), device="cuda"),
                       k=k, lambda2=lam, M=M, lipschitz=solver.lipschitz(X, "ls"), max_iters=int(rng.integers(2, 12)))
        beta, res, code = h.solve(gap_tol=1e-300)
        h.close()
        assert code in (0, 4)
        assert res.primal == pytest.approx(res.primal_loop, rel=1e-5)
