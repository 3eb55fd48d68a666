"""The node p-phase (one thread-block cluster per problem) against the FP64
oracle at the edges of its layout: p around a warp's 32 and a CTA's 224
coordinates, one CTA to sixteen, a slack budget (k >= p), every coordinate
tied (equal columns: no bracket separates the thresholds and the searches end
without lists), and a batch that leaves its clusters unequal shares.

Tolerances: those of the solve's trajectory tests at a fixed step and iteration
count: FP64 1e-9 of the largest coefficient; FP32 data 1e-5 of it."""
import numpy as np
import pytest

import synth
from oracle import solver

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

N = 40


def _problem(p, loss, dtype, tied=False):
    w = synth.Workload("pnode", N, p, 0.5, 4, 0.3, loss, seed=p)
    X, y = synth.make_problem_cpu(w, dtype=np.float64)
    if tied:
        X = np.repeat(X[:, :1], p, axis=1)
        if loss == "ls":
            y = 3.0 * X[:, 0]
    return X.astype(dtype).astype(np.float64), y.astype(dtype).astype(np.float64)


def _check(got, want, dtype):
    scale = max(np.abs(want).max(), 1e-3)
    np.testing.assert_allclose(got, want, rtol=0, atol=(1e-9 if dtype == np.float64 else 1e-5) * scale)


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("p", [1, 31, 33, 224, 225, 449, 897, 3601])
def test_solve_at_the_edges(lib, p, loss, dtype):
    X, y = _problem(p, loss, dtype)
    L = solver.lipschitz(X, loss)
    k = min(5, p)
    fix = np.zeros(p, dtype=np.int8)
    if p > 30:
        fix[[0, p - 1]] = 1
        fix[3:9] = -1
    Xd, yd = torch.tensor(X.astype(dtype), device="cuda"), torch.tensor(y.astype(dtype), device="cuda")
    for K in (1, 12):
        ref = solver.solve(X, y, loss, k, 0.3, 2.0, fix=fix, gap_tol=1e-300, L=L, max_iters=K)
        h = lib.Handle(Xd, yd, loss=loss, k=k, lambda2=0.3, M=2.0, lipschitz=L, max_iters=K)
        beta, res, _ = h.solve(fixings=torch.tensor(fix, device="cuda"), gap_tol=1e-300)
        h.close()
        _check(beta.double().cpu().numpy(), ref.beta, dtype)
        assert res.dual_bound <= ref.primal + 1e-6 * max(1.0, abs(ref.primal))


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("p,k", [(40, 40), (300, 5), (1500, 7)])
def test_ties_and_slack_budgets(lib, p, k, loss, dtype):
    X, y = _problem(p, loss, dtype, tied=True)
    L = solver.lipschitz(X, loss)
    Xd, yd = torch.tensor(X.astype(dtype), device="cuda"), torch.tensor(y.astype(dtype), device="cuda")
    ref = solver.solve(X, y, loss, k, 0.3, 2.0, gap_tol=1e-300, L=L, max_iters=8)
    h = lib.Handle(Xd, yd, loss=loss, k=k, lambda2=0.3, M=2.0, lipschitz=L, max_iters=8)
    beta, res, _ = h.solve(gap_tol=1e-300)
    _, resb, _ = h.solve_batch(3, gap_tol=1e-300)
    h.close()
    _check(beta.double().cpu().numpy(), ref.beta, dtype)
    bar = 1e-9 if dtype == np.float64 else 1e-6
    assert abs(res.dual_bound - ref.dual_bound) <= bar * max(1.0, abs(ref.dual_bound))
    for r in resb:   # the batch's bar (2e-6): its products are rounded otherwise
        assert abs(r.dual_bound - ref.dual_bound) <= max(bar, 2e-6 if dtype == np.float32 else 0.0) * max(1.0, abs(ref.dual_bound))


@pytest.mark.parametrize("dtype", [np.float64, np.float32])
@pytest.mark.parametrize("loss", ["ls", "logistic"])
def test_batch_with_unequal_shares(lib, loss, dtype):
    p, nb, K = 1003, 9, 12
    X, y = _problem(p, loss, dtype)
    L = solver.lipschitz(X, loss)
    fix = np.stack([synth.node_fixings(p, 1, j, 20, 3, k=5) for j in range(nb)])
    h = lib.Handle(torch.tensor(X.astype(dtype), device="cuda"), torch.tensor(y.astype(dtype), device="cuda"), loss=loss, k=5,
                   lambda2=0.3, M=2.0, lipschitz=L, max_iters=K)
    betas, _, _ = h.solve_batch(nb, fixings=torch.tensor(fix, device="cuda"), gap_tol=1e-300)
    h.close()
    for s in range(nb):
        ref = solver.solve(X, y, loss, 5, 0.3, 2.0, fix=fix[s], gap_tol=1e-300, L=L, max_iters=K)
        _check(betas[s].double().cpu().numpy(), ref.beta, dtype)
