"""The precision ladder's FP32 rung (BF16 storage, FP32 passes over the master X)
takes its loss terms in FP64: the loop's own Phi is that of its point.

A weak signal (large lambda2, z about 0.02) makes the rounding of the loss terms
themselves the largest error there could be: FP32 terms of about ln 2 are each off
by up to 2^-25, a sum of 64 by 7e-8 to 5e-7 here (the same terms in NumPy).  What
FP32 passes leave is z's error, at most 2^-24 of a row's magnitudes, times the
link's slope 1/2, independent over the rows: three standard deviations, plus 2^-40
for the sums."""
import numpy as np
import pytest

import synth
from oracle import losses, regularizer, solver

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("seed", range(5))
def test_fp32_rung_sums_the_loss_in_fp64(lib, seed):
    lam, k, M = 1000.0, 5, 2.0
    X, y = synth.make_problem_cpu(synth.Workload("ladder", 64, 400, 0.5, k, lam, "logistic", seed=seed), dtype=np.float64)
    X = X.astype(np.float32).astype(np.float64)
    h = lib.Handle(torch.tensor(X.astype(np.float32), device="cuda"), torch.tensor(y.astype(np.float32), device="cuda"),
                   loss="logistic", k=k, lambda2=lam, M=M, lipschitz=solver.lipschitz(X, "logistic"),
                   precision=lib.RELAX_BF16)
    beta, res, code = h.solve(gap_tol=1e-7)
    h.close()
    assert code == 0 and res.ladder == 1
    b = beta.double().cpu().numpy()
    phi = losses.F(X @ b, y, "logistic") + 2 * lam * regularizer.g_alg1(b, None, k, M, domain_rtol=1e-6)
    tol = 3 * 0.5 * 2.0 ** -24 * np.linalg.norm(np.abs(X) @ np.abs(b)) + 2.0 ** -40 * phi
    assert abs(res.primal_loop - phi) <= tol
