"""Fixed-step solves of FP64 data whose magnitudes lie beyond FP32's range at
either end (the node p-phase brackets its thresholds on FP32 keys): the problem
is scaled by a power of ten, so that beta scales with it.  Against the FP64
oracle after the same iterations, 1e-9 of the largest coefficient as in the
trajectory tests at ordinary magnitudes."""
import numpy as np
import pytest

import synth
from oracle import solver

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("scale", [1e-60, 1e-42, 1.0, 1e42, 1e60])
@pytest.mark.parametrize("p,k", [(60, 60), (300, 5), (2000, 12)])
def test_fp64_solve_over_the_range(lib, p, k, scale):
    X, y = synth.make_problem_cpu(synth.Workload("range", 50, p, 0.5, min(k, 5), 0.3, "ls", seed=p), dtype=np.float64)
    L = solver.lipschitz(X, "ls")
    y = y * scale
    for K in (1, 10):
        ref = solver.solve(X, y, "ls", k, 0.3, 2.0 * scale, gap_tol=1e-300, L=L, max_iters=K)
        h = lib.Handle(torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda"), k=k, lambda2=0.3, M=2.0 * scale,
                       lipschitz=L, max_iters=K)
        beta, res, code = h.solve(gap_tol=1e-300)
        h.close()
        assert code != 6   # ENUMERIC
        np.testing.assert_allclose(beta.cpu().numpy(), ref.beta, rtol=0, atol=1e-9 * np.abs(ref.beta).max())
