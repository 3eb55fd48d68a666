"""relax_result.launches of a batched call: the kernels that it launched, the same
from the first call (which captures its graphs) and from later ones (which only
launch them).  A round is 16 iterations and the test of the nodes' ends; an
iteration of FP32 data is two products, the link and the p-phase, with the
operand's packing once per round; of FP64 data and with backtracking the packing,
two products, the link, the gradients and the p-phase.  Around the rounds: the
starts, the results and, with fixings, their count.  The nodes stop together at
max_iters; certificates add a pass per node and an evaluation per 32."""
import numpy as np
import pytest

import synth
from oracle import solver

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype,backtrack", [(np.float32, False), (np.float64, False), (np.float32, True)])
@pytest.mark.parametrize("certify", [True, False])
@pytest.mark.parametrize("fixed", [True, False])
def test_batch_counts_its_launches(lib, dtype, backtrack, certify, fixed):
    p, nb, K = 500, 35, 20
    X, y = synth.make_problem_cpu(synth.Workload("count", 60, p, 0.5, 5, 0.3, "ls", seed=1), dtype=dtype)
    h = lib.Handle(torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda"), k=5, lambda2=0.3, M=2.0,
                   lipschitz=solver.lipschitz(X.astype(np.float64), "ls"), max_iters=K, certify=certify,
                   step="backtracking" if backtrack else "fixed")
    fix = torch.zeros(nb, p, dtype=torch.int8, device="cuda") if fixed else None
    per_iter, per_round = (4, 2) if dtype == np.float32 and not backtrack else (6, 1)
    rounds = K // 16 + 1
    want = 2 + fixed + rounds * (16 * per_iter + per_round) + certify * (nb + 2)
    for _ in range(2):
        _, res, _ = h.solve_batch(nb, fixings=fix, gap_tol=1e-300)
        assert [r.iters for r in res] == [K] * nb
        assert [r.launches for r in res] == [want] * nb
    h.close()
