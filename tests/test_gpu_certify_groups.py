"""Certificates of many points at once (relax_certify_batch, groups of 32 that share
a launch) at sizes between the small parity cases and the large configurations:
clusters of 4 to 16 CTAs, 8 and 16 warps, few and many row groups whose partial
gradients a CTA's lanes sum on their own.

Phi and Psi against the FP64 oracle on the same points: 1e-9 relative to the terms'
magnitudes (FP32 data, float-float products), 1e-10 (FP64 data), the bars of
test_gpu_certify.py."""
import numpy as np
import pytest

from oracle import solver

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("n,p,nb,k", [(1079, 2668, 45, 30), (970, 2970, 27, 10), (2830, 2007, 35, 10), (4724, 1099, 33, 20),
                                      (300, 700, 64, 8)])
def test_groups_match_the_oracle(lib, n, p, nb, k, loss, dtype):
    rng = np.random.default_rng(n + p)
    X = rng.standard_normal((n, p)).astype(dtype)
    sup = np.arange(k) * p // k
    s = X[:, sup].sum(1)
    y = (s + rng.standard_normal(n) if loss == "ls" else np.where(s + 0.5 * rng.standard_normal(n) >= 0, 1.0, -1.0)).astype(dtype)
    fix = np.zeros((nb, p), dtype=np.int8)
    pts = np.zeros((nb, p), dtype=dtype)
    for j in range(nb):
        at = rng.permutation(p)
        n0, n1 = int(rng.integers(0, 41)), int(rng.integers(0, k))
        fix[j, at[:n0]] = -1
        fix[j, at[n0:n0 + n1]] = 1
        pts[j, sup] = 0.4 + 0.4 * rng.random(k)
        tail = rng.random(p) < 3 * k / p
        pts[j, tail & (pts[j] == 0)] = 0.02
        pts[j, fix[j] < 0] = 0.0
    X64, y64 = X.astype(np.float64), y.astype(np.float64)
    h = lib.Handle(torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda"), loss=loss, k=k, lambda2=0.5, M=2.0,
                   lipschitz=1.0)
    fd, pd = torch.tensor(fix, device="cuda"), torch.tensor(pts, device="cuda")
    got = np.asarray(h.certify_batch(pd, fd))
    h.close()
    bar = 1e-9 if dtype == np.float32 else 1e-10
    for j in range(nb):
        b = pts[j].astype(np.float64)
        phi = solver.primal(b, X64, y64, loss, fix[j], k, 2.0, 0.5)
        psi = solver.dual(solver.induced_dual(b, X64, y64, loss), X64, y64, loss, fix[j], k, 2.0, 0.5)
        scale = max(1.0, abs(phi) if np.isfinite(phi) else 1.0, abs(psi))
        assert (np.isinf(phi) and np.isinf(got[j, 0])) or abs(got[j, 0] - phi) <= bar * scale
        assert abs(got[j, 1] - psi) <= bar * scale
