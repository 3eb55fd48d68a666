"""Float-float pass over FP32 X at the edges of its tiles: blocks of 16 rows taken
in pairs, strips of at most 192 four-column vectors in boxes of at most 64, one
and several strips and row groups.  The certificate of a point (one product,
every row's z, every column's X' r) against the oracle in FP64.

Tolerance: z and X' r are sums of exact products kept to about 2^-46 of their
terms' magnitudes, r is an FP32 pair (2^-47) and the values are sums of squares,
or softplus terms, of them; 2^-37 (7e-12) of the magnitudes leaves room for the
up to 2^9 terms' signs.
"""
import numpy as np
import pytest

from oracle import solver

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
SHAPES = [(1, 1), (15, 3), (16, 4), (17, 767), (33, 768), (40, 769), (300, 1537), (1000, 30), (64, 9217)]


@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("shape", SHAPES)
def test_certificate_at_the_edges(lib, loss, shape):
    n, p = shape
    rng = np.random.default_rng(31 * n + p)
    X = rng.standard_normal((n, p)).astype(np.float32)
    y = rng.standard_normal(n).astype(np.float32)
    if loss == "logistic":
        y = np.where(y >= 0, 1.0, -1.0).astype(np.float32)
    k, M, lam = min(p, 5), 2.0, 0.5
    pts = np.zeros((3, p), dtype=np.float32)
    for s in range(3):
        idx = rng.choice(p, k, replace=False)
        pts[s, idx] = rng.uniform(-1.8, 1.8, k) * 10.0 ** rng.uniform(-4, 0, k)
    h = lib.Handle(torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda"), loss=loss, k=k, lambda2=lam, M=M,
                   lipschitz=1.0)
    got = h.certify_batch(torch.tensor(pts, device="cuda"), torch.zeros((3, p), dtype=torch.int8, device="cuda"))
    h.close()
    X64, y64, fo = X.astype(np.float64), y.astype(np.float64), np.zeros(p, dtype=np.int8)
    for s in range(3):
        b = pts[s].astype(np.float64)
        zeta = solver.induced_dual(b, X64, y64, loss)
        phi = solver.primal(b, X64, y64, loss, fo, k, M, lam)
        psi = solver.dual(zeta, X64, y64, loss, fo, k, M, lam)
        zmag = np.abs(X64) @ np.abs(b) + np.abs(y64)
        gmag = np.abs(X64).T @ (np.abs(zeta) + zmag)
        mag = 1.0 + (zmag ** 2).sum() + M * np.sort(gmag)[-k:].sum()
        assert abs(got[s, 0] - phi) <= 2.0 ** -37 * mag, (got[s, 0], phi)
        assert abs(got[s, 1] - psi) <= 2.0 ** -37 * (mag + (gmag ** 2).max() / lam), (got[s, 1], psi)
