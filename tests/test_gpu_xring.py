"""Pass over FP32 and FP64 X at the edges of its tiles: blocks of 8 (FP32) or 16
rows, strips of at most 192 16-byte vectors in boxes of at most 256 columns, one
and several strips and row groups, strips of fewer vectors than axpy warps.

z = X beta and g = X' r against FP64.  Tolerance: FP64 sums of at most 2^12
terms stay within 2^-41 of the terms' magnitudes (2^12 roundings of 2^-53), the
link's exp adds a few more; FP32 sums run over at most 24 columns per lane or 8
rows before they are compensated, and z, g and the logistic link are rounded to
FP32: within 2^-19.  The error of z passes into g with the link's slope (2, 1/4).
"""
import numpy as np
import pytest

from oracle import losses

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
SHAPES = [(1, 1), (7, 3), (8, 4), (9, 255), (16, 257), (17, 383), (31, 384), (33, 385), (64, 769), (129, 1537), (700, 97), (40, 9217)]


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("shape", SHAPES)
def test_pass_at_the_edges(lib, loss, shape, dtype):
    n, p = shape
    rng = np.random.default_rng(13 * n + p)
    X = rng.standard_normal((n, p)).astype(dtype)
    y = rng.standard_normal(n).astype(dtype)
    if loss == "logistic":
        y = np.where(y >= 0, 1.0, -1.0).astype(dtype)
    beta = (rng.standard_normal(p) * 10.0 ** rng.uniform(-3, 0, p)).astype(dtype)
    h = lib.Handle(torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda"), loss=loss, k=1, lambda2=0.5, lipschitz=1.0)
    z, g, _ = h.xpass(torch.tensor(beta, device="cuda"))
    zg, gg = z.double().cpu().numpy(), g.double().cpu().numpy()
    h.close()
    X64, b64 = X.astype(np.float64), beta.astype(np.float64)
    z_ref = X64 @ b64
    r_ref = losses.grad_F(z_ref, y.astype(np.float64), loss)
    g_ref = X64.T @ r_ref
    tol = 2.0 ** -41 if dtype == np.float64 else 2.0 ** -19
    zmag = np.abs(X64) @ np.abs(b64) + 1e-300
    gmag = np.abs(X64).T @ np.abs(r_ref) + (2.0 if loss == "ls" else 0.25) * (np.abs(X64).T @ zmag) + 1e-300
    assert np.all(np.abs(zg - z_ref) <= tol * zmag)
    assert np.all(np.abs(gg - g_ref) <= tol * gmag)
