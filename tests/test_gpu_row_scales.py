"""Pass over X whose rows or columns differ by orders of magnitude: z travels in
fixed point whose unit follows from the largest row and the largest |beta_j|, and
a row far below that bound keeps its bits.

z and g against FP64.  Tolerance: that of the passes at their tile edges, 2^-19
of the row's (column's) own magnitude sums.  The error of z passes into g with
the link's slope (2 and 1/4)."""
import numpy as np
import pytest

from oracle import losses
from test_gpu_precision import PREC, dequantized

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("store", ["f32", "bf16"])
@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("ratio", [1e4, 1e6, 1e8])
@pytest.mark.parametrize("heavy", ["row", "column"])
def test_light_rows_keep_their_bits(lib, heavy, ratio, loss, store):
    n, p = 67, 9001
    dtype = np.float32
    rng = np.random.default_rng(int(ratio) % 1000 + p)
    X = rng.standard_normal((n, p))
    beta = rng.standard_normal(p) * 10.0 ** rng.uniform(-3, 0, p)
    if heavy == "row":
        X[11] *= ratio
        X[40:] *= ratio ** rng.uniform(-1, 0, (n - 40, 1))
    else:   # a column in other units, which beta leaves out
        X[:, 5] *= ratio
        beta[5] = 0.0
    X, beta = X.astype(dtype), beta.astype(dtype)
    y = rng.standard_normal(n).astype(dtype)
    if loss == "logistic":
        y = np.where(y >= 0, 1.0, -1.0).astype(dtype)
    h = lib.Handle(torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda"), loss=loss, k=1, lambda2=0.5,
                   lipschitz=1.0, precision=PREC["bf16"] if store == "bf16" else 0)
    z, g, _ = h.xpass(torch.tensor(beta, device="cuda"))
    zg, gg = z.double().cpu().numpy(), g.double().cpu().numpy()
    h.close()
    X64 = dequantized(X, "bf16") if store == "bf16" else X.astype(np.float64)
    b64 = beta.astype(np.float64)
    z_ref = X64 @ b64
    r_ref = losses.grad_F(z_ref, y.astype(np.float64), loss)
    g_ref = X64.T @ r_ref
    tol = 2.0 ** -19
    zmag = np.abs(X64) @ np.abs(b64)
    gmag = np.abs(X64).T @ np.abs(r_ref) + (2.0 if loss == "ls" else 0.25) * (np.abs(X64).T @ zmag)
    assert np.all(np.abs(zg - z_ref) <= tol * zmag)
    assert np.all(np.abs(gg - g_ref) <= tol * gmag)
