"""Pass over a BF16 / FP8 copy of X at the edges of its tiles: blocks of 16 rows,
steps of two 16-byte vectors, boxes of an odd number of vectors, strips of
several boxes, one and several strips and row groups, odd counts of blocks.

z = Xq (s beta) and g = s (Xq' r) against FP64 products with the emulated
values.  Tolerance: products are exact, the operand's planes leave out at most
2^-17 of the smaller values and 2^-28 of the largest, each MMA's sum is off by
at most 2^-22 of its terms' magnitudes and the results are rounded to FP32; the
link of the logistic loss is FP32 (2^-21).  Together within 2^-19 of the
magnitude sums; the error of z passes into g with the link's slope (2 and 1/4).
"""
import numpy as np
import pytest

import synth
from oracle import losses
from test_gpu_precision import PREC, dequantized

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
SHAPES = [(1, 1), (15, 8), (16, 16), (17, 17), (31, 249), (33, 240), (48, 801), (65, 960), (129, 961), (500, 1633), (47, 20011)]


@pytest.mark.parametrize("fmt", ["bf16", "fp8"])
@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("shape", SHAPES)
def test_quantized_pass_edges(lib, fmt, loss, shape):
    n, p = shape
    rng = np.random.default_rng(17 * n + p)
    X = rng.standard_normal((n, p)).astype(np.float32)
    y = rng.standard_normal(n).astype(np.float32)
    if loss == "logistic":
        y = np.where(y >= 0, 1.0, -1.0).astype(np.float32)
    beta = (rng.standard_normal(p) * 10.0 ** rng.uniform(-3, 0, p)).astype(np.float32)
    h = lib.Handle(torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda"), loss=loss, k=1, lambda2=0.5,
                   lipschitz=1.0, precision=PREC[fmt])
    z, g, _ = h.xpass(torch.tensor(beta, device="cuda"))
    zg, gg = z.double().cpu().numpy(), g.double().cpu().numpy()
    h.close()
    Xq, b64 = dequantized(X, fmt), beta.astype(np.float64)
    z_ref = Xq @ b64
    r_ref = losses.grad_F(z_ref, y.astype(np.float64), loss)
    g_ref = Xq.T @ r_ref
    tol = 2.0 ** -19
    zmag = np.abs(Xq) @ np.abs(b64) + 1e-300
    gmag = np.abs(Xq).T @ np.abs(r_ref) + (2.0 if loss == "ls" else 0.25) * (np.abs(Xq).T @ zmag) + 1e-300
    assert np.all(np.abs(zg - z_ref) <= tol * zmag)
    assert np.all(np.abs(gg - g_ref) <= tol * gmag)
