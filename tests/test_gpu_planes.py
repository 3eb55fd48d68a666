"""Pass over a BF16 / FP8 copy of X with entries of beta and row weights far below
the largest of their strip or block, which X leaves out: z and g consist of the
small ones alone and have to keep their FP32 precision.

Against FP64 products with the emulated values; 2^-19 of the magnitude sums as at
the tile edges (test_gpu_xmma.py): the planes hold FP32 values exactly down to
2^-34 of the largest."""
import numpy as np
import pytest

from oracle import losses
from test_gpu_precision import PREC, dequantized

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("fmt", ["bf16", "fp8"])
@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("depth", [1e-2, 1e-4, 1e-8])
@pytest.mark.parametrize("shape", [(33, 240), (129, 961), (66, 20011)])
def test_small_entries_keep_their_bits(lib, shape, depth, loss, fmt):
    n, p = shape
    rng = np.random.default_rng(n + p)
    X = rng.standard_normal((n, p)).astype(np.float32)
    beta = depth * rng.standard_normal(p) * 10.0 ** rng.uniform(-1, 0, p)
    big = np.arange(3, p, 37)            # large coefficients, in the last third of the rows only
    beta[big] = rng.standard_normal(big.size)
    heavy = np.arange(n) % 3 == 2
    X[np.ix_(~heavy, big)] = 0.0
    light = np.arange(0, p, 5)           # columns that the rows of large weight leave out
    X[np.ix_(heavy, light)] = 0.0
    beta = beta.astype(np.float32)
    Xq, b64 = dequantized(X, fmt), beta.astype(np.float64)
    z_ref = Xq @ b64
    if loss == "ls":                     # residuals of the light rows are `depth` times the others'
        y = (z_ref + np.where(heavy, 1.0, depth) * rng.standard_normal(n)).astype(np.float32)
    else:                                # labels at random: the weights are about 1/2
        y = np.where(rng.standard_normal(n) >= 0, 1.0, -1.0).astype(np.float32)
    h = lib.Handle(torch.tensor(X, device="cuda"), torch.tensor(y, device="cuda"), loss=loss, k=1, lambda2=0.5,
                   lipschitz=1.0, precision=PREC[fmt])
    z, g, _ = h.xpass(torch.tensor(beta, device="cuda"))
    zg, gg = z.double().cpu().numpy(), g.double().cpu().numpy()
    h.close()
    r_ref = losses.grad_F(z_ref, y.astype(np.float64), loss)
    g_ref = Xq.T @ r_ref
    tol = 2.0 ** -19
    zmag = np.abs(Xq) @ np.abs(b64) + 1e-300
    gmag = np.abs(Xq).T @ np.abs(r_ref) + (2.0 if loss == "ls" else 0.25) * (np.abs(Xq).T @ zmag) + 1e-300
    assert np.all(np.abs(zg - z_ref) <= tol * zmag)
    assert np.all(np.abs(gg - g_ref) <= tol * gmag)
