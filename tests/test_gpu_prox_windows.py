"""The standalone prox with few coordinates between z = 0 and z = 1: a box far below
the magnitudes (the window (c, c + M) holds a few of them, and the roots of two
neighbouring pieces of the threshold's equation can name each other), and budgets
that the largest coordinates fill exactly (any c between two of them is a root).

Values to 1e-12 of the largest magnitude (FP64) or one rounding to FP32 plus that
of the input's own magnitudes (m - c: 2^-23), counts bit-exact: the inputs have no
ties."""
import math

import numpy as np
import pytest

from oracle import regularizer as R

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _check(lib, v, rho, k, M, dtype):
    if dtype == torch.float32:
        v = v.astype(np.float32).astype(np.float64)
    want, info = R.prox_g(v, rho, None, k, M, return_info=True)
    vin = torch.tensor(v, dtype=dtype, device="cuda")
    out = torch.empty_like(vin)
    counts = torch.zeros(2, dtype=torch.int32, device="cuda")
    lib.prox_persp(vin, out, rho / 2, k, 1.0, M, None, counts)
    got = out.double().cpu().numpy()
    scale = np.abs(v).max()
    tol = 1e-12 * scale + (2.0 ** -22 * np.abs(want) if dtype == torch.float32 else 0.0)
    assert np.all(np.abs(got - want) <= tol), (np.abs(got - want).max(), scale)
    assert tuple(counts.cpu().tolist()) == tuple(info)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("p", [9, 33, 225, 700, 5000])
def test_narrow_windows(lib, p, dtype):
    rng = np.random.default_rng(p)
    for _ in range(40):
        scale = 10.0 ** rng.uniform(-3, 3)
        v = scale * rng.standard_normal(p)
        M = scale * 10.0 ** rng.uniform(-4, 0)
        _check(lib, v, 10.0 ** rng.uniform(-4, 1), int(rng.integers(1, min(p, 60))), M, dtype)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("p", [9, 33, 225, 5000])
def test_budgets_filled_exactly(lib, p, dtype):
    rng = np.random.default_rng(p + 1)
    for _ in range(20):
        v = 10.0 ** rng.uniform(-3, 3) * rng.standard_normal(p)
        _check(lib, v, 10.0 ** rng.uniform(1, 3), int(rng.integers(1, min(p, 60))), [math.inf, 2.0][int(rng.integers(2))], dtype)
