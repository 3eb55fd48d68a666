"""The standalone prox where the candidates' rounded sums cross the target more
than once: sums beyond FP32's largest value, one magnitude far above many equal
ones.

Tolerances are those of the ordinary magnitudes: 1e-12 relative (FP64) or one
rounding to FP32 (2^-22 relative).
"""
import numpy as np
import pytest

from oracle import regularizer as R

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _dev(a, dtype):
    return torch.tensor(np.asarray(a), dtype=dtype, device="cuda")


def _as(v, dtype):
    return v.astype(np.float32).astype(np.float64) if dtype == torch.float32 else v


def _check_prox(lib, v, rho, k, M, dtype):
    want, (ntop, nnz) = R.prox_g(v, rho, None, k, M, return_info=True)
    vin = _dev(v, dtype)
    out = torch.empty_like(vin)
    counts = torch.zeros(2, dtype=torch.int32, device="cuda")
    lib.prox_persp(vin, out, rho / 2, k, 1.0, M, None, counts)
    got = out.double().cpu().numpy()
    scale = np.abs(v).max()
    if dtype == torch.float64:
        np.testing.assert_allclose(got, want, rtol=1e-12, atol=1e-14 * scale)
    else:
        np.testing.assert_allclose(got, want, rtol=2.0 ** -22, atol=2.0 ** -149)
    assert counts.cpu().tolist() == [ntop, nnz]


@pytest.mark.parametrize("dtype", [torch.float64])
def test_sums_beyond_fp32(lib, dtype):
    rng = np.random.default_rng(5)
    for t in range(8):
        v = _as(10.0 ** rng.uniform(35.5, 38.4, 600) * rng.choice([-1.0, 1.0], 600), dtype)
        _check_prox(lib, v, 10.0 ** rng.uniform(-6, 2), int(rng.integers(2, 40)), 10.0 ** rng.uniform(36, 39), dtype)


@pytest.mark.parametrize("dtype", [torch.float64])
@pytest.mark.parametrize("big", [1e6, 1e10, 1e14])
def test_one_magnitude_far_above_ties(lib, big, dtype):
    # counts are left out: on ties they depend on the rounding of the threshold
    for m, rho in ((300, 1e-3), (900, 1e-8)):
        v = np.concatenate([[big, -big], np.ones(m)])
        want = R.prox_g(v, rho, None, 2, 10 * big)
        out = torch.empty(v.size, dtype=dtype, device="cuda")
        lib.prox_persp(_dev(v, dtype), out, rho / 2, 2, 1.0, 10 * big)
        got = out.double().cpu().numpy()
        # the ties' common value is a difference of sums of about `big`
        np.testing.assert_allclose(got, want, rtol=1e-12 if dtype == torch.float64 else 2.0 ** -22, atol=2.0 ** -48 * big)
