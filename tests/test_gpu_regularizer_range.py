"""The standalone prox, g and g* over the range of their inputs' type: magnitudes
whose squares leave FP32's range at either end, sums beyond FP32's largest
value, one magnitude far above many equal ones (the candidates' rounded sums
then cross the target more than once), M = inf.

Tolerances are those of the ordinary magnitudes: the sums run in FP64, so g and
g* agree with the FP64 oracle to 1e-12 relative, the prox to 1e-12 (FP64) or one
rounding to FP32 (2^-22 relative; subnormal outputs 2^-149 absolute).
"""
import math

import numpy as np
import pytest

from oracle import regularizer as R

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
SCALES = [1e-38, 1e-24, 1e-17, 1.0, 1e20, 3e37]


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


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("p,k,rho,box", [(40, 3, 0.5, 2.0), (700, 10, 0.05, math.inf), (3001, 30, 3.0, 0.3)])
def test_prox_over_the_range(lib, p, k, rho, box, scale, dtype):
    v = _as(scale * np.clip(np.random.default_rng(p).standard_normal(p) * 3.0, -9.0, 9.0), dtype)
    _check_prox(lib, v, rho, k, box * scale, dtype)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("scale", SCALES)
@pytest.mark.parametrize("p,k,box", [(40, 3, 2.0), (700, 10, math.inf), (3001, 30, 0.3)])
def test_g_and_gstar_over_the_range(lib, p, k, box, scale, dtype):
    rng = np.random.default_rng(p + 1)
    b = np.zeros(p)
    at = rng.permutation(p)[:2 * k]
    b[at] = 0.25 * min(box, 1.0) * rng.uniform(-1, 1, at.size) * scale
    b = _as(b, dtype)
    M = box * scale
    # the squares themselves leave FP64's normal range at the lowest scale: 2^-1074 absolute
    assert lib.gval_persp(_dev(b, dtype), k, M) == pytest.approx(R.g_alg1(b, None, k, M, domain_rtol=1e-6), rel=1e-12, abs=1e-320)
    a = _as(scale * np.clip(rng.standard_normal(p) * 2.0, -9.0, 9.0), dtype)
    assert lib.gstar_persp(_dev(a, dtype), k, M) == pytest.approx(R.gstar(a, None, k, M), rel=1e-12, abs=1e-320)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_sums_beyond_fp32(lib, dtype):
    rng = np.random.default_rng(5)
    for t in range(8):
        v = _as(10.0 ** rng.uniform(35.5, 38.4, 600) * rng.choice([-1.0, 1.0], 600), dtype)
        _check_prox(lib, v, 10.0 ** rng.uniform(-6, 2), int(rng.integers(2, 40)), 10.0 ** rng.uniform(36, 39), dtype)


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
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
