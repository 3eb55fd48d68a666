"""The loop's own passes where standalone ones do not reach: two right-hand sides
(logistic loss: the gradient at the momentum point too) over BF16 / FP8 storage at
the edges of the tiles, and FP32 X beyond L2 (blocks of 8 rows) at odd sizes.

A solve of K iterations at a fixed step, without certification (no precision
ladder), on the stored X against the FP64 oracle on the same values: 1e-5 of the
largest coefficient, the bar of the FP32 trajectory tests.  The standalone pass
beyond L2: 2^-19 of the magnitude sums, as at the tile edges (test_gpu_xring.py)."""
import numpy as np
import pytest

import synth
from oracle import solver
from test_gpu_precision import PREC, dequantized

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def _solve_and_compare(lib, X, Xref, y, loss, k, L, precision, Ks):
    h_args = dict(loss=loss, k=k, lambda2=0.3, M=2.0, lipschitz=L, precision=precision, certify=False)
    Xd, yd = torch.tensor(X, device="cuda"), torch.tensor(y.astype(np.float32), device="cuda")
    for K in Ks:
        ref = solver.solve(Xref, y, loss, k, 0.3, 2.0, gap_tol=1e-300, L=L, max_iters=K)
        h = lib.Handle(Xd, yd, max_iters=K, **h_args)
        beta, res, _ = h.solve(gap_tol=1e-300)
        h.close()
        assert res.ladder == 0 and res.iters == ref.iters
        atol = 1e-5 * max(np.abs(ref.beta).max(), 1e-3)
        np.testing.assert_allclose(beta.double().cpu().numpy(), ref.beta, rtol=0, atol=atol)


@pytest.mark.parametrize("fmt", ["bf16", "fp8"])
@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("n,p", [(17, 249), (33, 961), (129, 240), (500, 1633), (47, 20011)])
def test_quantized_loop_at_the_edges(lib, n, p, loss, fmt):
    X, y = synth.make_problem_cpu(synth.Workload("loop", n, p, 0.5, 4, 0.3, loss, seed=n + p), dtype=np.float64)
    X, y = X.astype(np.float32), y.astype(np.float32).astype(np.float64)
    Xq = dequantized(X, fmt)
    _solve_and_compare(lib, X, Xq, y, loss, 4, solver.lipschitz(Xq, loss), PREC[fmt], (1, 10))


# (beyond three quarters of L2: 110 MB; remainders of rows, strips and boxes)
BIG = [(5003, 5501), (27509, 1003), (277, 99991)]


def _big(n, p, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(n, p, generator=g, device="cuda"), g


@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("n,p", BIG)
def test_pass_beyond_l2(lib, n, p, loss):
    X, g = _big(n, p, n)
    b = torch.randn(p, generator=g, device="cuda") * 10.0 ** (-3 * torch.rand(p, generator=g, device="cuda"))
    y = torch.randn(n, generator=g, device="cuda")
    y = torch.where(y >= 0, 1.0, -1.0) if loss == "logistic" else y
    h = lib.Handle(X, y, loss=loss, k=1, lambda2=0.5, lipschitz=1.0)
    z, gr, _ = h.xpass(b)
    h.close()
    X64, b64, y64 = X.double(), b.double(), y.double()
    z_ref = X64 @ b64
    r = 2 * (z_ref - y64) if loss == "ls" else -y64 * torch.sigmoid(-y64 * z_ref)
    g_ref = X64.t() @ r
    X64.abs_()
    zmag = X64 @ b64.abs()
    gmag = X64.t() @ r.abs() + (2.0 if loss == "ls" else 0.25) * (X64.t() @ zmag)
    assert bool(((z.double() - z_ref).abs() <= 2.0 ** -19 * zmag).all())
    assert bool(((gr.double() - g_ref).abs() <= 2.0 ** -19 * gmag).all())


@pytest.mark.parametrize("loss", ["ls", "logistic"])
@pytest.mark.parametrize("n,p", BIG[:2])
def test_loop_beyond_l2(lib, n, p, loss):
    X, g = _big(n, p, n + 1)
    z = X[:, ::p // 4].sum(dim=1)
    y = torch.where(z >= 0, 1.0, -1.0) if loss == "logistic" else z + torch.randn(n, generator=g, device="cuda")
    v = torch.ones(p, dtype=torch.float64, device="cuda")
    X64 = X.double()
    for _ in range(30):
        w = X64.t() @ (X64 @ (v / v.norm()))
        v = w
    L = (2.0 if loss == "ls" else 0.25) * 1.1 * float(v.norm())
    _solve_and_compare(lib, X.cpu().numpy(), X64.cpu().numpy(), y.double().cpu().numpy(), loss, 4, L, 0, (1, 6))
