"""The network's gradient kernel at the edges of its tiles: 64 rows up to half of
the SMs' worth of 128-row tiles, 128 rows from there, one tile per CTA and
several.  The bar is the one of the oracle comparison: the FP32 sums run over at
most a few hundred rows per partial and the partials are summed in order, 1e-5
of the gradient's norm.
"""
import numpy as np
import pytest

from oracle import mlp
from test_gpu_warmstart import _dev, _feats, _rel, _theta

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("bf16", [False, True])
@pytest.mark.parametrize("N", [1, 15, 63, 64, 65, 9727, 9728, 9729, 19585])
def test_gradient_at_tile_edges(lib, bf16, N):
    F = _feats(N, seed=3 + N)
    th = _theta(seed=4, rows=F if N > 10 else None)
    rng = np.random.default_rng(N)
    base = F[:, 0]
    target = (base + 0.3 * rng.standard_normal(N)).astype(np.float32).astype(np.float64)
    grad = torch.empty(mlp.N_PARAM, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    lib.relax_mlp_grad(_dev(th), _dev(F), _dev(base), _dev(target), grad, loss, bf16=bf16)
    L_ref, g_ref = mlp.loss_and_grad(mlp.bf16_weights(th) if bf16 else th, F, base, target)
    assert _rel(grad.double().cpu().numpy(), g_ref) <= 1e-5
    assert float(loss.item()) == pytest.approx(L_ref, rel=1e-5)
