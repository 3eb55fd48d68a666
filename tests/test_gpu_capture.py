"""Calls that do not synchronise can be captured in a CUDA graph, also as the first
call of a process: the prox (on a cluster, and wide enough for the cooperative grid
and its scratch) and the network's gradient.  A replay gives what a plain call
gives."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

CHILD = """
import sys, torch
import paper_2603_01306_gb300 as relax
relax.load()
gen = torch.Generator(device="cuda").manual_seed(1)
if sys.argv[1] == "mlp":
    theta = 0.1 * torch.randn(relax.MLP_NPARAM, generator=gen, device="cuda")
    theta[-5:] = 1.0
    feat = torch.randn(5000, 5, generator=gen, device="cuda")
    base, target = feat[:, 0].contiguous(), feat[:, 1].contiguous()
    call = lambda out: relax.relax_mlp_grad(theta, feat, base, target, out)
    new = lambda: torch.zeros(relax.MLP_NPARAM, device="cuda")
else:
    v = torch.randn(int(sys.argv[1]), generator=gen, device="cuda")
    call = lambda out: relax.prox_persp(v, out, 0.5, 10, 1.0, 1.0)
    new = lambda: torch.empty_like(v)
got, want = new(), new()
torch.cuda.synchronize()
graph = torch.cuda.CUDAGraph()
with torch.cuda.graph(graph):
    call(got)
graph.replay()
graph.replay()
torch.cuda.synchronize()
call(want)
torch.cuda.synchronize()
assert torch.equal(got, want)
"""


@pytest.mark.parametrize("what", ["1000", "150000", "mlp"])
def test_first_call_in_a_capture(lib, what):
    r = subprocess.run([sys.executable, "-c", CHILD, what], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
