"""Host threads of one fresh process whose first calls are standalone prox calls
of different sizes: every thread's plan raises the same kernel's limit of dynamic
shared memory, and no launch may be refused for another thread's smaller one.
Each thread's results equal those of the same calls made by one thread."""
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
pytest.importorskip("torch")

CHILD = """
import threading, torch
import paper_2603_01306_gb300 as relax
relax.load()
sizes = [[1000 * (1 + (7 * t + 13 * i) % 100) for i in range(12)] for t in range(12)]
v = torch.randn(101000, generator=torch.Generator().manual_seed(1)).cuda()
torch.cuda.synchronize()
got, errors = {}, []
start = threading.Barrier(len(sizes))
def work(t):
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        start.wait()
        try:
            for p in sizes[t]:
                out = torch.empty(p, device="cuda")
                relax.prox_persp(v[:p], out, 0.1, 10, 1.0, 2.0)
                st.synchronize()
                got[t, p] = out
        except Exception as e:
            errors.append(repr(e))
threads = [threading.Thread(target=work, args=(t,)) for t in range(len(sizes))]
[t.start() for t in threads]
[t.join() for t in threads]
assert not errors, errors
for (t, p), g in got.items():
    want = torch.empty(p, device="cuda")
    relax.prox_persp(v[:p], want, 0.1, 10, 1.0, 2.0)
    torch.cuda.synchronize()
    assert torch.equal(g, want), (t, p)
"""


@pytest.mark.parametrize("run", range(3))
def test_first_calls_from_several_threads(lib, run):
    r = subprocess.run([sys.executable, "-c", CHILD], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
