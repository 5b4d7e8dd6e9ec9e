"""The process's first calls from several host threads at once, each with a context of its own (needs a GB300)."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# Every kernel's per-device set-up is done by whichever thread comes first; the
# others must not launch before it is done.  A fresh process each time: the
# kernels are loaded, slowly, on first use, which is when the threads meet.
SCRIPT = """
import sys, threading, traceback
sys.path.insert(0, %r)
import torch
from paper_2109_10375_gb300 import binding as B
T, n = 8, 64
torch.cuda.init()
J = torch.randn(n ** 3, device="cuda").exp_()
S, m = J.view(n, n, n), torch.ones(n, n, n, device="cuda")
psi = tuple(0.3 * torch.randn(n, n, n, device="cuda") for _ in range(3))
ref = torch.sort(J, descending=True, stable=True).indices.to(torch.int32)
h = B.history(8.0, 4.0, 3.0)
ctxs = [B.Context(n ** 3) for _ in range(T)]
streams = [torch.cuda.Stream() for _ in range(T)]
orders = [torch.empty_like(ref) for _ in range(T)]
zs = [torch.empty_like(S) for _ in range(T)]
rhos = [torch.empty_like(S) for _ in range(T)]
torch.cuda.synchronize()
start, failed = threading.Barrier(T), []
def work(i):
    try:
        start.wait()
        ctxs[i].rank(J, out=orders[i], stream=streams[i])
        ctxs[i].solve(S, m, 50.0, 3.0, h, out=zs[i], stream=streams[i])
        ctxs[i].mesh_density(psi, 50.0, 3, True, out=rhos[i], stream=streams[i])
        assert ctxs[i].sync_status(stream=streams[i]) == 0
    except Exception:
        failed.append(traceback.format_exc())
threads = [threading.Thread(target=work, args=(i,)) for i in range(T)]
[t.start() for t in threads]
[t.join() for t in threads]
torch.cuda.synchronize()
assert not failed, failed[0]
assert all(torch.equal(o, ref) for o in orders)
assert all(torch.equal(z, zs[0]) for z in zs)
assert all(torch.allclose(r, rhos[0], rtol=1e-5, atol=1e-4) for r in rhos)
"""


@pytest.mark.parametrize("attempt", range(3))
def test_first_calls_of_several_threads(attempt):
    import __graft_entry__ as g
    g.build()
    r = subprocess.run([sys.executable, "-c", SCRIPT % ROOT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
