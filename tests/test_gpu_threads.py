"""First launches of the kernels from several threads at once, each with its own context
and stream: the launchers' per-device settings (shared memory allowed, SM count)
must be in force for every thread's first launch."""
import subprocess
import sys
from pathlib import Path

import pytest

pytestmark = pytest.mark.gpu

CHILD = '''
import threading
import numpy as np, torch
from paper_1607_06834_gb300 import rok, workloads as W
probs = []
for n in (24, 300):
    probs.append(W.taylor_green(n))
    p, y, _ = W.cylinder_ogrid(n // 2, n)
    probs.append((p, y))
    probs.append(W.isentropic_vortex(n))
states = [(p, torch.from_numpy(np.ascontiguousarray(y)).cuda()) for p, y in probs] * 3
torch.cuda.synchronize()
out, start = [None] * len(states), threading.Barrier(len(states))
def work(k):
    p, y = states[k]
    stream = torch.cuda.Stream()
    ctx = rok.rok_init(p, krylov_max=2, stream=stream)
    f, jv = torch.empty_like(y), torch.empty_like(y)
    start.wait()
    rok.rok_residual(ctx, y, f)
    rok.rok_jvp(ctx, y, y, mode=rok.ROK_JVP_EXACT, out=jv)
    rok.rok_sync(ctx)
    out[k] = (f, jv)
threads = [threading.Thread(target=work, args=(k,)) for k in range(len(states))]
for t in threads: t.start()
for t in threads: t.join()
third = len(states) // 3
for k in range(third):
    assert all(out[k + third * i] is not None for i in range(3)), 'a thread failed'
    for a, b in ((0, 1), (0, 2)):
        for u, v in zip(out[k + third * a], out[k + third * b]):
            assert torch.equal(u, v) and torch.isfinite(u).all()
print('ok')
'''


def test_first_launches_from_several_threads():
    r = subprocess.run([sys.executable, '-c', CHILD], cwd=Path(__file__).resolve().parents[1], capture_output=True,
                       text=True, timeout=300)
    assert r.returncode == 0 and 'ok' in r.stdout, r.stdout + r.stderr
