"""The FP64 pair table is filled on first use, by several threads: the first FP64
contexts of a process, created by four host threads at once, give the oracle's
short-range forces (FP64 parity bound, 1e-9 of |g| + 1e-3 g_rms) and each other's
bit for bit."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUN = """
import threading
import numpy as np
import oracle as O
import paper_2005_05328_gb300 as dzs
kw = dict(n1d=16, mesh=32, box=32.0, merge_level=1)
rng = np.random.default_rng(3)
n = 4096
u = rng.integers(0, 2 ** 32, size=(3, n), dtype=np.uint64).astype(np.uint32)
u[:, : n // 2] = (u[:, n // 2:].astype(np.uint64) + rng.integers(0, 2 ** 26, size=(3, n // 2), dtype=np.uint64)) % 2 ** 32
k = np.ones(n, np.uint32)
st = dict(u=u, p=np.zeros((3, n)), g=np.zeros((3, n)), k=k, id=np.arange(n, dtype=np.uint32), fl=np.zeros(n, np.uint8))
dzs.load()
out = [None] * 4
def one(i):
    with dzs.Context(**kw, precision=1) as ctx:
        ctx.set_state(st, 0)
        out[i] = ctx.accel(dzs.ACC_TREE)
th = [threading.Thread(target=one, args=(i,)) for i in range(4)]
[t.start() for t in th]
[t.join() for t in th]
assert all(np.array_equal(o, out[0]) for o in out)
want = O.accel(O.params(**kw), u, k, parts=2)
err, ref = np.linalg.norm(out[0] - want, axis=0), np.linalg.norm(want, axis=0)
assert np.all(err <= 1e-9 * (ref + 1e-3 * np.sqrt((ref ** 2).mean())))
"""


def test_first_contexts_by_threads():
    from paper_2005_05328_gb300 import build
    build.build()
    subprocess.run([sys.executable, "-c", RUN], cwd=ROOT, check=True, timeout=300)
