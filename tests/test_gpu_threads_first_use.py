"""The first calls of a process from several threads at once, each on a stream of its own: the tables of cluster launches
and the kernels' attributes are set up once, and every thread gets what a single-threaded call gets, bit for bit. Runs in
a child process, so that the calls are the first."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

CHILD = """
import threading
import numpy as np, torch
import paper_2201_05529_gb300 as pkg
capi = pkg.load()
m, n, batch, threads = 300, 96, 3, 8
rng = np.random.default_rng(5)
A = torch.from_numpy(rng.standard_normal((batch, n, m)) + 1j * rng.standard_normal((batch, n, m))).cuda()
work = [(A.clone(), torch.zeros((batch, n, n), dtype=torch.complex128, device="cuda"), torch.cuda.Stream())
        for _ in range(threads + 1)]
torch.cuda.synchronize()
sizes, errors, go = [None] * threads, [], threading.Barrier(threads)
def one(i):
    try:
        if i < threads:
            go.wait()
        with torch.cuda.stream(work[i][2]):
            size = capi.qr_scratch_bytes(m, n, batch)
            capi.qr_f64(work[i][0], work[i][1], torch.empty(size, dtype=torch.uint8, device="cuda"))
            if i < threads:
                sizes[i] = capi.svd_scratch_bytes(m, n, batch)
    except Exception as e:
        errors.append(repr(e))
ts = [threading.Thread(target=one, args=(i,)) for i in range(threads)]
[t.start() for t in ts]; [t.join() for t in ts]
one(threads)
torch.cuda.synchronize()
assert not errors, errors
assert set(sizes) == {capi.svd_scratch_bytes(m, n, batch)}
for q, r, _ in work[:-1]:
    assert torch.equal(q, work[-1][0]) and torch.equal(r, work[-1][1])
print("SAME")
"""


def test_first_calls_from_several_threads():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2201_05529_gb300 as pkg
    pkg.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "SAME" in r.stdout, r.stdout + r.stderr
