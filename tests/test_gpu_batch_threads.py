"""A batched solve when the process can have no more threads: the failure of
std::thread must not leave the C entry (it would end the process), and the
calling thread solves every system itself.  Thread creation is made to fail on
the host, by a default stack size that no address space holds, after the
process's CUDA context and first solves exist; the solve's results must be
those of the solve with threads, to 1e-9 as for a system alone (the FP64
spreading of a second refinement sweep sums with atomics)."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SCRIPT = r"""
import ctypes
import threading
import numpy as np
import paper_2607_25161_gb300 as fsd
import synth

systems = [synth.suspension(30 + 5 * k, 4, 0.1, 80 + k) for k in range(4)]
b = fsd.Batch(systems, dict(precision=fsd.FSD_MIXED, lub_cutoff=3.0))
ft = synth.random_forces(b.n_agg, 4)
want = b.solve(ft, 1.0)[:2]
b.solve(ft, 1.0)
libc = ctypes.CDLL(None, use_errno=True)
attr = ctypes.create_string_buffer(256)
assert libc.pthread_attr_init(attr) == 0
assert libc.pthread_attr_setstacksize(attr, ctypes.c_size_t(1 << 50)) == 0
assert libc.pthread_setattr_default_np(attr) == 0
try:
    threading.Thread(target=int).start()
    raise SystemExit("a thread could still be started")
except RuntimeError:
    pass
got = b.solve(ft, 1.0)[:2]
for x, y in zip(got, want):
    assert np.linalg.norm(x - y) <= 1e-9 * np.linalg.norm(y)
b.close()
print("done")
"""


def test_batch_solves_without_more_threads():
    import __graft_entry__ as g

    g.build()
    r = subprocess.run([sys.executable, "-c", SCRIPT], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "done" in r.stdout, r.stdout[-2000:] + r.stderr[-2000:]
