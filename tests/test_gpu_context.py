"""The library after cudaDeviceReset, in a process of its own (the reset ends only that process's context):
what it keeps for the life of the process (memory pools, pinned result blocks, kernel attributes) belongs
to a context and is made again in the next one."""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = r"""
import ctypes, sys
import numpy as np
import paper_1606_04473_gb300 as ara
cr = ctypes.CDLL("libcudart.so")
L = ara.lib()
P = ctypes.c_void_p

def ok(st):
    assert st == 0, (st, cr.cudaGetLastError())

def up(a):
    p = P()
    ok(cr.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(a.nbytes)))
    ok(cr.cudaMemcpy(p, a.ctypes.data_as(P), ctypes.c_size_t(a.nbytes), 1))
    return p

def session():
    g = np.random.default_rng(1)
    C, n, nl = 20_000, 30_011, 40
    ids = [g.choice(C, size=900, replace=False).astype(np.int32) for _ in range(nl)]
    z = np.zeros(nl)
    pf = ara.Portfolio(C, ids, [np.exp(g.normal(11, 2, 900)) for _ in ids], z, z + 1e9, [[l] for l in range(nl)], z + 1e4,
                       z + 1e6, z, z + 1e8)
    off, ev = np.arange(n + 1, dtype=np.int64) * 30, g.integers(0, C, 30 * n, dtype=np.int32)
    y = np.zeros((nl, n))
    d_off, d_ev, d_y = up(off), up(ev), up(y)
    n0 = ara.launch_count()
    ok(L.ara_run_ylt(pf._h, n, d_off, ev.size, d_ev, None, 0, None, d_y, None, 0, None))
    assert ara.launch_count() - n0 <= 3          # by rows, with scratch from the pool
    ok(L.ara_check(pf._h, None))
    out = []
    rp, lv = np.array([100.0, 10.0]), np.array([0.99])
    for rows, fn in ((2, L.ara_risk_metrics), (nl, L.ara_risk_metrics), (2, L.ara_risk_metrics_static)):
        a, b, m = np.zeros((rows, 2)), np.zeros((rows, 1)), np.zeros(rows)
        ok(fn(d_y, n, rows, 2, rp.ctypes.data_as(P), 1, lv.ctypes.data_as(P), a.ctypes.data_as(P), b.ctypes.data_as(P),
              m.ctypes.data_as(P), None))
        out += [a, b, m]
    ok(cr.cudaMemcpy(y.ctypes.data_as(P), d_y, ctypes.c_size_t(y.nbytes), 2))
    pf.close()
    for d in (d_off, d_ev, d_y):
        ok(cr.cudaFree(d))
    return out + [y]

first = session()
assert (first[-1] > 0).any()
for again in range(2):
    ok(cr.cudaDeviceReset())
    for x, y in zip(first, session()):
        assert np.array_equal(x, y)
    ok(L.ara_release_memory())
    for x, y in zip(first, session()):
        assert np.array_equal(x, y)
print("done")
"""


def test_calls_after_a_device_reset():
    env = dict(os.environ, LD_LIBRARY_PATH="/usr/local/cuda/lib64:" + os.environ.get("LD_LIBRARY_PATH", ""))
    if not os.path.exists("/usr/local/cuda/lib64/libcudart.so"):
        pytest.skip("no shared CUDA runtime to reset the device with")
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and r.stdout.strip() == "done", r.stdout + r.stderr
