"""Networks in CUDA contexts of the caller's own (lattices live in their
device's primary context): what the library keeps between objects belongs to
one context and goes with it.  Each case is a process of its own, without
torch."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PRELUDE = r"""
import ctypes
import numpy as np
import paper_1412_7228_gb300.lbm as L
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0
lib = L.lib()


def context():
    c = ctypes.c_void_p()
    assert cu.cuCtxCreate_v2(ctypes.byref(c), 0, 0) == 0     # and current
    return c


def fp(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_float))


rng = np.random.default_rng(3)
X = rng.uniform(-1, 1, (300, 3)).astype(np.float32)
Y = np.stack([X[:, 0] - 2 * X[:, 2], X[:, 1], X[:, 0] * X[:, 1], X[:, 2]], 1).astype(np.float32)


def surrogate():
    # a network trained, its predictions and an inversion
    m = ctypes.c_void_p()
    assert lib.lbm_mlp_create(ctypes.byref(m), 300, 7, None) == 0
    loss, out, k = np.zeros(3, np.float32), np.zeros((300, 4), np.float32), np.zeros(2, np.float32)
    assert lib.lbm_mlp_train(m, fp(X), fp(Y), 300, 3, 64, 1e-2, 5, fp(loss)) == 0
    assert lib.lbm_mlp_predict(m, fp(X), 300, fp(out)) == 0
    assert lib.lbm_mlp_invert_kappa(m, fp(X[:2, 0].copy()), fp(X[:2, 1].copy()), fp(out[:2, 0].copy()), 2, -2.0, 2.0, fp(k)) == 0
    lib.lbm_mlp_destroy(m)
    return loss, out, k
"""


def run(body):
    r = subprocess.run([sys.executable, "-c", PRELUDE + body], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr


def test_networks_in_a_second_context():
    run(r"""
a = context()
want = surrogate()
b = context()
for got in (surrogate(), surrogate()):
    assert all(np.array_equal(x, y, equal_nan=True) for x, y in zip(want, got))
""")


def test_networks_where_an_earlier_context_is_gone():
    run(r"""
a = context()
want = surrogate()
kept = ctypes.c_void_p()                                   # its block is still taken when its context goes
assert lib.lbm_mlp_create(ctypes.byref(kept), 300, 7, None) == 0
assert cu.cuCtxDestroy_v2(a) == 0
b = context()
for got in (surrogate(), surrogate()):
    assert all(np.array_equal(x, y, equal_nan=True) for x, y in zip(want, got))
c = context()
assert all(np.array_equal(x, y, equal_nan=True) for x, y in zip(want, surrogate()))
assert cu.cuCtxDestroy_v2(c) == 0
assert cu.cuCtxSetCurrent(b) == 0
assert all(np.array_equal(x, y, equal_nan=True) for x, y in zip(want, surrogate()))
""")
