"""When and how results are waited for: a status is that of all the work issued
so far, and a device set to block leaves the core to others."""
import numpy as np
import pytest

from test_gpu_reductions import _law

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1412_7228_gb300 as P
    P.lib()
    return P


def test_a_status_asked_for_is_that_of_all_the_work_issued(P):
    """A read of no field returns the status alone: after the steps still
    running, and after the reset by a new initial field."""
    eos, A = _law(P, "cs")
    rg, rl, _ = P.lbm_eos_maxwell(eos)
    n = 2048                      # an FP64 step takes more than a millisecond
    lat = P.Lattice(n, n, P.LBM_FP64)
    lat.set_params(eos, A, 0.3, rho_ref=rg)
    good = np.full((n, n), 0.2)
    bad = good.copy()
    bad[n - 3, n - 3] = 0.7       # outside psi's domain, in the step's last tile
    for _ in range(5):
        lat.init_density(bad)
        lat.step(1)
        with pytest.raises(P.LbmError) as ei:
            lat.read_fields(which=())
        assert ei.value.code == P.lbm.LBM_EUNSTABLE
        lat.init_density(good)
        assert lat.read_fields(which=()) == {}
    lat.close()


BLOCKING = r"""
import ctypes, sys, time
cu = ctypes.CDLL("libcuda.so.1")
assert cu.cuInit(0) == 0 and cu.cuDevicePrimaryCtxSetFlags_v2(0, 4) == 0     # CU_CTX_SCHED_BLOCKING_SYNC
import numpy as np
import paper_1412_7228_gb300 as P
eos = P.Eos(kind=P.LBM_EOS_CS, a=1.0, b=4.0, R=1.0, K=1.0, T=0.066)
lat = P.Lattice(1024, 1024, P.LBM_FP64)
lat.set_params(eos, -0.85, 0.3, rho_ref=0.2)
lat.init_density(np.full((1024, 1024), 0.2))
for call in (lambda: lat.measure(0, 512.0, 512.0, 100.0, 200.0), lat.stats, lambda: lat.read_fields(which=("rho",))):
    lat.step(10)
    call()
    lat.step(1500)
    w, c = time.perf_counter(), time.thread_time()
    call()
    w, c = time.perf_counter() - w, time.thread_time() - c
    print("%.4f %.4f" % (w, c))
    assert w > 0.1 and c < 0.3 * w, (w, c)
"""


def test_long_waits_leave_the_core_where_the_device_is_set_to_block(P):
    import os
    import subprocess
    import sys
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", BLOCKING], cwd=root, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
