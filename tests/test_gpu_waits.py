"""When results are waited for: a status is that of all the work issued so
far."""
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
