"""The cluster schedule against the one-step kernels, bit for bit, at the
edges of its strips and vectors: lattices narrower than a vector, widths that
no vector divides, one-strip lattices, short last strips, the largest of each
configuration; every law, the viscosity law and G = 0; and its ghost cells,
by going on with the one-step kernels."""
import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu

SIZES = [(2, 2), (3, 3), (5, 6), (64, 64), (64, 5), (63, 62), (61, 10), (64, 7), (64, 100), (33, 127), (64, 256),
         (65, 20), (120, 120), (127, 126), (128, 128)]


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1412_7228_gb300 as P
    P.lib()
    return P


def _law(P, kind):
    from paper_1412_7228_gb300 import experiments as X
    if kind == "vdw":
        return X.vdw_eos(0.9, 0.3), -0.5
    if kind == "pr":
        return X.pr_eos(0.8, 0.5), -0.3
    eos = P.Eos(kind=P.LBM_EOS_CS, a=1.0, b=4.0, R=1.0, K=1.0)
    _, Tc, _ = P.lbm_eos_critical(eos)
    eos.T = 0.7 * Tc
    return eos, -0.85


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_cluster_steps_are_the_one_step_kernels_bits(P, nx, ny, prec):
    if prec == P.LBM_FP64 and (nx > 64 or ny > 128):
        pytest.skip("beyond the FP64 cluster's size")
    ran = 0
    for kind, visc, G in (("cs", False, -1.0), ("pr", True, -1.0), ("vdw", False, -1.0), ("cs", False, 0.0),
                          ("cs", True, 0.0)):
        eos, A = _law(P, kind)
        rg, rl, _ = P.lbm_eos_maxwell(eos)
        rho0 = I.droplet_density(nx, ny, 0.3 * min(nx, ny), rl, rg, width=4.0, cx=0.4 * nx, cy=0.55 * ny)
        got = []
        for plan in (((0, 14),), ((4, 1), (4, 2), (4, 7), (0, 4)), ((0, 3), (4, 6), (0, 1), (4, 4))):
            lat = P.Lattice(nx, ny, prec)
            lat.set_params(eos, A, 0.3, G=G, rho_ref=rg)
            if visc:
                lat.set_viscosity(0.2, 0.05, rg, rl)
            lat.init_density(rho0, 0.01 * np.ones((ny, nx)), -0.02 * np.ones((ny, nx)))
            for sched, n in plan:
                lat.set_schedule(0, sched)
                lat.step(n)
            lat.sync()
            got.append(lat.read_populations())
            ran += 1
            lat.close()
        assert np.array_equal(got[0], got[1]) and np.array_equal(got[0], got[2]), (kind, visc, G)
    assert ran == 15
