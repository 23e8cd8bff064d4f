"""Fields and statistics at the edges of their arguments: densities
beyond the law's pole, FP32 populations below the normal range, FP64 ones at
both ends of theirs, a density on the pole.

Tolerances.  psi^2 is a difference of terms of the size of the pressure; with
|1 - b rho| >= 0.09 and 2^-53 per operation over some 40 operations its
relative error is below 40 x 2^-53 x 3 / 0.09 = 1.5e-13: 1e-12 covers it, and
the velocity's share of it too.
"""
import numpy as np
import pytest

import oracle as O
from test_gpu_reductions import _fields, _law, _pressure

pytestmark = pytest.mark.gpu

BEYOND = {"cs": ((0.05, 0.42), (1.2, 1.6)), "vdw": ((0.5, 7.0), (11.6, 14.0)), "pr": ((0.5, 7.0), (11.6, 14.0))}


@pytest.fixture(scope="module")
def P():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1412_7228_gb300 as P
    P.lib()
    return P


def _across_the_pole(P, kind, prec, nx=45, ny=37):
    """A lattice whose nodes lie on both sides of the law's pole: without the
    interaction any positive density is a valid initial one."""
    eos, A = _law(P, kind)
    (a, b), (c, d) = BEYOND[kind]
    rng = np.random.default_rng(5)
    rho0 = np.where(rng.random((ny, nx)) < 0.5, rng.uniform(a, b, (ny, nx)), rng.uniform(c, d, (ny, nx)))
    lat = P.Lattice(nx, ny, prec)
    lat.set_params(eos, A, 0.2, G=0.0, s=[1.0] * 9, rho_ref=a)
    lat.init_density(rho0)
    lat.set_params(eos, A, 0.2, G=-1.0, s=[1.0] * 9, rho_ref=a)
    return lat, eos, A, rho0


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("kind", ["cs", "vdw", "pr"])
def test_psi_is_the_positive_root_on_both_sides_of_the_pole(P, kind, prec):
    lat, eos, A, _ = _across_the_pole(P, kind, prec)
    rho, ux, uy, psi = _fields(P, eos, A, lat.read_populations())
    assert (-2.0 * (_pressure(P, eos, rho) - rho / 3.0) > 0.0).all() and (rho * eos.b / (4.0 if kind == "cs" else 1.0) > 1.0).any()
    for which in (("psi",), ("rho", "ux", "uy", "psi")):
        got = lat.read_fields(which=which)
        assert (np.abs(got["psi"] - psi) <= 1e-12 * psi).all()
    assert np.abs(got["ux"] - ux).max() <= 1e-12 * np.abs(ux).max()
    assert np.abs(got["uy"] - uy).max() <= 1e-12 * np.abs(uy).max()
    st = lat.stats()
    assert abs(st["umax"] - np.sqrt((ux * ux + uy * uy).max())) <= 1e-12 * st["umax"]
    lat.close()


@pytest.mark.parametrize("kind", ["cs", "vdw", "pr"])
def test_an_fp64_step_across_the_pole_is_the_oracle_s(P, kind):
    lat, eos, A, rho0 = _across_the_pole(P, kind, P.LBM_FP64)
    law = {P.LBM_EOS_CS: O.EOS_CS, P.LBM_EOS_VDW: O.EOS_VDW, P.LBM_EOS_PR: O.EOS_PR}[eos.kind]
    op = O.Params(eos=law, a=eos.a, b=eos.b, R=eos.R, K=eos.K, T=eos.T, omega=eos.omega, Tc=eos.Tc, A=A, kappa=0.2,
                  G=-1.0, s=[1.0] * 9)
    f = O.init_equilibrium(rho0)
    O.step(op, f, 1)
    lat.step(1)
    assert np.abs(lat.read_populations() - f).max() <= 1e-12 * np.abs(f).max()
    lat.close()


def test_denormal_populations_are_read_as_they_are(P):
    """Multiples of 2^-149 below 2^-99: sums of a few are exact in FP64, and
    the velocity is one division of two of them (within 2 ulp)."""
    nx, ny = 67, 41
    rng = np.random.default_rng(11)
    eos, A = _law(P, "cs")
    lat = P.Lattice(nx, ny, P.LBM_FP32)
    lat.set_params(eos, A, 0.0, G=0.0, rho_ref=0.0)
    lat.init_density(10.0 ** rng.uniform(-42, -31, (ny, nx)), rng.uniform(-0.1, 0.1, (ny, nx)), rng.uniform(-0.1, 0.1, (ny, nx)))
    f = lat.read_populations()
    rho, jx, jy = f.sum(0), f[1] - f[3] + f[5] - f[6] - f[7] + f[8], f[2] - f[4] + f[5] + f[6] - f[7] - f[8]
    assert (np.abs(f) < 1e-38).any() and (rho > 0.0).all()
    got = lat.read_fields()
    assert np.array_equal(got["rho"], rho)
    assert np.array_equal(lat.read_fields(which=("rho",))["rho"], rho)
    assert (np.abs(got["ux"] - jx / rho) <= 2.0 ** -51 * np.abs(jx / rho)).all()
    assert (np.abs(got["uy"] - jy / rho) <= 2.0 ** -51 * np.abs(jy / rho)).all()
    lat.close()


@pytest.mark.parametrize("lo,hi", [(-309, -305), (-2, 2), (304, 307)])
def test_velocities_at_both_ends_of_the_fp64_range(P, lo, hi):
    """u is the quotient of the read populations' sums, within 2 ulp of the
    division (of denormal sums: of its own rounding), also where the
    reciprocal of the density is no normal number."""
    nx, ny = 43, 39
    rng = np.random.default_rng(17)
    eos, A = _law(P, "cs")
    lat = P.Lattice(nx, ny, P.LBM_FP64)
    lat.set_params(eos, A, 0.0, G=0.0, rho_ref=0.0)
    lat.init_density(10.0 ** rng.uniform(lo, hi, (ny, nx)), rng.uniform(-0.1, 0.1, (ny, nx)), rng.uniform(-0.1, 0.1, (ny, nx)))
    f = lat.read_populations()
    rho = sum(f[a] for a in range(9))
    jx, jy = f[1] - f[3] + f[5] - f[6] - f[7] + f[8], f[2] - f[4] + f[5] + f[6] - f[7] - f[8]
    got = lat.read_fields()
    assert np.array_equal(got["rho"], rho) and np.isfinite(rho).all()
    for k, j in (("ux", jx), ("uy", jy)):
        assert (np.abs(got[k] - j / rho) <= 2.0 ** -51 * np.abs(j / rho)).all(), k
    lat.close()


def test_pressure_of_a_density_on_the_pole(P):
    """Without the interaction any positive density is allowed: on the pole
    the law is infinite, and the sample says so."""
    eos, A = _law(P, "cs")
    lat = P.Lattice(40, 24, P.LBM_FP64)
    lat.set_params(eos, A, 0.0, G=0.0, rho_ref=1.0)       # 4 / b
    lat.init_density(np.ones((24, 40)))
    m = lat.measure(0, 20.0, 12.0, 5.0, 8.0)
    assert m["rho_in"] == 1.0 and m["p_in"] == np.inf and m["p_out"] == np.inf
    lat.close()
    import torch
    field = torch.ones((24, 40), dtype=torch.float64, device="cuda")
    field[12, 20] = 0.1                                   # p_in over the other nodes too
    m = P.lbm.lbm_field_pressure_jump_static(field.data_ptr(), 40, 24, eos, 20.0, 12.0, 5.0, 8.0)
    assert m["p_in"] == np.inf and m["p_out"] == np.inf
    field[:] = 0.1
    m = P.lbm.lbm_field_pressure_jump_static(field.data_ptr(), 40, 24, eos, 20.0, 12.0, 5.0, 8.0)
    assert abs(m["p_in"] - P.lbm_eos_pressure(eos, 0.1)) < 1e-15


@pytest.mark.parametrize("kind", ["cs", "vdw", "pr"])
def test_psi_is_accurate_to_a_few_ulp(P, kind):
    """psi from the folded reciprocal square root against the square root in
    extended precision, hot and repulsive (G = 1), where no terms cancel: W
    and D carry up to 14 roundings, of which the root halves the effect, and
    the fold 2.5 more, so 9.5 x 2^-53 < 1.1e-15; the constants' 4 make 1.4e-15."""
    eos, A = _law(P, kind)
    eos.T *= 40.0
    lat = P.Lattice(61, 47, P.LBM_FP64)
    lat.set_params(eos, A, 0.0, G=1.0, s=[1.0] * 9)
    rng = np.random.default_rng(23)
    top = 0.2 if kind == "cs" else 0.2 / eos.b
    lat.init_density(rng.uniform(1e-3 * top, top, (47, 61)))
    got = lat.read_fields()
    for field in (got["psi"], lat.read_fields(which=("psi",))["psi"]):
        r = got["rho"].astype(np.longdouble)
        want = np.sqrt(2 * (_pressure(P, eos, r) - r / 3))
        assert np.abs(field / want - 1).max() <= 1.4e-15
    lat.close()


def test_the_mirrors_hold_to_the_last_bit_in_fp64(P):
    """As in FP32: a centred drop stays symmetric under x -> -x and y -> -y."""
    import lbm_inputs as I
    eos, A = _law(P, "cs")
    rg, rl, _ = P.lbm_eos_maxwell(eos)
    n = 64
    mx, my, xs = [0, 3, 2, 1, 4, 6, 5, 8, 7], [0, 1, 4, 3, 2, 8, 7, 6, 5], (-np.arange(64)) % 64
    for sched in (0, 4):
        lat = P.Lattice(n, n, P.LBM_FP64)
        lat.set_params(eos, A, 0.3, rho_ref=rg)
        lat.set_schedule(0, sched)
        lat.init_density(I.droplet_density(n, n, 15, rl, rg))
        lat.step(1000)
        f = lat.read_populations()
        lat.close()
        for a in range(9):
            assert np.array_equal(f[a], f[mx[a]][:, xs]) and np.array_equal(f[a], f[my[a]][xs, :]), a
