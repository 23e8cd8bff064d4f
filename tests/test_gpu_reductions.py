"""The one-launch FP64 reductions and the fused field read-back against plain
numpy on the same populations, at the edges of their tiles: lattices smaller
than a tile, one node wider, ragged, and larger than the resident grid.

Tolerances.  Both sides evaluate the same FP64 expressions in another order
from the same populations: density and momentum within 2^-53 x 20 of the
largest population sum, the pressure and the psi radicand within 2^-53 x 40
of rho / 3 (they are differences of terms of that size), hence psi within
that over psi (>= 0.07 here) and the velocity within the force's share of it
over the gas density (>= 0.009): 1e-12 covers each.  Sums: 1e-12 of the sum of
magnitudes.  Node counts are equal.
"""
import numpy as np
import pytest

import lbm_inputs as I

pytestmark = pytest.mark.gpu

EX = np.array([0, 1, 0, -1, 0, 1, -1, -1, 1])
EY = np.array([0, 0, 1, 0, -1, 1, 1, -1, -1])
SIZES = [(2, 2), (3, 40), (32, 16), (33, 17), (64, 64), (65, 5), (130, 300), (1031, 1029), (2049, 1100)]


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


def _pressure(P, e, r):
    if e.kind == P.LBM_EOS_CS:
        n = e.b * r / 4.0
        return e.K * (r * e.R * e.T * (1 + n + n * n - n ** 3) / (1 - n) ** 3 - e.a * r * r)
    if e.kind == P.LBM_EOS_VDW:
        return e.K * (r * e.R * e.T / (1 - e.b * r) - e.a * r * r)
    m = 0.37464 + 1.54226 * e.omega - 0.26992 * e.omega ** 2
    al = (1 + m * (1 - np.sqrt(e.T / e.Tc))) ** 2
    return e.K * (r * e.R * e.T / (1 - e.b * r) - e.a * al * r * r / (1 + 2 * e.b * r - (e.b * r) ** 2))


def _fields(P, eos, A, f):
    rho = f.sum(0)
    psi = np.sqrt(2.0 / -1.0 * (_pressure(P, eos, rho) - rho / 3.0))
    g = np.zeros((4,) + rho.shape)
    for a in range(1, 9):
        w = 1.0 / 3.0 if a < 5 else 1.0 / 12.0
        n = np.roll(psi, (-EY[a], -EX[a]), (0, 1))
        for k, v in enumerate((EX[a] * n, EY[a] * n, EX[a] * n * n, EY[a] * n * n)):
            g[k] += w * v
    F = [0.5 * A * g[2 + k] + (1 - A) * psi * g[k] for k in (0, 1)]   # G = -1
    j = [np.tensordot(e, f, 1) for e in (EX.astype(float), EY.astype(float))]
    return rho, (j[0] + 0.5 * F[0]) / rho, (j[1] + 0.5 * F[1]) / rho, psi


def _lattice(P, nx, ny, prec, kind):
    eos, A = _law(P, kind)
    rg, rl, _ = P.lbm_eos_maxwell(eos)
    lat = P.Lattice(nx, ny, prec)
    lat.set_params(eos, A, 0.2, s=[1.0] * 9, rho_ref=rg)
    y, x = np.mgrid[0:ny, 0:nx]
    rho0 = I.droplet_density(nx, ny, 0.3 * min(nx, ny), rl, rg, width=4.0)
    lat.init_density(rho0, 0.02 + 0.01 * np.sin(2 * np.pi * y / ny), 0.01 * np.cos(2 * np.pi * x / nx))
    lat.step(1)
    return lat, eos, A


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("nx,ny", SIZES)
def test_fields_and_sums(P, nx, ny, prec):
    kind = ("cs", "vdw", "pr")[(nx + ny) % 3]
    lat, eos, A = _lattice(P, nx, ny, prec, kind)
    rho, ux, uy, psi = _fields(P, eos, A, lat.read_populations())
    scale = {"rho": rho.max(), "ux": 1.0, "uy": 1.0, "psi": psi.max()}
    want = dict(rho=rho, ux=ux, uy=uy, psi=psi)
    whole = lat.read_fields()
    for k in want:
        assert np.abs(whole[k] - want[k]).max() <= 1e-12 * scale[k], k
    # every choice of fields, in either type, gives the same values
    for which in (("rho",), ("psi",), ("ux",), ("uy", "rho"), ("ux", "uy", "psi"), ("rho", "psi")):
        got = lat.read_fields(which=which)
        got32 = lat.read_fields(which=which, dtype=np.float32)
        for k in which:
            np.testing.assert_array_equal(got[k], whole[k])
            np.testing.assert_array_equal(got32[k], whole[k].astype(np.float32))
    st = lat.stats()
    u2 = ux * ux + uy * uy
    for k, v in dict(mass=rho, mom_x=rho * ux, mom_y=rho * uy, ke=0.5 * rho * u2).items():
        assert abs(st[k] - v.sum()) <= 1e-12 * np.abs(v).sum(), k
    assert abs(st["umax"] - np.sqrt(u2.max())) <= 1e-12
    p = _pressure(P, eos, rho)
    for cx, cy, ri, ro in ((nx / 2, ny / 2, 0.2 * min(nx, ny), 0.3 * min(nx, ny) + 1), (0.0, 1.0, 5.0, 5.0),
                           (nx - 0.25, ny + 3.0, 0.0, 0.0), (1.5, 0.5, 13.0, 2.5)):
        dx, dy = np.arange(nx)[None, :] - cx, np.arange(ny)[:, None] - cy
        dx, dy = dx - nx * np.round(dx / nx), dy - ny * np.round(dy / ny)
        d = np.sqrt(dx * dx + dy * dy)
        i, o = d <= ri, d >= ro
        m = lat.measure(0, cx, cy, ri, ro)
        assert (m["n_in"], m["n_out"]) == (i.sum(), o.sum())
        assert abs(m["mass"] - rho.sum()) <= 1e-12 * rho.sum()
        for k, v, s in (("rho_in", rho, i), ("p_in", p, i), ("rho_out", rho, o), ("p_out", p, o)):
            if s.any():
                assert abs(m[k] - v[s].mean()) <= 1e-12 * rho.max(), k
            else:
                assert np.isnan(m[k])
    for c in (float("nan"), float("inf")):
        m = lat.measure(0, c, 1.0, 1.0, 1.0)
        assert (m["n_in"], m["n_out"]) == (0, 0)
    lat.close()


@pytest.mark.parametrize("nx,ny", [(1, 1), (3, 4), (64, 4), (65, 33), (500, 4097), (4096, 4096)])
def test_field_sums_of_a_device_field(P, nx, ny):
    import torch
    from paper_1412_7228_gb300 import lbm as L
    eos, _ = _law(P, "cs")
    rng = np.random.default_rng(nx * 10007 + ny)
    rho = rng.uniform(0.01, 0.36, (ny, nx))
    dev = torch.from_numpy(rho).cuda()
    p = _pressure(P, eos, rho)
    for cx, cy, ri, ro in ((nx / 2, ny / 2, 5.0, 5.0), (0.25, 3.0, 0.3 * nx, 0.2 * ny)):
        dx, dy = np.arange(nx)[None, :] - cx, np.arange(ny)[:, None] - cy
        dx, dy = dx - nx * np.round(dx / nx), dy - ny * np.round(dy / ny)
        d = np.sqrt(dx * dx + dy * dy)
        i, o = d <= ri, d >= ro
        for _ in range(2):
            m = L.lbm_field_pressure_jump_static(dev.data_ptr(), nx, ny, eos, cx, cy, ri, ro,
                                                 stream_ptr=torch.cuda.current_stream().cuda_stream)
            assert (m["n_in"], m["n_out"]) == (i.sum(), o.sum())
            assert abs(m["mass"] - rho.sum()) <= 1e-12 * rho.sum()
            for k, v, s in (("rho_in", rho, i), ("p_in", p, i), ("rho_out", rho, o), ("p_out", p, o)):
                if s.any():
                    assert abs(m[k] - v[s].mean()) <= 1e-12, k


@pytest.mark.parametrize("nx,ny", [(5, 3), (181, 180), (700, 150), (2900, 3000)])
def test_reads_into_every_kind_of_memory(P, nx, ny):
    """Pinned arrays are written by the kernels, small pageable ones come
    through the context's stage, larger ones and those read in bands by
    copies: the same values in each, and nothing beside them."""
    import torch
    lat, _, _ = _lattice(P, nx, ny, P.LBM_FP32, "cs")
    for dtype in (np.float32, np.float64):
        tdt = torch.float32 if dtype == np.float32 else torch.float64
        want = lat.read_fields(dtype=dtype)
        pinned = torch.full((6 * nx * ny + 6,), -7.0, dtype=tdt).pin_memory().numpy()
        plain = np.full(6 * nx * ny + 6, -7.0, dtype=dtype)
        for mem in (pinned, plain):
            out = {k: mem[1 + j * (nx * ny + 1):1 + j * (nx * ny + 1) + nx * ny].reshape(ny, nx)
                   for j, k in enumerate(("rho", "ux", "uy", "psi"))}
            for which in (("rho",), ("rho", "psi"), ("rho", "ux", "uy", "psi")):
                mem[:] = -7.0
                got = lat.read_fields(which=which, out=out, dtype=dtype)
                for k in which:
                    assert np.array_equal(got[k], want[k]), k
                assert (mem == -7.0).sum() == mem.size - len(which) * nx * ny
        mixed = {"rho": pinned[:nx * ny].reshape(ny, nx), "ux": np.empty((ny, nx), dtype=dtype)}
        got = lat.read_fields(which=("rho", "ux"), out=mixed, dtype=dtype)
        assert np.array_equal(got["rho"], want["rho"]) and np.array_equal(got["ux"], want["ux"])
    lat.close()


@pytest.mark.parametrize("nx,ny", [(30, 20), (1100, 1000)])
def test_a_refused_field_leaves_one_lattice_as_it_was(P, nx, ny):
    """The equilibrium of a context of one lattice is written beside its
    current state before the check is known."""
    lat, eos, A = _lattice(P, nx, ny, P.LBM_FP32, "cs")
    lat.step(2)
    before = lat.read_populations()
    bad = np.full((ny, nx), 0.2)
    bad[ny - 1, nx - 1] = -1.0
    for args in ((bad,), (np.full((ny, nx), 0.2), np.full((ny, nx), np.inf), np.zeros((ny, nx)))):
        with pytest.raises(P.LbmError) as ei:
            lat.init_density(*args)
        assert ei.value.code == P.lbm.LBM_EINVAL
        assert np.array_equal(lat.read_populations(), before) and lat.status(0) == 0
    lat.step(3)
    after = lat.read_populations()
    fresh, _, _ = _lattice(P, nx, ny, P.LBM_FP32, "cs")
    fresh.step(5)
    assert np.array_equal(fresh.read_populations(), after)
    lat.close()
    fresh.close()
