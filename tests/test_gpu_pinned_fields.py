"""Initial fields and read-backs in pinned memory, which the kernels reach
where it lies, against the same calls on pageable arrays: equal bits, in one
pass and in row bands, with and without a velocity, with fields of both kinds
in one call, and a refused field leaves the state as it was."""
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


def _pin(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).pin_memory().numpy()


def _lattice(P, nx, ny, prec):
    eos, A = _law(P, "cs")
    lat = P.Lattice(nx, ny, prec)
    lat.set_params(eos, A, 0.3, rho_ref=0.2)
    return lat


def _inputs(nx, ny, dtype):
    rng = np.random.default_rng(nx + ny)
    return (rng.uniform(0.1, 0.3, (ny, nx)).astype(dtype), rng.uniform(-0.05, 0.05, (ny, nx)).astype(dtype),
            rng.uniform(-0.05, 0.05, (ny, nx)).astype(dtype))


@pytest.mark.parametrize("prec", [1, 2])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("nx,ny", [(2, 3), (65, 33), (1100, 1000)])
def test_pinned_initial_fields_give_the_bits_of_pageable_ones(P, nx, ny, dtype, prec):
    rho, ux, uy = _inputs(nx, ny, dtype)
    pr, pu, pv = _pin(rho), _pin(ux), _pin(uy)
    lat = _lattice(P, nx, ny, prec)
    for args, pinned in (((rho,), ((pr,),)),
                         ((rho, ux, uy), ((pr, pu, pv), (pr, ux, uy), (rho, pu, pv), (pr, pu, uy))),
                         ((rho, None, uy), ((pr, None, pv), (pr, None, uy)))):
        lat.init_density(*args)
        want = lat.read_populations()
        lat.step(2)
        later = lat.read_populations()
        for p in pinned:
            lat.init_density(np.full((ny, nx), 0.25))
            lat.init_density(*p)
            assert np.array_equal(lat.read_populations(), want)
            lat.step(2)
            assert np.array_equal(lat.read_populations(), later)
    lat.close()


@pytest.mark.parametrize("nx,ny", [(30, 20), (1100, 1000)])
def test_a_refused_pinned_field_leaves_the_lattice_as_it_was(P, nx, ny):
    rho, ux, uy = _inputs(nx, ny, np.float32)
    lat = _lattice(P, nx, ny, P.LBM_FP32)
    lat.init_density(rho, ux, uy)
    lat.step(3)
    before = lat.read_populations()
    bad, wild = rho.copy(), ux.copy()
    bad[ny - 1, nx - 1] = -1.0
    wild[0, nx - 1] = np.nan
    for args in ((bad,), (bad, ux, uy), (rho, wild, uy)):
        with pytest.raises(P.LbmError) as ei:
            lat.init_density(*[_pin(a) for a in args])
        assert ei.value.code == P.lbm.LBM_EINVAL
        assert np.array_equal(lat.read_populations(), before) and lat.status(0) == 0 and lat.steps_done == 3
    lat.close()


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("nx,ny", [(5, 3), (181, 180), (1100, 1000)])
def test_pinned_arrays_at_any_address(P, nx, ny, dtype):
    """A view of pinned bytes behind a header need not be aligned: such arrays
    go through the copies, read and written."""
    import torch
    lat = _lattice(P, nx, ny, P.LBM_FP32)
    rho, ux, uy = _inputs(nx, ny, dtype)
    lat.init_density(rho, ux, uy)
    want, state = lat.read_fields(dtype=dtype), lat.read_populations()
    size = rho.nbytes
    raw = torch.zeros(4 * (size + 3) + 8, dtype=torch.uint8).pin_memory().numpy()
    views = [raw[k * (size + 3) + 1:k * (size + 3) + 1 + size].view(dtype).reshape(ny, nx) for k in range(4)]
    assert not any(v.ctypes.data % rho.itemsize == 0 for v in views[:1] + views[2:3])
    out = dict(zip(("rho", "ux", "uy", "psi"), views))
    for which in (("rho",), ("rho", "psi"), ("rho", "ux", "uy", "psi")):
        raw[:] = 0
        got = lat.read_fields(which=which, out=out, dtype=dtype)
        for k in which:
            assert got[k] is out[k] and np.array_equal(got[k], want[k]), k
    for v, a in zip(views, (rho, ux, uy)):
        v[...] = a
    lat.init_density(np.full((ny, nx), 0.25))
    lat.init_density(*views[:3])
    assert np.array_equal(lat.read_populations(), state)
    lat.close()


def test_small_reads_of_many_lattices_in_threads(P):
    """Small pageable fields come through a stage from a slab of blocks: more
    lattices than a slab has, read by several threads."""
    import threading
    lats, wants = [], []
    for k in range(18):
        nx, ny = 20 + 3 * k, 40
        lat = _lattice(P, nx, ny, P.LBM_FP32 if k % 2 else P.LBM_FP64)
        lat.init_density(*_inputs(nx, ny, np.float64))
        lat.step(3)
        lats.append(lat)
        wants.append((lat.read_fields(which=("rho", "psi")), lat.measure(0, 10.0, 20.0, 4.0, 9.0)))
    wrong = []

    def work(mine):
        for _ in range(40):
            for k in mine:
                got, m = lats[k].read_fields(which=("rho", "psi")), lats[k].measure(0, 10.0, 20.0, 4.0, 9.0)
                same = [a == b or (np.isnan(a) and np.isnan(b)) for a, b in ((m[f], wants[k][1][f]) for f in m)]   # R_eq may be none
                if not (all(np.array_equal(got[f], wants[k][0][f]) for f in got) and all(same)):
                    wrong.append(k)

    threads = [threading.Thread(target=work, args=(range(t, 18, 6),)) for t in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not wrong
    for lat in lats:
        lat.close()
