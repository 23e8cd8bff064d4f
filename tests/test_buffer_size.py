"""The memory a context asks for stays within what callers have reserved for
it, and that suffices for the smallest FP64 tiles' tables and step counters:
the interleaved and the multi-step schedules of a ragged batch give the
one-step launches' bits, also when a context changes between them."""
import numpy as np
import pytest

import lbm_inputs as I
import paper_1412_7228_gb300 as P


@pytest.mark.parametrize("nx,ny,prec,most", [(2, 2, 1, 28672), (2, 2, 2, 28672), (33, 16, 1, 103168),
                                             (64, 64, 1, 511232), (64, 64, 2, 824576),
                                             (3000, 3000, 2, 1517914624), (4096, 4096, 1, 1617191936),
                                             (4096, 4096, 2, 2826986496)])
def test_required_bytes_do_not_grow(nx, ny, prec, most):
    assert 0 < P.lbm_required_bytes(nx, ny, prec) <= most


def test_batch_required_bytes_do_not_grow():
    assert 0 < P.lbm_batch_required_bytes([128] * 6, [4] * 6, P.LBM_FP64) <= 977664


@pytest.mark.gpu
@pytest.mark.parametrize("prec", [1, 2])
def test_smallest_tiles_in_every_schedule(prec):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    cfgs = P.lbm_tile_configs(prec)
    tile = min(range(len(cfgs)), key=lambda k: (cfgs[k][3], cfgs[k][0] * cfgs[k][1]))
    sizes = [(17, 9), (2, 2), (64, 33), (16, 8), (130, 5)]
    eos = P.Eos(kind=P.LBM_EOS_CS, a=1.0, b=4.0, R=1.0, K=1.0)
    _, Tc, _ = P.lbm_eos_critical(eos)
    eos.T = 0.7 * Tc
    rg, rl, _ = P.lbm_eos_maxwell(eos)
    got = []
    for plan in ((0,), (1,), (3,), (1, 3, 1), (3, 1, 2, 3)):
        b = P.Batch([s[0] for s in sizes], [s[1] for s in sizes], prec)
        for i, (nx, ny) in enumerate(sizes):
            b.set_params(i, eos, -0.85, 0.3, rho_ref=rg)
            b.init_density(i, I.droplet_density(nx, ny, 0.3 * min(nx, ny), rl, rg, width=3.0))
        for sched in plan:
            b.set_schedule(tile, sched)
            b.step(12 // len(plan))
        b.sync()
        got.append([b.read_populations(i) for i in range(len(sizes))])
        b.close()
    for other in got[1:]:
        assert all(np.array_equal(x, y) for x, y in zip(got[0], other))
