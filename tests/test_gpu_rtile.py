"""The register tiles of the FP32 inner sweep at the depths the plan picks by itself: k sweeps per
launch equal the oracle's one-sweep-at-a-time results bit for bit, at the edges of the tiles (96 to
124 stored columns per strip and 16 to 120 rows per block, whatever the depth), on grids smaller
than a tile's halo, and with a remainder shorter than the depth."""
import numpy as np
import pytest

from oracle import oracle as orc

pytestmark = pytest.mark.gpu


def _check(st, Nx, Ny, count, inner=64, **kw):
    import torch

    import paper_1705_00103_gb300 as cj
    rng = np.random.default_rng(5 * Nx + Ny + 7 * st)
    r = rng.standard_normal((Ny, Nx)).astype(np.float32)
    e = rng.standard_normal((Ny, Nx)).astype(np.float32)
    with cj.Plan(Nx, Ny, st, 1e-8, precision=cj.CJ_FP32_INNER, inner_cycle=inner, **kw) as p:
        kmin, kmax = orc.kappa_bounds(st, Nx, Ny)
        w32 = orc.sweep_coeffs(st, kmin, kmax, inner).astype(np.float32)
        ed = torch.from_numpy(e.copy()).cuda()
        cj.cj_sweeps_f32(p.handle, torch.from_numpy(r).cuda(), ed, 3, count)
    ref = e.copy()
    for k in range(count):
        ref = orc.sweep_f32(st, ref, r, w32[(3 + k) % inner])
    np.testing.assert_array_equal(ed.cpu().numpy(), ref)


@pytest.mark.parametrize("st", [5, 9, 17])
@pytest.mark.parametrize("Nx,Ny", [(1, 1), (3, 200), (200, 2), (96, 48), (97, 49), (104, 40), (113, 97), (120, 33),
                                   (225, 24), (384, 250), (641, 640)])
def test_default_depth_bit_exact(st, Nx, Ny):
    _check(st, Nx, Ny, 37)


@pytest.mark.parametrize("st,Nx,Ny", [(5, 1025, 1023), (9, 1500, 700), (9, 2049, 1601), (17, 1023, 1025),
                                      (17, 1501, 2047)])
def test_default_depth_large_tiles_bit_exact(st, Nx, Ny):
    """Sizes whose model picks the tall shapes (one, two and several blocks per SM)."""
    _check(st, Nx, Ny, 19)


@pytest.mark.parametrize("st", [9, 17])
@pytest.mark.parametrize("count", [0, 1, 2, 3, 15, 16, 17])
def test_counts_around_the_depth(st, count):
    _check(st, 150, 131, count, inner=16)
