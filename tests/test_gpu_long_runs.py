"""Many launches one after the other in one call, each beginning while the one before ends and reading
what it has just written, on grids that stay in the caches; the 17-point 8192^2 sweeps at their default
depth; and the batch engine's tall tiles (problems of more than 2^20 nodes), each against the oracle."""
import numpy as np
import pytest

from oracle import oracle as orc
import workloads

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def cj():
    import paper_1705_00103_gb300 as cj
    cj.build.build()
    return cj


@pytest.fixture(scope="module")
def torch():
    import torch
    return torch


@pytest.mark.parametrize("st", [5, 9, 17])
@pytest.mark.parametrize("Nx,Ny", [(200, 150), (333, 250), (1000, 700)])
@pytest.mark.parametrize("ff", [False, True])
def test_many_sweeps_in_one_call(cj, torch, st, Nx, Ny, ff):
    """Forty Jacobi sweeps (w = 1/c) of a rough iterate.  FP64: the oracle's bits.  Float-float: a sweep's
    error is at most 1e-12 (max|u| + w (9 max|u| + max|b|)), and a sweep multiplies an earlier one's by at
    most the sum of its neighbours' coefficients over c: 1 for 5 and 9 points, 340/300 for 17."""
    rng = np.random.default_rng(st + Nx)
    u, f = rng.standard_normal((Ny, Nx)), rng.standard_normal((Ny, Nx)) * Nx * Nx * 0.01
    c = orc.centre(st)
    grow = 340.0 / 300.0 if st == 17 else 1.0
    b, ref, tol = orc.scale_rhs(f), u, 0.0
    with cj.Plan(Nx, Ny, st, 1e-6, method=cj.CJ_JACOBI, launch=cj.CJ_LAUNCH_STREAM) as p:
        ud = torch.from_numpy(u.copy()).cuda()
        (cj.cj_sweeps_ff if ff else cj.cj_sweeps)(p.handle, torch.from_numpy(f).cuda(), ud, 0, 40)
        got = ud.cpu().numpy()
        w = float(p.info()["w"][0])
    for _ in range(40):
        m = np.abs(ref).max()
        tol = grow * tol + 1e-12 * (m + w * (9.0 * m + np.abs(b).max()))
        ref = orc.sweep(st, ref, b, w)
    assert abs(w * c - 1.0) < 1e-15
    if ff:
        assert np.abs(got - ref).max() <= tol
    else:
        np.testing.assert_array_equal(got, ref)


def test_17_point_8192_default_depth_bit_exact(cj, torch):
    N, st = 8192, 17
    rng = np.random.default_rng(31)
    r = rng.standard_normal((N, N)).astype(np.float32)
    e = rng.standard_normal((N, N)).astype(np.float32)
    with cj.Plan(N, N, st, 1e-10, precision=cj.CJ_FP32_INNER, inner_cycle=64) as p:
        kmin, kmax = orc.kappa_bounds(st, N, N)
        w32 = orc.sweep_coeffs(st, kmin, kmax, 64).astype(np.float32)
        ed = torch.from_numpy(e).cuda()
        cj.cj_sweeps_f32(p.handle, torch.from_numpy(r).cuda(), ed, 3, 9)
    for k in range(9):
        e = orc.sweep_f32(st, e, r, w32[(3 + k) % 64])
    np.testing.assert_array_equal(ed.cpu().numpy(), e)


@pytest.mark.parametrize("Nx,Ny,st,depth", [(1100, 1000, 5, 8), (2301, 2100, 9, 8), (1900, 1801, 17, 4),
                                            (1025, 1025, 17, 8), (1025, 1025, 9, 3)])
def test_tall_tiles_of_the_batch_engine_match_the_oracle(cj, torch, Nx, Ny, st, depth):
    """Two outer steps; the second and third have more tiles than the engine has blocks, so that blocks
    take a second one."""
    f = workloads.smooth_random_rhs(Nx, Ny, 7, kmax=40)
    pr = dict(Nx=Nx, Ny=Ny, st=st, tol=1e-12, precision=1, inner_cycle=32, max_sweeps=64, temporal_depth=depth,
              f=torch.from_numpy(f).cuda(), u=torch.zeros((Ny, Nx), dtype=torch.float64, device="cuda"))
    res = cj.cj_solve_batch([pr])
    ref = orc.solve_mixed(st, f, 1e-12, 32, max_outer=2)
    assert res[0]["sweeps"] == ref["sweeps"] == 64
    np.testing.assert_array_equal(pr["u"].cpu().numpy(), ref["u"])
