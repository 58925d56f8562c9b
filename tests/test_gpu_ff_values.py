"""Float-float sweeps of isolated nodes of widely different magnitudes: what the import's and the
export's conversions on the integer pipe make of each value (ties of its 24-bit rounding, carries,
zeros of both signs, values whose low part leaves the normal float range), node by node.

A node u alone among zeros becomes (1 - c w) u and its neighbours w a u (a their coefficients, c the
centre's): |got - ref| <= 2^-42 |u| (1 + |w| c), 32 times the few units of 2^-47 that one import, three
float-float operations and one export may take, and 2^-21 in place of 2^-42 below 2^-70, where low
parts are lost."""
import numpy as np
import pytest

from oracle import oracle as orc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("st", [5, 9, 17])
@pytest.mark.parametrize("Nx,Ny", [(60, 41), (61, 40)])
def test_isolated_nodes(st, Nx, Ny):
    import torch

    import paper_1705_00103_gb300 as cj
    u = np.zeros((Ny, Nx))
    rng = np.random.default_rng(st + Nx)
    ys, xs = np.meshgrid(np.arange(2, Ny - 2, 5), np.arange(2, Nx - 2, 5), indexing="ij")
    m = rng.choice([0, 1, 2 ** 28, 2 ** 28 - 1, 2 ** 28 + 1, 3 * 2 ** 28, 2 ** 52 - 1, 2 ** 52 - 2 ** 28], ys.shape)
    m = np.where(rng.random(ys.shape) < 0.5, m, rng.integers(0, 2 ** 52, ys.shape))
    e = rng.choice([0, 1, 60, 100, -40, -69, -73, -74, -80, -110], ys.shape)
    v = np.ldexp((2 ** 52 + m).astype(np.float64), e - 52) * rng.choice([-1.0, 1.0], ys.shape)
    u[ys, xs] = v
    u[0, :] = -0.0
    scale = np.zeros_like(u)  # |u| of the node that reaches each node
    for dy in range(-2, 3):
        for dx in range(-2, 3):
            scale[ys + dy, xs + dx] = np.abs(v)
    f = np.zeros_like(u)
    c = {5: 4.0, 9: 20.0 / 6.0, 17: 300.0 / 72.0}[st]
    with cj.Plan(Nx, Ny, st, 1e-6) as p:
        w = p.info()["w"]
        for k in (0, 1, len(w) - 1):
            ud = torch.from_numpy(u.copy()).cuda()
            cj.cj_sweeps_ff(p.handle, torch.from_numpy(f).cuda(), ud, k, 1)
            ref = orc.sweep(st, u, f, w[k])
            rel = np.where(scale < 2.0 ** -70, 2.0 ** -21, 2.0 ** -42)
            assert np.all(np.abs(ud.cpu().numpy() - ref) <= rel * scale * (1.0 + abs(w[k]) * c))


@pytest.mark.parametrize("st", [5, 9, 17])
@pytest.mark.parametrize("Nx,Ny", [(60, 41), (61, 40), (1, 1), (2, 3), (127, 130)])
def test_plan_after_float_float_sweeps(st, Nx, Ny):
    """FP64 calls of a plan give the oracle's bits after float-float sweeps have used its buffers in
    their own form (an odd number of sweeps and an even one)."""
    import torch

    import paper_1705_00103_gb300 as cj
    rng = np.random.default_rng(Nx + 10 * st)
    f, u = rng.standard_normal((Ny, Nx)), rng.standard_normal((Ny, Nx))
    b = orc.scale_rhs(f)
    fd = torch.from_numpy(f).cuda()
    with cj.Plan(Nx, Ny, st, 1e-6) as p:
        w = p.info()["w"]
        ref = u
        for k in range(3):
            ref = orc.sweep(st, ref, b, w[k % len(w)])
        for count in (1, 2):
            cj.cj_sweeps_ff(p.handle, fd, torch.from_numpy(u.copy()).cuda(), 0, count)
            ud = torch.from_numpy(u.copy()).cuda()
            cj.cj_sweeps(p.handle, fd, ud, 0, 3)
            np.testing.assert_array_equal(ud.cpu().numpy(), ref)
            cj.cj_sweeps_ff(p.handle, fd, torch.from_numpy(u.copy()).cuda(), 0, count)
            ud = torch.zeros((Ny, Nx), dtype=torch.float64, device="cuda")
            res = cj.cj_solve(p.handle, fd, ud)
            want = orc.solve(st, f, 1e-6)
            assert res["sweeps"] == want["sweeps"]
            np.testing.assert_array_equal(ud.cpu().numpy(), want["u"])
