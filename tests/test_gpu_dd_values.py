"""The double-FP64 defect and correction node by node on values at the edges of their arithmetic (ties
and carries, equal and widely spread exponents, signs that differ, zeros of both signs): two outer
steps with inner cycles of one FP64 sweep, whose u_hi and u_lo equal the oracle's bit for bit."""
import numpy as np
import pytest

from oracle import oracle as orc

pytestmark = pytest.mark.gpu


def _values(kind, shape, rng):
    one = (1.0 + rng.random(shape)) * rng.choice([-1.0, 1.0], shape)
    if kind == "near":
        return np.ldexp(np.abs(one), rng.integers(-1, 2, shape))
    if kind == "ties":  # few low bits set, or all high ones
        m = rng.choice([0, 1, 2, 3, 2 ** 51, 2 ** 52 - 1, 2 ** 52 - 2, 2 ** 9 + 1], shape)
        return np.sign(one) * np.ldexp((2 ** 52 + m).astype(np.float64), rng.integers(-55, -49, shape))
    if kind == "equal":  # equal leading words, other low words
        m = rng.integers(0, 2 ** 32, shape)
        return np.sign(one) * np.ldexp((2 ** 52 + m).astype(np.float64), rng.choice([-52, -50, -46], shape))
    if kind == "zeros":
        return one * rng.choice([0.0, -0.0, 1.0, 1.0], shape)
    return np.ldexp(one, rng.integers(-60, 61, shape))  # "wide"


@pytest.mark.parametrize("st", [5, 9, 17])
@pytest.mark.parametrize("kind", ["near", "ties", "equal", "zeros", "wide"])
@pytest.mark.parametrize("Nx,Ny", [(130, 41), (3, 2)])
def test_values_bit_exact(st, kind, Nx, Ny):
    import torch

    import paper_1705_00103_gb300 as cj
    rng = np.random.default_rng(Nx + st)
    u, f = _values(kind, (Ny, Nx), rng), _values(kind, (Ny, Nx), rng)
    ref = orc.solve_fp64_dd(st, f, 1e-14, 1, u0=u, max_outer=2)
    with cj.Plan(Nx, Ny, st, 1e-14, precision=cj.CJ_FP64_INNER_DD, inner_cycle=1, max_sweeps=2) as p:
        ud = torch.from_numpy(u.copy()).cuda()
        res = cj.cj_solve(p.handle, torch.from_numpy(f).cuda(), ud)
        lo = torch.empty_like(ud)
        cj.cj_solution_lo(p.handle, lo)
    assert res["sweeps"] == ref["sweeps"]
    np.testing.assert_array_equal(ud.cpu().numpy(), ref["u"])
    np.testing.assert_array_equal(lo.cpu().numpy(), ref["u_lo"])
