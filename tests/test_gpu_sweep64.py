"""FP64 sweeps with additions on the integer pipe: equal to the oracle bit for bit where every
addition takes that way, where none does, and at the ends of its conditions (exponents 9 to 11
apart, ties of the rounding, sums that carry, signs that differ, zeros, subnormals, the ends of the
exponent range, non-finite values), at the edges of a thread's rows and of the blocks."""
import numpy as np
import pytest

from oracle import oracle as orc

pytestmark = pytest.mark.gpu


def _values(kind, shape, rng):
    one = 1.0 + rng.random(shape)
    if kind == "near":  # one sign, exponents within 8
        return np.ldexp(one, rng.integers(-4, 5, shape))
    if kind == "edge":  # exponents 0 or 8..12 apart
        return np.ldexp(one, rng.choice([0, 8, 9, 10, 11, 12], shape))
    if kind == "ties":  # few low bits set, all high bits set, or neither: ties and carries of the rounding
        m = rng.choice([0, 1, 2, 3, 2 ** 51, 2 ** 52 - 1, 2 ** 52 - 2, 2 ** 52 - 2 ** 9, 2 ** 9 + 1], shape)
        return np.ldexp((2 ** 52 + m).astype(np.float64), rng.integers(-55, -44, shape))
    if kind == "signs":
        return one * rng.choice([-1.0, 1.0, 1.0, 1.0], shape)
    if kind == "zeros":
        return one * rng.choice([0.0, -0.0, 1.0, 1.0, 1.0, 1.0], shape)
    if kind == "tiny":  # around the lower end of the range and in the subnormals
        return np.ldexp(one, rng.integers(-1074, -980, shape))
    if kind == "huge":
        return np.ldexp(one, rng.integers(985, 1023, shape))
    v = one.copy()  # non-finite nodes here and there
    v[rng.random(shape) < 0.02] = np.inf
    v[rng.random(shape) < 0.02] = np.nan
    return v


def _check(st, Nx, Ny, kind, count=3):
    import torch

    import paper_1705_00103_gb300 as cj
    rng = np.random.default_rng(7 * Nx + Ny + st)
    u, f = _values(kind, (Ny, Nx), rng), _values(kind, (Ny, Nx), rng)
    with cj.Plan(Nx, Ny, st, 0.5 if max(Nx, Ny) > 1000 else 1e-6, launch=cj.CJ_LAUNCH_STREAM) as p:
        w = p.info()["w"]
        ud = torch.from_numpy(u.copy()).cuda()
        cj.cj_sweeps(p.handle, torch.from_numpy(f).cuda(), ud, 1, count)
    b, ref = orc.scale_rhs(f), u
    with np.errstate(all="ignore"):
        for k in range(count):
            ref = orc.sweep(st, ref, b, w[(1 + k) % len(w)])
    np.testing.assert_array_equal(ud.cpu().numpy(), ref)


@pytest.mark.parametrize("st", [5, 9, 17])
@pytest.mark.parametrize("kind", ["near", "edge", "ties", "signs", "zeros", "tiny", "huge", "nonfinite"])
def test_values_bit_exact(st, kind):
    _check(st, 131, 70, kind)


@pytest.mark.parametrize("st", [5, 9, 17])
@pytest.mark.parametrize("Nx,Ny", [(1, 1), (1, 9), (9, 1), (2, 3), (31, 5), (127, 3), (129, 2), (640, 487), (1600, 1750)])
def test_sizes_bit_exact(st, Nx, Ny):
    """Chunks of 1 to 5 rows, a shorter last chunk, warps that straddle two chunks, a part block."""
    _check(st, Nx, Ny, "near", count=2)
