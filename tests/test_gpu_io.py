"""GPU test of the mixed form's conversions at the boundary: populations are
rounded to FP32 (nearest even) on the way in and widened exactly on the way
out, over signs, ties, subnormals, overflow and NaN, as NumPy rounds them.
"""
import numpy as np
import pytest

from paper_1806_05089_gb300 import pond

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lattice", [pond.POND_D2Q16, pond.POND_D2Q9])
def test_mixed_populations_are_rounded_as_numpy_rounds(lattice):
    Q, ny, nx = (9 if lattice == pond.POND_D2Q9 else 16), 24, 40
    rng = np.random.default_rng(3)
    n = Q * ny * nx
    f = rng.standard_normal(n) * np.exp2(rng.integers(-160, 135, n))
    ties = (1.0 + (2.0 * rng.integers(0, 1 << 22, 500) + 1.0) * 2.0 ** -24) * np.exp2(rng.integers(-126, 127, 500))
    near = np.nextafter(ties, np.where(rng.random(500) < 0.5, 0.0, np.inf))
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 3.4028235677973366e38, 3.4028235e38,
                        1.1754943508222875e-38, 1.17549429e-38, 1.4e-45, 7e-46, 5e-324, 1.0, -1.0])
    f[:1000], f[1000:1000 + len(special)] = np.concatenate([ties, -near]), special
    f = f.reshape(Q, ny, nx)
    T = np.full((ny, nx), 1.0 / 3.0 if lattice == pond.POND_D2Q9 else 1.0)
    zero = np.zeros((ny, nx))
    with pond.Sim(nx, ny, pond.POND_FP32_MIXED, lattice=lattice) as s:
        s.set_state(None, zero, zero, T, f)
        got = s.state().f
    with np.errstate(over="ignore"):
        want = f.astype(np.float32).astype(np.float64)
    assert np.array_equal(got.view(np.int64), want.view(np.int64)) or (
        np.array_equal(np.isnan(got), np.isnan(want))
        and np.array_equal(got[~np.isnan(got)].view(np.int64), want[~np.isnan(want)].view(np.int64)))
