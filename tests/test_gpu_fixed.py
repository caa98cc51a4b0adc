"""GPU tests of the fixed-point form of the FP64 staged step: the sizes at a
tile's edges, tiles inside and outside its range of magnitudes and gauge
spreads in one grid, and its scale.

Tolerances: 1e-12 with fixed passes against the oracle, as the other FP64
parity tests.  The step is homogeneous in the populations and every scale of
the kernel is a power of two, so populations scaled by one scale the result
exactly.
"""
import numpy as np
import pytest

import oracle
from paper_1806_05089_gb300 import pond, workloads

pytestmark = pytest.mark.gpu

TOL64 = 1e-12


def run(fields, steps, f=None, **cfg):
    ny, nx = fields.shape
    with pond.Sim(nx, ny, pond.POND_FP64, **cfg) as s:
        s.set_state(fields.rho, fields.ux, fields.uy, fields.T, f)
        stats = s.step(steps)
        return s.state(), stats


def against_oracle(fields, steps, lattice, **cfg):
    T_ref = 1.0 / 3.0 if lattice == pond.POND_D2Q9 else 1.0
    g, stats = run(fields, steps, fixed_iter=4, lattice=lattice, T_ref=T_ref, **cfg)
    o = oracle.init_equilibrium(fields.rho, fields.ux, fields.uy, fields.T, lattice=lattice)
    for _ in range(steps):
        o, _, fl = oracle.step(o, oracle.Params(fixed_iter=4, lattice=lattice, T_ref=T_ref))
        assert not fl.any()
    assert stats["nonphysical"] == 0 and stats["halo_fallback"] == 0
    speed = max(np.abs(o.ux).max(), np.abs(o.uy).max(), float(np.sqrt(o.T.mean())))
    assert np.abs(g.f - o.f).max() <= TOL64 * np.abs(o.f).max()
    assert np.max(np.abs(g.f.sum(0) - o.f.sum(0)) / o.f.sum(0)) <= TOL64
    assert max(np.abs(g.ux - o.ux).max(), np.abs(g.uy - o.uy).max()) <= TOL64 * speed
    assert np.max(np.abs(g.T - o.T) / o.T) <= TOL64


def field(name, nx, ny, T_L):
    f = workloads.supersonic(nx=nx, ny=ny)
    x, y = np.arange(nx)[None, :] / nx, np.arange(ny)[:, None] / ny
    if name == "density":  # a factor 400 in density: windows with and without a factor 64
        f.rho = np.exp(3.0 * np.sin(2 * np.pi * x)) * np.ones((ny, 1))
    if name == "shear":    # gauge spreads on both sides of the tile limit
        f.ux = f.ux + 0.5 * np.sin(2 * np.pi * y) ** 3 * np.ones((1, nx))
    c = np.sqrt(T_L)
    return workloads.Fields(f.rho, f.ux * c, f.uy * c, f.T * T_L)


@pytest.mark.parametrize("lattice", [pond.POND_D2Q16, pond.POND_D2Q9])
@pytest.mark.parametrize("tile_rows", [4, 8])
@pytest.mark.parametrize("name,nx,ny", [("plain", 31, 7), ("plain", 33, 9), ("plain", 64, 17),
                                        ("density", 160, 12), ("shear", 40, 64)])
def test_matches_oracle(name, nx, ny, tile_rows, lattice):
    T_L = 1.0 / 3.0 if lattice == pond.POND_D2Q9 else 1.0
    against_oracle(field(name, nx, ny, T_L), 2, lattice, tile_rows=tile_rows)


@pytest.mark.parametrize("power", [-700, -3, 5, 700])
def test_scaled_populations_scale_the_result_exactly(power):
    fields = field("plain", 45, 21, 1.0)
    rng = np.random.default_rng(1)
    f = oracle.init_equilibrium(fields.rho, fields.ux, fields.uy, fields.T).f
    f = f * (1.0 + 0.1 * rng.standard_normal(f.shape))
    a, _ = run(fields, 2, f=f)
    b, _ = run(fields, 2, f=np.ldexp(f, power))
    assert np.array_equal(np.ldexp(a.f, power), b.f)
    assert np.array_equal(a.ux, b.ux) and np.array_equal(a.T, b.T)
