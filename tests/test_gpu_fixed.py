"""GPU tests of the forms of the staged step: the fixed-point form of FP64 at
the sizes of a tile's edges, with tiles inside and outside its range of
magnitudes and gauge spreads in one grid, and its scale; the mixed form with
one, two and four lanes per node.

Tolerances: 1e-12 with fixed passes against the oracle, as the other FP64
parity tests.  The step is homogeneous in the populations and every scale of
the kernel is a power of two, so populations scaled by one scale the result
exactly.
"""
import numpy as np
import pytest

import oracle
from paper_1806_05089_gb300 import decomp, pond, workloads

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
    if name == "spots":    # parts of tiles out of range by gauge, and by a dense source
        x, y = np.arange(nx)[None, :], np.arange(ny)[:, None]
        f.ux = f.ux + 0.7 * np.exp(-((x - nx // 3) ** 2 + (y - ny // 2) ** 2) / 8.0)
        f.rho = f.rho * (1.0 + 60.0 * np.exp(-((x - nx // 2) ** 2 + (y - ny // 3) ** 2) / 8.0))
    if name == "vortex":   # nodes that leave the range in a pass
        f = workloads.vortex(nx, 0.1 * nx, 0.5, 1.0)
    c = np.sqrt(T_L)
    return workloads.Fields(f.rho, f.ux * c, f.uy * c, f.T * T_L)


@pytest.mark.parametrize("lattice", [pond.POND_D2Q16, pond.POND_D2Q9])
@pytest.mark.parametrize("tile_rows", [4, 8])
@pytest.mark.parametrize("name,nx,ny", [("plain", 31, 7), ("plain", 33, 9), ("plain", 64, 17),
                                        ("density", 160, 12), ("shear", 40, 64),
                                        ("spots", 100, 30), ("vortex", 44, 44)])
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


@pytest.mark.parametrize("lattice,tile_rows,nx,ny,px,py", [
    (pond.POND_D2Q16, 8, 512, 160, 2, 2),   # 320 whole tiles against 80 by parts of 8
    (pond.POND_D2Q16, 8, 256, 176, 1, 2),   # 176 half tiles against 88 by parts
    (pond.POND_D2Q16, 4, 256, 128, 2, 2),   # 256 against 64, four rows
    (pond.POND_D2Q9, 8, 512, 160, 2, 2), (pond.POND_D2Q9, 4, 256, 128, 2, 2)])
@pytest.mark.parametrize("name", ["plain", "spots"])
def test_parts_of_tiles_match_whole_tiles_bit_for_bit(name, lattice, tile_rows, nx, ny, px, py):
    T_L = 1.0 / 3.0 if lattice == pond.POND_D2Q9 else 1.0
    fields = field(name, nx, ny, T_L)
    cfg = dict(lattice=lattice, T_ref=T_L)
    whole, _ = run(fields, 2, tile_rows=tile_rows, **cfg)
    with decomp.DecomposedSim(nx, ny, px, py, 14, precision=pond.POND_FP64, tile_rows=tile_rows,
                              **cfg) as d:
        d.set_state(fields.rho, fields.ux, fields.uy, fields.T)
        d.step(2)
        f, g = d.gather_state()
    assert np.array_equal(whole.f, f)
    for a, b in zip((whole.ux, whole.uy, whole.T), g):
        assert np.array_equal(a, b)


def test_a_window_too_large_for_whole_tiles_runs_by_halves():
    """T = 6: the staged window of a 32 x 8 tile exceeds the shared memory."""
    fields = field("plain", 640, 200, 1.0)
    fields.T = 6.0 * fields.T
    a, _ = run(fields, 1, fixed_iter=4)
    b, _ = run(fields, 1, fixed_iter=4, kernel=pond.POND_KERNEL_DIRECT)
    assert np.abs(a.f - b.f).max() <= TOL64 * np.abs(b.f).max()
    assert np.abs(a.ux - b.ux).max() <= TOL64 * np.sqrt(6.0)
    assert np.max(np.abs(a.T - b.T) / b.T) <= TOL64


@pytest.mark.parametrize("lattice", [pond.POND_D2Q16, pond.POND_D2Q9])
@pytest.mark.parametrize("name,nx,ny", [("plain", 1, 1), ("plain", 37, 1), ("plain", 1, 70),
                                        ("plain", 500, 90), ("density", 160, 12), ("shear", 300, 96)])
def test_allocation_free_step_matches_the_context_step(name, nx, ny, lattice):
    """Windows sized by capacity against windows sized by the velocities: the
    same staged values and sums, so bit for bit."""
    import torch
    T_L = 1.0 / 3.0 if lattice == pond.POND_D2Q9 else 1.0
    fields = field(name, nx, ny, T_L)
    cfg = pond.pond_config_default(pond.POND_FP64)
    cfg.lattice, cfg.T_ref = lattice, T_L
    with pond.Sim(nx, ny, pond.POND_FP64, lattice=lattice, T_ref=T_L) as s:
        s.set_state(fields.rho, fields.ux, fields.uy, fields.T)
        start = s.state()
        s.set_state(None, start.ux, start.uy, start.T, start.f)
        s.step(1)
        want = s.state()
    cur = [torch.tensor(a, device="cuda") for a in (start.f, start.ux, start.uy, start.T)]
    out = [torch.empty_like(a) for a in cur]
    stats = pond.pond_step_fp64_noalloc(cfg, *cur, *out)
    assert stats["nonphysical"] == 0 and stats["halo_fallback"] == 0
    for a, b in zip(out, (want.f, want.ux, want.uy, want.T)):
        assert np.array_equal(a.cpu().numpy(), b)


@pytest.mark.parametrize("lattice", [pond.POND_D2Q16, pond.POND_D2Q9])
@pytest.mark.parametrize("name,nx,ny,hot", [("plain", 33, 9, 1.0), ("plain", 70, 30, 3.0),
                                            ("plain", 70, 30, 6.0), ("density", 160, 12, 1.0),
                                            ("shear", 40, 64, 1.0)])
def test_adjoint_step_matches_the_direct_kernels(name, nx, ny, hot, lattice):
    """Tiles in and out of the fixed-point tangents' range (gauge spread,
    magnitudes, tau > 1.9 at T = 6), the 32 x 4 tiles of wide windows, against
    the per-pair kernels; 1e-9 of the largest, as the adjoint's other checks."""
    import torch
    T_L = 1.0 / 3.0 if lattice == pond.POND_D2Q9 else 1.0
    fields = field(name, nx, ny, T_L)
    Q = 9 if lattice == pond.POND_D2Q9 else 16
    rng = np.random.default_rng(5)
    fbar = torch.tensor(rng.standard_normal((Q, ny, nx)), device="cuda")
    gbar = torch.tensor(rng.standard_normal((3, ny, nx)), device="cuda")
    got = []
    for kernel in (pond.POND_KERNEL_STAGED, pond.POND_KERNEL_DIRECT):
        with pond.Sim(nx, ny, pond.POND_FP64, lattice=lattice, T_ref=T_L, kernel=kernel) as s:
            s.set_state(fields.rho, fields.ux, fields.uy, hot * fields.T)
            out = torch.empty_like(fbar), torch.empty_like(gbar)
            nu = pond.pond_adjoint_step(s.ctx, fbar, gbar, *out)
            got.append([a.cpu().numpy() for a in out] + [np.array(nu)])
    for a, b in zip(*got):
        assert np.abs(a - b).max() <= 1e-9 * np.abs(b).max()


@pytest.mark.parametrize("lattice", [pond.POND_D2Q16, pond.POND_D2Q9])
@pytest.mark.parametrize("tile_rows,nx,ny", [(8, 31, 7), (8, 70, 45), (8, 161, 100), (4, 97, 65), (16, 130, 90)])
def test_mixed_lanes_change_no_bit(tile_rows, nx, ny, lattice):
    """A small grid by itself runs with two or four lanes per node; as the first
    grid of a batch that fills the chip it runs with one."""
    T_L = 1.0 / 3.0 if lattice == pond.POND_D2Q9 else 1.0
    small, large = field("shear", nx, ny, T_L), field("plain", 512, 512, T_L)
    out = []
    for grids in ([small], [small, large]):
        with pond.Sim([g.shape[1] for g in grids], [g.shape[0] for g in grids], pond.POND_FP32_MIXED,
                      lattice=lattice, T_ref=T_L, tile_rows=tile_rows) as s:
            for i, g in enumerate(grids):
                s.set_state(g.rho, g.ux, g.uy, g.T, grid=i)
            assert s.step(3)["halo_fallback"] == 0
            out.append(s.state())
    a, b = out
    for name in ("f", "ux", "uy", "T"):
        assert np.array_equal(getattr(a, name), getattr(b, name)), name
