"""GPU tests of the FP32 step's default strip height and of gauge groups.

The default height depends on the grid size (4 rows on small grids, up to 36
on large ones, with a ragged last band); the results must not.  Gauges of a
recorded step are sampled 32 at a time by the warps that run out of strips;
they must equal swa_gauge_sample's values.  Both are exact.
"""
import numpy as np
import pytest

from paper_1605_05320_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def S():
    from paper_1605_05320_gb300 import build
    build.build()
    from paper_1605_05320_gb300 import swadj
    swadj.load()
    assert torch.cuda.is_available()
    return swadj


def grid(S, sc, **kw):
    d = S.make_desc(2, sc.grid.nx, sc.grid.ny, 0.0, 0.0, sc.grid.dx, sc.grid.dy,
                    precision=S.SWA_FP32, **kw)
    g = S.Grid(d, sc.B)
    g.set_state(sc.eta0, sc.hu0, sc.hv0, 0.0)
    return g


@pytest.mark.parametrize("nx,ny", [(2, 2), (3, 9), (28, 4), (57, 5), (2, 1500), (1500, 3),
                                   (130, 90), (700, 701), (1025, 700)])
@pytest.mark.parametrize("order,bc", [(2, (0, 0, 0, 0)), (1, (1, 1, 1, 1))])
def test_default_height_equals_a_fixed_one(S, nx, ny, order, bc):
    sc = synth.small_2d(nx, ny, seed=nx + ny, L=nx * 5e3)
    a, b = grid(S, sc, order=order, bc=bc), grid(S, sc, order=order, bc=bc)
    S.swa_grid_set_strip_rows(b.h, 64)
    a.step(12, 1e300)
    b.step(12, 1e300)
    assert a.time() == b.time()
    x, y = a.get_state(), b.get_state()
    for k in x:
        assert np.array_equal(x[k], y[k]), k
    assert S.swa_sync_status() == 0


@pytest.mark.parametrize("n", [1, 32, 33, 70])
def test_gauge_groups_equal_samples(S, n):
    sc = synth.small_2d(90, 64, seed=31)
    xy = torch.tensor(np.random.default_rng(n).uniform(-2e4, 1.02e6, (n, 2)),
                      dtype=torch.float64, device="cuda")
    g1, g2 = grid(S, sc), grid(S, sc)
    steps, cap = 9, 7
    ref = torch.zeros((steps, n), dtype=torch.float64, device="cuda")
    tref = []
    for k in range(steps):
        S.swa_gauge_sample(g1.h, n, xy, ref[k])
        tref.append(g1.time()[0])
        g1.step(1, 1e300)
    series = torch.full((cap, n), -7.0, dtype=torch.float64, device="cuda")
    times = torch.zeros(cap, dtype=torch.float64, device="cuda")
    S.swa_grid_record_gauges(g2.h, n, xy, series, times, cap)
    g2.step(steps, 1e300)
    assert S.swa_grid_gauge_rows(g2.h) == steps
    assert torch.equal(series, ref[:cap])
    assert np.array_equal(times.cpu().numpy(), np.array(tref[:cap]))


@pytest.mark.parametrize("count,side", [(1, 2), (3, 37), (40, 33), (30, 260)])
@pytest.mark.parametrize("order", [1, 2])
def test_default_patch_strips_equal_fixed_ones(S, count, side, order):
    """A level's default strips (4 to 36 rows, bands of equal height, taken
    from a counter) give the bits of the 16- and 32-row ones."""
    rng = np.random.default_rng(count)
    pats, fields = [], []
    for k in range(count):
        nx, ny = (2, 2) if side == 2 else (int(rng.integers(2, side)), int(rng.integers(2, side)))
        pats.append((1, 0.0, 0.0, nx, ny, 1e3, 1e3))
        n = nx * ny
        B = -rng.uniform(50.0, 4000.0) * np.ones(n)
        eta = rng.uniform(-1, 1, n) if k % 3 else np.zeros(n)
        hu = rng.uniform(-5, 5, n) if k % 3 else np.zeros(n)
        fields.append((B, eta, hu, -hu))
    common = S.make_desc(2, 2, 2, 0.0, 0.0, 1e3, 1e3, precision=S.SWA_FP32, order=order)
    ref = None
    for rows in (0, 16, 32):
        ps = S.PatchSet(pats, [f[0] for f in fields], common)
        for k, f in enumerate(fields):
            ps.set_state(k, *f[1:])
        S.swa_patches_set_tile_rows(ps.h, 1, rows)
        ps.start(1, 0.0)
        ps.step(1, 9)
        got = [ps.get_state(k) for k in range(count)]
        t = ps.time(1)
        if ref is None:
            ref, t_ref = got, t
        assert t == t_ref
        for a, b in zip(ref, got):
            for key in a:
                assert np.array_equal(a[key], b[key])
    assert S.swa_sync_status() == 0
