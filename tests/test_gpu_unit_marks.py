"""Forward units left alone while they and their neighbours are at rest: the
FP32 2D step gives the state and clock it gives with the shortcut switched off
(an exact zero may differ in sign), through changes of the unit height, the
scheme and the switch, a second state in the same buffers, wet/dry steps in
between, and a hierarchy that averages a wave into a coarse grid at rest.
All comparisons are exact."""
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


def _compare(a, b, what):
    assert a.time() == b.time(), what
    x, y = a.get_state(), b.get_state()
    for k in ("eta", "hu", "hv"):
        assert np.array_equal(x[k], y[k]), (what, k)
    return np.abs(x["eta"]).max()


# widths of whole strips (28), one column over and one less; heights that
# leave a last unit of one row at 4, 16, 32 or 64 rows a unit
@pytest.mark.parametrize("nx,ny", [(28, 5), (57, 33), (113, 129), (280, 129), (500, 257)])
@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 1, 1, 1)])
def test_marks_match_the_full_computation(S, nx, ny, bc):
    sc = synth.small_2d(nx, ny, seed=nx, L=nx * 5e3)
    d = S.make_desc(2, nx, ny, 0.0, 0.0, sc.grid.dx, sc.grid.dy, precision=S.SWA_FP32, bc=bc)
    a, b = S.Grid(d, sc.B), S.Grid(d, sc.B)
    S.swa_grid_set_rest_skip(b.h, 0)

    def both(f):
        f(a)
        f(b)

    z = np.zeros(nx * ny)
    for x, y in [(0, 0), (nx - 1, ny - 1), (min(28, nx - 1), ny // 2)]:
        eta = z.copy()
        eta[y * nx + x] = 0.25
        both(lambda g: g.set_state(eta, z, z, 0.0))
        for rows in (0, 64, 16, 64, 0, 32):
            both(lambda g: S.swa_grid_set_strip_rows(g.h, rows))
            both(lambda g: g.step(3, 1e300))
            assert _compare(a, b, (x, y, rows)) > 0.0
        both(lambda g: g.set_scheme(S.SWA_SCHEME_CTU))
        both(lambda g: g.step(3, 1e300))
        both(lambda g: g.set_scheme(S.SWA_SCHEME_SPLIT))
        S.swa_grid_set_rest_skip(a.h, 0)
        both(lambda g: g.step(2, 1e300))
        S.swa_grid_set_rest_skip(a.h, 1)
        both(lambda g: g.step(3, 1e300))
        _compare(a, b, (x, y, "switched"))
        both(lambda g: g.set_wetdry(1))
        both(lambda g: g.step(2, 1e300))
        both(lambda g: g.set_wetdry(0))
        both(lambda g: g.step(3, 1e300))
        _compare(a, b, (x, y, "wet/dry"))
    assert S.swa_sync_status() == 0


@pytest.mark.parametrize("r", [2, 4])
def test_marks_after_averaging(S, r):
    """A wave that starts on the patch alone reaches the coarse grid, which
    has been at rest for some steps, by averaging."""
    case = synth.amr_basin(120, r, [(70, 60, 20, 24)], rest=True)
    nc, dx, p = 120, case["dx"], case["patches"][0]
    wave = np.asarray(p["eta"]).copy()
    n = int(round(wave.size ** 0.5))
    wave[wave.size // 2 + n // 2] = 0.3
    out = []
    for on in (1, 0):
        d = S.make_desc(2, nc, nc, 0.0, 0.0, dx, dx, precision=S.SWA_FP32, bc=(1, 1, 1, 1))
        g = S.Grid(d, case["coarse"]["B"])
        S.swa_grid_set_rest_skip(g.h, on)
        z = np.zeros(nc * nc)
        g.set_state(z, z, z, 0.0)
        ps = S.PatchSet([p["desc"]], [p["B"]],
                        S.make_desc(2, nc, nc, 0.0, 0.0, dx, dx, precision=S.SWA_FP32))
        ps.set_state(0, p["eta"], p["hu"], p["hv"])
        ps.start(1, 0.0)
        amr = S.Amr(g, ps, 1, r)
        dt, t = 0.6 * 0.75 * dx / np.sqrt(9.81 * 130.0), 0.0
        for k in range(12):
            if k == 4:
                ps.set_state(0, wave, p["hu"], p["hv"])
                ps.start(1, t)
            amr.step(t, dt)
            t += dt
        out.append((g, ps.get_state(0), (ps, amr)))
    assert S.swa_sync_status() == 0
    assert _compare(out[0][0], out[1][0], r) > 0.0
    for k in ("eta", "hu", "hv"):
        assert np.array_equal(out[0][1][k], out[1][1][k]), k
