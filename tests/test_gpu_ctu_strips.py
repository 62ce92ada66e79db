"""GPU tests of the FP32 unsplit step's strips against the oracle's unsplit
step at sizes beside the strip edges: calm water with part of it at rest under
every boundary condition, and smooth flow faster than its waves along x, y or
both (the forms for edges that are not subsonic).

Tolerance: an FP32 step rounds sums of fluxes.  With E the scale of the surface
(max |eta| + max |momentum| / s, s the largest wave speed) and M = s E that of
the momenta, each of the some 60 roundings a value takes in a step is at most
2^-24 of its scale (the CFL condition bounds nu times a flux by it), and the
steps' errors add: 64 * 2^-24 * steps of E and M."""
import numpy as np
import pytest

import oracle as O
from paper_1605_05320_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny", [(2, 2), (27, 5), (28, 4), (29, 37), (57, 66), (130, 3)])
@pytest.mark.parametrize("order,bc,fast", [(2, (0, 0, 0, 0), ""), (2, (1, 1, 1, 1), ""),
                                           (1, (0, 1, 1, 0), ""), (2, (0, 0, 0, 0), "x"),
                                           (2, (0, 0, 0, 0), "y"), (1, (0, 0, 0, 0), "xy")])
def test_strips_match_the_oracle(nx, ny, order, bc, fast):
    from paper_1605_05320_gb300 import build
    build.build()
    from paper_1605_05320_gb300 import swadj as S
    S.load()
    sc = synth.small_2d(nx, ny, seed=nx * ny, L=nx * 5e3)
    steps, n = 6, nx * ny
    i, j = np.arange(n) % nx, np.arange(n) // nx

    def f32(a):
        return np.float32(a).astype(np.float64)

    B = -f32(-sc.B)
    eta, hu, hv = f32(sc.eta0), f32(sc.hu0), f32(sc.hv0)
    if fast:
        B = np.full(n, -10.0)
        hu = f32((150.0 if "x" in fast else 3.0) + np.sin(0.4 * i) * np.cos(0.3 * j))
        hv = f32((-140.0 if "y" in fast else -2.0) + np.cos(0.3 * i + 0.2 * j))
        eta = f32(0.3 * np.sin(0.3 * i) * np.cos(0.2 * j))
    else:
        still = i > (2 * nx) // 3
        eta[still], hu[still], hv[still] = 0.0, 0.0, 0.0
    d = S.make_desc(2, nx, ny, 0.0, 0.0, sc.grid.dx, sc.grid.dy, precision=S.SWA_FP32,
                    order=order, bc=bc, cfl=0.5)
    g = S.Grid(d, B)
    g.set_scheme(S.SWA_SCHEME_CTU)
    g.set_state(eta, hu, hv, 0.0)
    g.step(steps, 1e300)
    st = g.get_state()
    assert S.swa_sync_status() == 0
    og = O.Grid.from_spec(sc.grid, order=order, bc=bc, cfl=0.5, scheme=O.SCHEME_CTU)
    h, u, v, t, k = O.fwd_run(og, eta - B, hu, hv, B, steps, 1e300)
    tol = 64 * 2.0 ** -24 * steps
    assert k == steps and abs(g.time()[0] - t) <= tol * t
    s = (np.maximum(np.abs(u), np.abs(v)) / h + np.sqrt(9.81 * h)).max()
    E = np.abs(h + B).max() + max(np.abs(u).max(), np.abs(v).max()) / s
    assert np.abs(st["eta"] - (h + B)).max() <= tol * E
    assert np.abs(st["hu"] - u).max() <= tol * s * E
    assert np.abs(st["hv"] - v).max() <= tol * s * E
