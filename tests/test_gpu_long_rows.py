"""GPU test of the FP64 2D step on grids of a few long rows, which take the
tiled kernel where the sweeps' segments would grow: the oracle's bits on either
side of the rule's line (the x-pass's segments, one wave of tiles), with and
without wet/dry, gauges recorded by the step included."""
import numpy as np
import pytest

import oracle as O
from paper_1605_05320_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny", [(1200, 3), (1900, 4), (3001, 2), (4864, 4), (4865, 4),
                                   (2400, 8), (2500, 9)])
@pytest.mark.parametrize("order,bc,wetdry", [(2, (0, 0, 0, 0), 0), (1, (1, 0, 0, 1), 0),
                                             (2, (1, 1, 1, 1), 1)])
def test_long_rows_match_the_oracle_bit_for_bit(nx, ny, order, bc, wetdry):
    from paper_1605_05320_gb300 import build
    build.build()
    from paper_1605_05320_gb300 import swadj as S
    S.load()
    sc = synth.small_2d(nx, ny, seed=nx + ny, L=nx * 5e3)
    Bt, eta, hu, hv = sc.B.copy(), sc.eta0.copy(), sc.hu0.copy(), sc.hv0.copy()
    i = np.arange(nx * ny) % nx
    still = i > nx // 2
    eta[still], hu[still], hv[still] = 0.0, 0.0, 0.0
    if wetdry:
        land = i > (4 * nx) // 5
        Bt[land] = 3.0
        eta[land] = 3.0
    d = S.make_desc(2, nx, ny, 0.0, 0.0, sc.grid.dx, sc.grid.dy, precision=S.SWA_FP64,
                    order=order, bc=bc, cfl=0.5 if wetdry else 0.75)
    g = S.Grid(d, Bt)
    if wetdry:
        g.set_wetdry(True)
    g.set_state(eta, hu, hv, 0.0)
    steps = 9
    xy = torch.tensor([[0.3 * nx * sc.grid.dx, 0.5 * ny * sc.grid.dy]], dtype=torch.float64,
                      device="cuda")
    series = torch.zeros((steps, 1), dtype=torch.float64, device="cuda")
    S.swa_grid_record_gauges(g.h, 1, xy, series, None, steps)
    og = O.Grid.from_spec(sc.grid, order=order, bc=bc, cfl=d.cfl, wetdry=wetdry)
    h, u, v, t = eta - Bt, hu, hv, 0.0
    for k in range(steps):
        ref = O.gauge(og, h, Bt, xy.cpu().numpy())[0]
        g.step(1, 1e300)
        h, u, v, dt, n = O.fwd_run(og, h, u, v, Bt, 1, 1e300)
        assert series[k, 0].item() == ref and n == 1
    st = g.get_state()
    assert S.swa_sync_status() == 0 and g.time()[2] == steps
    assert np.array_equal(st["h"], h)
    assert np.array_equal(st["hu"], u)
    assert np.array_equal(st["hv"], v)
