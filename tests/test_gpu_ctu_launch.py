"""GPU test of the FP64 unsplit step on either side of one block (16 x 8 cells)
per SM, where its launches are chained up to: the oracle's bits over steps that
follow one another, gauges included."""
import numpy as np
import pytest

import oracle as O
from paper_1605_05320_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# blocks: 152, 153 (both sides on a GPU of 152 SMs), 238, 475
@pytest.mark.parametrize("nx,ny", [(128, 152), (144, 130), (210, 136), (300, 200)])
def test_unsplit_step_matches_the_oracle_bit_for_bit(nx, ny):
    from paper_1605_05320_gb300 import build
    build.build()
    from paper_1605_05320_gb300 import swadj as S
    S.load()
    sc = synth.small_2d(nx, ny, seed=nx)
    d = S.make_desc(2, nx, ny, 0.0, 0.0, sc.grid.dx, sc.grid.dy, precision=S.SWA_FP64)
    g = S.Grid(d, sc.B)
    g.set_scheme(S.SWA_SCHEME_CTU)
    g.set_state(sc.eta0, sc.hu0, sc.hv0, 0.0)
    xy = torch.tensor([[0.4 * nx * sc.grid.dx, 0.6 * ny * sc.grid.dy]], dtype=torch.float64,
                      device="cuda")
    series = torch.zeros((12, 1), dtype=torch.float64, device="cuda")
    S.swa_grid_record_gauges(g.h, 1, xy, series, None, 12)
    g.step(12, 1e300)
    st = g.get_state()
    assert S.swa_sync_status() == 0
    og = O.Grid.from_spec(sc.grid, scheme=O.SCHEME_CTU)
    h, u, v, t = sc.eta0 - sc.B, sc.hu0, sc.hv0, 0.0
    for k in range(12):
        assert series[k, 0].item() == O.gauge(og, h, sc.B, xy.cpu().numpy())[0]
        h, u, v, _, n = O.fwd_run(og, h, u, v, sc.B, 1, 1e300)
    assert np.array_equal(st["h"], h)
    assert np.array_equal(st["hu"], u)
    assert np.array_equal(st["hv"], v)
