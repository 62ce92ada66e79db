"""GPU test of the FP64 1D step's strips: the oracle's bits at sizes beside the
strip edges and beyond one strip per block, with still water and with land."""
import numpy as np
import pytest

import oracle as O

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


@pytest.mark.parametrize("nx", [2, 3, 27, 28, 29, 57, 2000, 30001])
@pytest.mark.parametrize("order,wall,wetdry", [(2, 0, 0), (1, 1, 0), (2, 1, 1)])
def test_1d_strips_match_the_oracle_bit_for_bit(S, nx, order, wall, wetdry):
    rng = np.random.default_rng(nx)
    B = -rng.uniform(50.0, 300.0, nx)
    eta, hu = rng.uniform(-1, 1, nx), rng.uniform(-20, 20, nx)
    still = np.arange(nx) > (2 * nx) // 3
    eta[still], hu[still] = 0.0, 0.0
    if wetdry:
        land = np.arange(nx) % 17 == 11
        B[land], eta[land], hu[land] = 2.0, 2.0, 0.0
    d = S.make_desc(1, nx, 1, 0.0, 0.0, 500.0, 1.0, precision=S.SWA_FP64, order=order,
                    bc=(wall,) * 4, cfl=0.45)
    g = S.Grid(d, B)
    if wetdry:
        g.set_wetdry(True)
    g.set_state(eta, hu, None, 0.0)
    g.step(11, 1e300)
    st = g.get_state()
    assert S.swa_sync_status() == 0
    og = O.Grid(1, nx, 1, 0.0, 0.0, 500.0, 1.0, order=order, bc=(wall,) * 4, cfl=0.45,
                wetdry=wetdry)
    h, u, _, t, n = O.fwd_run(og, eta - B, hu, np.zeros(nx), B, 11, 1e300)
    assert g.time()[0] == t and n == 11
    assert np.array_equal(st["h"], h) and np.array_equal(st["hu"], u)
