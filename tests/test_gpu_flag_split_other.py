"""GPU test of the full flag pass over another grid where the snapshots of a cell
are shared among 1 to 32 threads, by the number of cells and of snapshots: m and
flags against the oracle, in both precisions.

Tolerance: FP64 m to the rounding of its float output and of sums of four weighted
values and three products (2^-22 of the largest); FP32 the bilinear sums and the
three products round at most 12 times, each 2^-24 of the sum of the absolute
products, and the stencil's float weights are within 2^-20 (16 * 2^-24 in all for
weights of a coordinate below 64 cells)."""
import numpy as np
import pytest

import oracle as O
from paper_1605_05320_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,anx,any_,K", [(6, 5, 4, 3, 16), (17, 9, 8, 5, 130),
                                              (64, 48, 16, 12, 70), (64, 50, 60, 44, 20),
                                              (160, 100, 40, 25, 40), (250, 160, 50, 32, 33),
                                              (300, 240, 60, 48, 9)])
@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("mode", [0, 1])
def test_full_pass_matches_the_oracle(nx, ny, anx, any_, K, precision, mode):
    from paper_1605_05320_gb300 import build
    build.build()
    from paper_1605_05320_gb300 import swadj as S
    S.load()
    fp32 = precision == S.SWA_FP32
    n, na, L = nx * ny, anx * any_, nx * 5e3
    sc, ac = synth.small_2d(nx, ny, seed=nx, L=L), synth.small_2d(anx, any_, seed=nx, L=L)
    adx, ady = L / anx, ny * sc.grid.dx / any_
    f32 = (lambda a: np.float32(a).astype(np.float64)) if fp32 else (lambda a: a)
    B, eta, hu, hv = -f32(-sc.B), f32(sc.eta0) + 0.25, f32(sc.hu0) + 3.0, f32(sc.hv0) - 2.0
    d = S.make_desc(2, nx, ny, 0.0, 0.0, sc.grid.dx, sc.grid.dy, precision=precision)
    ad = S.make_desc(2, anx, any_, 0.0, 0.0, adx, ady, precision=precision, bc=(1, 1, 1, 1))
    Ba = ac.B.copy()
    Ba[na // 2] = 1.0                      # a dry adjoint cell
    phi = np.random.default_rng(nx).uniform(-1.0, 1.0, (3, na))
    t_f = (K - 1) * 0.75 * min(adx, ady) / np.sqrt(9.81 * 4000.0)
    adj = S.Adjoint(ad, Ba, phi, t_f)
    store = S.SnapStore(adj, adj.info()[0] + 3, precision)
    store.run_adjoint(1)
    K, tau = store.info()
    esz, dt = (4, torch.float32) if fp32 else (8, torch.float64)
    snaps = store.ws[:K * 3 * na * esz].view(dt).cpu().numpy().astype(np.float64)
    snaps = snaps.reshape(K, 3, na)
    g = S.Grid(d, B)
    g.set_state(eta, hu, hv, 0.0)
    og = O.Grid(2, nx, ny, 0.0, 0.0, sc.grid.dx, sc.grid.dy)
    oa = O.Grid(2, anx, any_, 0.0, 0.0, adx, ady)
    fl = torch.zeros(n, dtype=torch.uint8, device="cuda")
    m = torch.zeros(n, dtype=torch.float32, device="cuda")
    c = torch.zeros(1, dtype=torch.int64, device="cuda")
    scale = max(np.abs(snaps[:, k]).max() * np.abs(q).max() for k, q in enumerate((eta, hu, hv)))
    tol = 3 * scale * (16 * 2.0 ** -24 if fp32 else 2.0 ** -22)
    for t_s in (0.0, 0.45 * t_f, 0.97 * t_f):
        S.swa_flag_cells(g.h, store.h, t_s, t_f, 0.3 * scale, mode, fl, m, c)
        torch.cuda.synchronize()
        got, f = m.cpu().numpy(), fl.cpu().numpy()
        _, ref, _ = O.flag(og, eta - B, hu, hv, B, 0.0, oa, np.maximum(-Ba, 0.0), snaps, tau, t_s,
                           t_f, 0.3 * scale, mode)
        assert np.abs(got - ref).max() <= tol
        near = np.abs(ref - 0.3 * scale) <= tol
        assert np.array_equal(f[~near], (ref >= 0.3 * scale)[~near]) and int(c.item()) == f.sum()
    assert S.swa_sync_status() == 0
