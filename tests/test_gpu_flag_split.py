"""GPU tests of the flag pass's two ways to share work among threads: the
pruned pass's tiles (flags and count equal the full pass's) and the full
pass's snapshots of one cell among several threads (equal the oracle's m).

The pruned pass is compared exactly.  m in FP64 is compared with the oracle's
to the rounding of its float output (2^-23 relative) plus that of a sum of
three products."""
import numpy as np
import pytest

import oracle as O
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


def flags_of(S, g, store, t_s, t_f, tol, mode, n, want_m, offset=0):
    buf = torch.full((n + 8,), 9, dtype=torch.uint8, device="cuda")
    fl = buf[offset:offset + n]
    m = torch.zeros(n, dtype=torch.float32, device="cuda") if want_m else None
    c = torch.zeros(1, dtype=torch.int64, device="cuda")
    S.swa_flag_cells(g.h, store.h, t_s, t_f, tol, mode, fl, m, c)
    torch.cuda.synchronize()
    assert (buf[:offset] == 9).all() and (buf[offset + n:] == 9).all()
    return fl.cpu().numpy(), int(c.item()), None if m is None else m.cpu().numpy()


@pytest.mark.parametrize("nx,ny,anx,any_", [(64, 40, 64, 40), (61, 40, 16, 10), (8, 4, 4, 3),
                                            (130, 90, 520, 360), (1023, 70, 128, 9), (260, 33, 65 * 4, 33)])
@pytest.mark.parametrize("mode", [0, 1])
def test_pruned_flags_equal_the_full_pass(S, nx, ny, anx, any_, mode):
    L = nx * 5e3
    sc = synth.small_2d(nx, ny, seed=nx, L=L)
    ac = synth.small_2d(anx, any_, seed=nx, L=L)
    ady = ny * sc.grid.dx / any_
    d = S.make_desc(2, nx, ny, 0.0, 0.0, sc.grid.dx, sc.grid.dy, precision=S.SWA_FP32)
    ad = S.make_desc(2, anx, any_, 0.0, 0.0, L / anx, ady, precision=S.SWA_FP32)
    Ba = ac.B.copy()
    Ba[7 % Ba.size] = 1.0                      # a dry adjoint cell
    t_f = 330 * 0.75 * min(L / anx, ady) / np.sqrt(9.81 * 4000.0)
    adj = S.Adjoint(ad, Ba, ac.phi, t_f)
    store = S.SnapStore(adj, adj.info()[0] + 3, S.SWA_FP32)
    store.run_adjoint(1)                       # more than 256 snapshots
    B, eta, hu, hv = sc.B.copy(), sc.eta0.copy(), sc.hu0.copy(), sc.hv0.copy()
    i = np.arange(nx * ny) % nx
    rest = i > (2 * nx) // 3
    eta[rest], hu[rest], hv[rest] = 0.0, 0.0, 0.0
    g = S.Grid(d, B)
    seen = 0
    for t in (0.0, 0.37 * t_f):
        g.set_state(eta, hu, hv, t)
        for t_s in (0.0, 0.9 * t_f, t_f):
            m = flags_of(S, g, store, t_s, t_f, 1.0, mode, nx * ny, True)[2]
            for tol in [0.0] + [float(np.quantile(m[m > 0], q)) for q in (0.3, 0.9, 0.999)]:
                full = flags_of(S, g, store, t_s, t_f, tol, mode, nx * ny, True)
                for offset in (0, 1):
                    f, c, _ = flags_of(S, g, store, t_s, t_f, tol, mode, nx * ny, False, offset)
                    assert np.array_equal(f, full[0]) and c == full[1]
                seen += full[1]
    assert seen > 0 and S.swa_sync_status() == 0


@pytest.mark.parametrize("nx,every", [(2, 1), (7, 1), (9, 3), (300, 1), (5000, 40)])
@pytest.mark.parametrize("mode", [0, 1])
def test_snapshots_shared_among_threads_match_the_oracle(S, nx, every, mode):
    sc = synth.config1(nx)
    B = np.where(np.arange(nx) % 50 == 49, 1.0, sc.B) if nx > 100 else sc.B
    t_f = 300 * 0.75 * sc.grid.dx / np.sqrt(9.81 * 4000.0)
    d = S.make_desc(1, nx, 1, sc.grid.x_lo, 0.0, sc.grid.dx, 1.0, precision=S.SWA_FP64)
    adj = S.Adjoint(d, B, sc.phi, t_f)
    store = S.SnapStore(adj, adj.info()[0] // every + 3, S.SWA_FP64)
    store.run_adjoint(every)
    g = S.Grid(d, sc.B)
    og = O.Grid.from_spec(sc.grid)
    snaps, tau, _, _ = O.adj_run(og, np.maximum(-B, 0.0), sc.phi, t_f, every)
    for t in (0.0, 0.31 * t_f):
        g.set_state(sc.eta0 + 0.1, sc.hu0 + 3.0, None, t)
        h = sc.eta0 + 0.1 - sc.B
        for t_s in (0.4 * t_f, t_f):
            f, c, m = flags_of(S, g, store, t_s, t_f, 1e-3, mode, nx, True)
            fr, mr, cr = O.flag(og, h, sc.hu0 + 3.0, sc.hv0, sc.B, t, og, np.maximum(-B, 0.0), snaps,
                                tau, t_s, t_f, 1e-3, mode)
            assert np.abs(m - mr).max() <= 2.0 ** -22 * max(np.abs(mr).max(), 1e-30)
            near = np.abs(mr - 1e-3) <= 1e-9
            assert np.array_equal(f[~near], fr[~near]) and c == int(f.sum())
