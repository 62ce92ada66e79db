"""GPU test of the FP64 full flag pass on the adjoint's own grid where the snapshots
of a cell are shared among 1 to 32 threads by the rounds they take: m and flags
against the oracle.

Tolerance: m is the largest |product| of three double multiply-adds, rounded to
float: 2^-23 of the largest sum of the absolute products."""
import numpy as np
import pytest

import oracle as O
from paper_1605_05320_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny,K", [(47, 45, 70), (161, 100, 40), (201, 199, 33), (40001, 1, 60),
                                     (20001, 1, 90), (20001, 1, 9)])
@pytest.mark.parametrize("mode", [0, 1])
def test_shared_cells_match_the_oracle(nx, ny, K, mode):
    from paper_1605_05320_gb300 import build
    build.build()
    from paper_1605_05320_gb300 import swadj as S
    S.load()
    n, ndim = nx * ny, 1 if ny == 1 else 2
    sc = synth.small_2d(nx, max(ny, 2), seed=nx, L=nx * 1e3)
    B, eta, hu, hv = sc.B[:n], sc.eta0[:n] + 0.25, sc.hu0[:n] + 3.0, sc.hv0[:n] - 2.0
    if ndim == 1:
        hv = np.zeros(n)
    dx, dy = sc.grid.dx, sc.grid.dy if ndim == 2 else 1.0
    d = S.make_desc(ndim, nx, ny, 0.0, 0.0, dx, dy, precision=S.SWA_FP64)
    rng = np.random.default_rng(nx)
    phi = rng.uniform(-1.0, 1.0, (ndim + 1, n))
    t_f = (K - 1) * 0.75 * dx / np.sqrt(9.81 * np.abs(B).max())
    adj = S.Adjoint(d, B, phi, t_f)
    store = S.SnapStore(adj, adj.info()[0] + 3, S.SWA_FP64)
    store.run_adjoint(1)
    K, tau = store.info()
    snaps = store.ws[:K * (ndim + 1) * n * 8].view(torch.float64).cpu().numpy()
    snaps = snaps.reshape(K, ndim + 1, n)
    g = S.Grid(d, B)
    g.set_state(eta, hu, hv if ndim == 2 else None, 0.0)
    og = O.Grid(ndim, nx, ny, 0.0, 0.0, dx, dy)
    hbar = np.maximum(-B, 0.0)
    fl = torch.zeros(n, dtype=torch.uint8, device="cuda")
    m = torch.zeros(n, dtype=torch.float32, device="cuda")
    c = torch.zeros(1, dtype=torch.int64, device="cuda")
    q = np.stack([eta, hu, hv][:ndim + 1])
    scale = np.abs(q[None] * snaps).sum(axis=1).max()
    for t_s in (0.0, 0.45 * t_f, 0.97 * t_f):
        S.swa_flag_cells(g.h, store.h, t_s, t_f, 0.5 * scale, mode, fl, m, c)
        torch.cuda.synchronize()
        got, f = m.cpu().numpy(), fl.cpu().numpy()
        _, ref, _ = O.flag(og, eta - B, hu, hv, B, 0.0, og, hbar, snaps, tau, t_s, t_f,
                           0.5 * scale, mode)
        tol = 2.0 ** -23 * scale
        assert np.abs(got - ref).max() <= tol
        near = np.abs(ref - 0.5 * scale) <= tol
        assert np.array_equal(f[~near], (ref >= 0.5 * scale)[~near]) and int(c.item()) == f.sum()
    assert S.swa_sync_status() == 0
