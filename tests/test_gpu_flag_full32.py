"""GPU test of the FP32 full flag pass on the adjoint's own grid where it keeps
several snapshots of a cell in flight: windows of every length from one
snapshot up, grids of odd size, cells shared among threads and not, against the
oracle on the stored (float) values.

Tolerance: m is the largest |product| of three float multiply-adds, at a
window's end interpolated with two more: at most 6 roundings, each 2^-24 of the
sum of the absolute products, and the two float weights: 8 * 2^-24."""
import numpy as np
import pytest

import oracle as O
from paper_1605_05320_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("nx,ny", [(33, 31), (401, 101), (257, 1), (1999, 1), (90001, 1)])
@pytest.mark.parametrize("mode", [0, 1])
def test_windows_of_every_length(nx, ny, mode):
    from paper_1605_05320_gb300 import build
    build.build()
    from paper_1605_05320_gb300 import swadj as S
    S.load()
    n, ndim = nx * ny, 1 if ny == 1 else 2
    sc = synth.small_2d(nx, max(ny, 2), seed=nx, L=nx * 1e3)
    f32 = lambda a: np.float32(a[:n]).astype(np.float64)
    B, eta, hu, hv = -f32(-sc.B), f32(sc.eta0) + 0.25, f32(sc.hu0) + 3.0, f32(sc.hv0) - 2.0
    if ndim == 1:
        hv = np.zeros(n)
    dx, dy = sc.grid.dx, sc.grid.dy if ndim == 2 else 1.0
    d = S.make_desc(ndim, nx, ny, 0.0, 0.0, dx, dy, precision=S.SWA_FP32)
    rng = np.random.default_rng(nx)
    phi = rng.uniform(-1.0, 1.0, (ndim + 1, n))
    K = 41
    t_f = (K - 1) * 0.75 * dx / np.sqrt(9.81 * np.abs(B).max())
    adj = S.Adjoint(d, B, phi, t_f)
    store = S.SnapStore(adj, adj.info()[0] + 3, S.SWA_FP32)
    store.run_adjoint(1)
    K, tau = store.info()
    snaps = store.ws[:K * (ndim + 1) * n * 4].view(torch.float32).cpu().numpy().astype(np.float64)
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
    for w in list(range(0, 20)) + [K - 1]:
        for part in (0.0, 0.4):    # window ends on a snapshot, and between two
            t_s = t_f - (w + part) * t_f / (K - 1)
            if t_s < 0:
                continue
            S.swa_flag_cells(g.h, store.h, t_s, t_f, 0.5 * scale, mode, fl, m, c)
            torch.cuda.synchronize()
            got, f = m.cpu().numpy(), fl.cpu().numpy()
            _, ref, _ = O.flag(og, eta - B, hu, hv, B, 0.0, og, hbar, snaps, tau, t_s, t_f,
                               0.5 * scale, mode)
            assert np.abs(got - ref).max() <= 8 * 2.0 ** -24 * scale, (w, part)
            assert np.array_equal(f, got >= np.float32(0.5 * scale)) and int(c.item()) == f.sum()
    assert S.swa_sync_status() == 0
