"""GPU test of the pruned flag pass over another grid at every tile size (32 to
256 quads, chosen from the number of quads) and on either side of the line
below which the full pass runs instead: flags and count equal the full pass's,
rows that do not split into quads and windows of more than 32 groups included."""
import numpy as np
import pytest

from paper_1605_05320_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# quads: 640, 14364, 15000, 29400, 58500, 61440; cells times snapshots beside
# 2^20 with 2440 cells
@pytest.mark.parametrize("nx,ny,anx,any_,K", [(61, 40, 16, 10, 500), (252, 228, 64, 57, 40),
                                              (249, 240, 332, 320, 30), (490, 240, 128, 63, 30),
                                              (975, 240, 244, 60, 24), (1024, 240, 256, 60, 24),
                                              (61, 40, 16, 10, 428), (61, 40, 16, 10, 431)])
@pytest.mark.parametrize("mode", [0, 1])
def test_pruned_pass_equals_the_full_pass(nx, ny, anx, any_, K, mode):
    from paper_1605_05320_gb300 import build
    build.build()
    from paper_1605_05320_gb300 import swadj as S
    S.load()
    n, L = nx * ny, nx * 5e3
    sc, ac = synth.small_2d(nx, ny, seed=nx, L=L), synth.small_2d(anx, any_, seed=nx, L=L)
    ady = ny * sc.grid.dx / any_
    d = S.make_desc(2, nx, ny, 0.0, 0.0, sc.grid.dx, sc.grid.dy, precision=S.SWA_FP32)
    ad = S.make_desc(2, anx, any_, 0.0, 0.0, L / anx, ady, precision=S.SWA_FP32,
                     bc=(1, 1, 1, 1))   # walls keep the adjoint in the domain
    Ba = ac.B.copy()
    Ba[7] = 1.0                      # a dry adjoint cell
    t_f = (K - 1) * 0.75 * min(L / anx, ady) / np.sqrt(9.81 * 4000.0)
    phi = np.random.default_rng(nx + K).uniform(-1.0, 1.0, (3, anx * any_))   # nonzero everywhere
    adj = S.Adjoint(ad, Ba, phi, t_f)
    store = S.SnapStore(adj, adj.info()[0] + 3, S.SWA_FP32)
    store.run_adjoint(1)
    eta, hu, hv = sc.eta0.copy(), sc.hu0.copy(), sc.hv0.copy()
    rest = np.arange(n) % nx > (2 * nx) // 3
    eta[rest], hu[rest], hv[rest] = 0.0, 0.0, 0.0
    g = S.Grid(d, sc.B)
    fl = torch.zeros(n, dtype=torch.uint8, device="cuda")
    m = torch.zeros(n, dtype=torch.float32, device="cuda")
    c = torch.zeros(1, dtype=torch.int64, device="cuda")

    def flags(t_s, tol, want_m):
        fl.fill_(9)
        S.swa_flag_cells(g.h, store.h, t_s, t_f, tol, mode, fl, m if want_m else None, c)
        torch.cuda.synchronize()
        return fl.cpu().numpy(), int(c.item())

    seen = 0
    for t in (0.0, 0.37 * t_f):
        g.set_state(eta, hu, hv, t)
        for t_s in (0.0, 0.9 * t_f, t_f):
            flags(t_s, 1.0, True)
            pos = m[m > 0].cpu().numpy()
            # (no product: a window of one instant just outside the stored times)
            for tol in ([float(np.quantile(pos, q)) for q in (0.3, 0.9, 0.999)] if pos.size
                        else [1e-6]):
                full, pruned = flags(t_s, tol, True), flags(t_s, tol, False)
                assert np.array_equal(pruned[0], full[0]) and pruned[1] == full[1]
                seen += full[1]
    assert seen > 0 and S.swa_sync_status() == 0
