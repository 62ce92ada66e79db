"""GPU test of the FP64 division and square root of the FP64 sweeps: equal to
the compiler's IEEE operations bit for bit over 2.7e8 operands (random,
beside powers of two, beside exact quotients and squares, any bit pattern),
and of the sweeps' segments: results do not depend on how a grid is cut."""
import os
import subprocess

import numpy as np
import pytest

import oracle as O
from paper_1605_05320_gb300 import build as B
from paper_1605_05320_gb300 import synth

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

HERE = os.path.dirname(os.path.abspath(__file__))


def test_division_and_root_round_as_the_compilers(tmp_path):
    exe = str(tmp_path / "ops64_check")
    src = os.path.join(HERE, "native", "ops64_check.cu")
    subprocess.run([B._nvcc(), "-fmad=false"] + B.NVCC_FLAGS + [src, "-o", exe], check=True,
                   capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("nx,ny", [(2, 2), (5, 3), (2, 130), (130, 2), (31, 33), (33, 65),
                                   (64, 200), (400, 37)])
@pytest.mark.parametrize("order,bc,wetdry", [(2, (0, 0, 0, 0), 0), (1, (1, 0, 0, 1), 0),
                                             (2, (1, 1, 1, 1), 1)])
def test_sweeps_match_the_oracle_bit_for_bit(nx, ny, order, bc, wetdry):
    """Odd sizes, still water beside waves, land: the oracle's bits."""
    B.build()
    from paper_1605_05320_gb300 import swadj as S
    S.load()
    sc = synth.small_2d(nx, ny, seed=nx + ny, L=nx * 5e3)
    Bt, eta, hu, hv = sc.B.copy(), sc.eta0.copy(), sc.hu0.copy(), sc.hv0.copy()
    i = np.arange(nx * ny) % nx
    still = i > nx // 2          # at rest to the right of the middle
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
    g.step(15, 1e300)
    st = g.get_state()
    assert S.swa_sync_status() == 0
    og = O.Grid.from_spec(sc.grid, order=order, bc=bc, cfl=d.cfl, wetdry=wetdry)
    h, u, v, t, n = O.fwd_run(og, eta - Bt, hu, hv, Bt, 15, 1e300)
    assert g.time()[0] == t and g.time()[2] == n
    assert np.array_equal(st["h"], h)
    assert np.array_equal(st["hu"], u)
    assert np.array_equal(st["hv"], v)


@pytest.mark.parametrize("nx,ny,order,bc", [(161, 130, 2, (0, 0, 0, 0)), (3, 700, 1, (1, 1, 1, 1)),
                                            (700, 33, 2, (1, 0, 0, 1)), (2, 650, 2, (0, 1, 1, 0))])
@pytest.mark.parametrize("precision", [0, 1])
def test_adjoint_sweeps_match_the_oracle_bit_for_bit(nx, ny, order, bc, precision):
    """Sizes that take the adjoint's sweep passes, with an island, snapshots
    in both storage types."""
    B.build()
    from paper_1605_05320_gb300 import swadj as S
    S.load()
    sc = synth.small_2d(nx, ny, seed=nx + ny, L=nx * 5e3)
    Bt = sc.B.copy()
    Bt[(np.arange(nx * ny) % 61) == 17] = 2.0
    t_f = 40 * 0.75 * sc.grid.dx / np.sqrt(9.81 * 4000.0)
    d = S.make_desc(2, nx, ny, 0.0, 0.0, sc.grid.dx, sc.grid.dy, precision=S.SWA_FP64,
                    order=order, bc=bc)
    adj = S.Adjoint(d, Bt, sc.phi, t_f)
    store = S.SnapStore(adj, adj.info()[0] // 7 + 3, precision)
    store.run_adjoint(7)
    og = O.Grid.from_spec(sc.grid, order=order, bc=bc)
    snaps, tau, N, _ = O.adj_run(og, np.maximum(-Bt, 0.0), sc.phi, t_f, 7)
    assert adj.info()[0] == N
    assert np.array_equal(adj.get_state().ravel(), snaps[-1].ravel())
    assert np.array_equal(store.info()[1], np.asarray(tau))
    esz, dt = (8, torch.float64) if precision == S.SWA_FP64 else (4, torch.float32)
    got = store.ws[:snaps.size * esz].view(dt).cpu().numpy()
    assert np.array_equal(got, snaps.ravel().astype(got.dtype))
