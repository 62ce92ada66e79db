"""Adjoint units left alone while they and their neighbours are zero: the
FP32 2D one-step launch gives every snapshot and the state that the two-step
launch gives, which computes every cell, from a target beside the edges of the
strips and of the grid, through a second initial state in the same buffers and
launches of both kinds in turn."""
import numpy as np
import pytest

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


def _spot(nx, ny, x, y):
    """A phi of one cell's elevation and its neighbour's momentum."""
    q = np.zeros((3, ny, nx))
    q[0, y, x] = 1.0
    q[1, y, max(x - 1, 0)] = -0.5
    return q.reshape(3, -1)


# widths of whole strips (28), one column and one less over; heights that
# leave a last strip of one row and of all
@pytest.mark.parametrize("shape", [(28, 4), (29, 5), (113, 97), (140, 64), (700, 333)])
@pytest.mark.parametrize("bc", [(0, 0, 0, 0), (1, 1, 1, 1)])
def test_still_units_match_the_full_computation(S, shape, bc):
    nx, ny = shape
    sc = synth.small_2d(nx, ny, seed=9)
    d = S.make_desc(2, nx, ny, 0.0, 0.0, sc.adj_grid.dx, sc.adj_grid.dy,
                    precision=S.SWA_FP32, order=2, bc=bc)
    spots = [(0, 0), (nx - 1, ny - 1), (27, ny // 2), (min(28, nx - 1), 0)]

    def run(k):
        adj = S.Adjoint(d, sc.B_adj, _spot(nx, ny, *spots[0]), sc.t_f)
        S.swa_adjoint_set_steps_per_pass(adj.h, k)
        out = []
        for n, (x, y) in enumerate(spots):
            if n:
                S.swa_set_adjoint_state(adj.h, np.ascontiguousarray(_spot(nx, ny, x, y)),
                                        S.SWA_HOST)
            for steps in (1, 2, 7):
                adj.step(steps)
                out.append(np.array(adj.get_state()))
            if k == 1:   # both kinds of launch in turn
                S.swa_adjoint_set_steps_per_pass(adj.h, 2)
                adj.step(2)
                S.swa_adjoint_set_steps_per_pass(adj.h, 1)
                adj.step(3)
            else:
                adj.step(5)
            out.append(np.array(adj.get_state()))
        return out

    a, b = run(1), run(2)
    assert S.swa_sync_status() == 0
    for n, (u, v) in enumerate(zip(a, b)):
        assert np.array_equal(u, v), (shape, bc, n)
        assert np.abs(u).max() > 0.0


def test_snapshots_of_still_units(S):
    """Snapshots are written in full while most units are still."""
    sc = synth.small_2d(300, 210, seed=4)
    d = S.make_desc(2, 300, 210, 0.0, 0.0, sc.adj_grid.dx, sc.adj_grid.dy,
                    precision=S.SWA_FP32, order=2)
    n, out = sc.adj_grid.n, []
    for k in (1, 2):
        adj = S.Adjoint(d, sc.B_adj, _spot(300, 210, 150, 100), sc.t_f)
        S.swa_adjoint_set_steps_per_pass(adj.h, k)
        N, _, _ = adj.info()
        store = S.SnapStore(adj, N // 3 + 3, S.SWA_FP32)
        store.ws[: (N // 3 + 3) * 3 * n * 4].fill_(255)   # not zero where nothing is written
        store.run_adjoint(3)
        K, _ = store.info()
        out.append(store.ws[: K * 3 * n * 4].cpu().numpy().view(np.float32).copy())
    assert S.swa_sync_status() == 0
    assert np.array_equal(out[0], out[1])
