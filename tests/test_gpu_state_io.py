"""GPU tests of setting and reading states from device arrays in one launch:
equal to the host path's values bit for bit, on the stream given, for the
fields asked for only."""
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


def dev(a):
    return torch.tensor(a, dtype=torch.float64, device="cuda")


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(2, 2), (257, 1), (130, 61)])
@pytest.mark.parametrize("wetdry", [0, 1])
def test_grid_state_from_and_to_the_device(S, precision, nx, ny, wetdry):
    ndim = 1 if ny == 1 else 2
    sc = synth.small_2d(nx, max(ny, 2), seed=nx)
    n = nx * ny
    B, eta, hu, hv = (a[:n].copy() for a in (sc.B, sc.eta0, sc.hu0, sc.hv0))
    if wetdry:
        B[n // 2] = eta[n // 2] = 5.0
        hu[n // 2] = hv[n // 2] = 0.0
    d = S.make_desc(ndim, nx, ny, 0.0, 0.0, 1e3, 1e3 if ndim == 2 else 1.0, precision=precision)
    st = torch.cuda.Stream()
    grids = []
    for on_device in (False, True):
        g = S.Grid(d, B)
        if wetdry:
            g.set_wetdry(True)
        a = (eta, hu, hv)
        if on_device:
            torch.cuda.synchronize()
            a = tuple(dev(x) for x in a)
            torch.cuda.synchronize()
            g.set_state(*a, 3.0, stream=st)
        else:
            g.set_state(*a, 3.0)
        g.step(3, 1e300, stream=st if on_device else None)
        st.synchronize()
        grids.append(g)
    assert grids[0].time() == grids[1].time()
    x, y = grids[0].get_state(), grids[1].get_state()
    for k in x:
        assert np.array_equal(x[k], y[k]), k
    out = {k: torch.full((n,), -7.0, dtype=torch.float64, device="cuda") for k in x}
    torch.cuda.synchronize()
    S.swa_get_state(grids[1].h, out["h"], None, out["hv"], out["eta"], S.SWA_DEVICE, st)
    st.synchronize()
    for k in x:
        ref = np.full(n, -7.0) if k == "hu" else x[k]
        assert np.array_equal(out[k].cpu().numpy(), ref), k
    assert S.swa_sync_status() == 0


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("nx,ny", [(33, 1), (41, 30)])
def test_adjoint_state_from_and_to_the_device(S, precision, nx, ny):
    ndim = 1 if ny == 1 else 2
    nc, n = ndim + 1, nx * ny
    phi = np.random.default_rng(nx).uniform(-1, 1, (nc, n))
    d = S.make_desc(ndim, nx, ny, 0.0, 0.0, 1e3, 1e3 if ndim == 2 else 1.0, precision=precision)
    a = S.Adjoint(d, np.full(n, -3000.0), phi, 200.0)
    a.step(7)
    ref = a.get_state()
    q = dev(phi)
    S.swa_set_adjoint_state(a.h, q, S.SWA_DEVICE)
    a.step(7)
    out = torch.zeros_like(q)
    S.swa_get_adjoint_state(a.h, out, S.SWA_DEVICE)
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), ref)
    assert np.array_equal(a.get_state(), ref)


def test_patch_states_on_the_device(S):
    rng = np.random.default_rng(3)
    pats = [(1, 0.0, 0.0, 9, 70, 1e3, 1e3), (2, 0.0, 0.0, 64, 31, 500.0, 500.0)]
    common = S.make_desc(2, 2, 2, 0.0, 0.0, 1e3, 1e3, precision=S.SWA_FP32)
    f = [[rng.uniform(-1, 1, p[3] * p[4]) for _ in range(3)] for p in pats]
    got = []
    for on_device in (False, True):
        ps = S.PatchSet(pats, [np.full(p[3] * p[4], -3000.0) for p in pats], common)
        for k in range(2):
            ps.set_state(k, *(dev(a) if on_device else a for a in f[k]))
        for lev in (1, 2):
            ps.start(lev, 1.0)
            ps.step(lev, 3)      # an odd number: the other buffer is current
        got.append((ps, [ps.get_state(k) for k in range(2)], ps.time(1), ps.time(2)))
    assert got[0][2:] == got[1][2:]
    for k in range(2):
        n = pats[k][3] * pats[k][4]
        out = [torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(4)]
        S.swa_patches_get_state(got[1][0].h, k, *out, S.SWA_DEVICE)
        torch.cuda.synchronize()
        for key, o in zip(("h", "hu", "hv", "eta"), out):
            assert np.array_equal(got[0][1][k][key], got[1][1][k][key])
            assert np.array_equal(o.cpu().numpy(), got[0][1][k][key])


def test_conversion_equals_the_hardwares(tmp_path):
    """Doubles at, beside and between floats and of any bit pattern to float:
    the hardware's bits."""
    import os
    import subprocess

    from paper_1605_05320_gb300 import build as B
    exe = str(tmp_path / "convert_check")
    src = os.path.join(os.path.dirname(os.path.abspath(__file__)), "native", "convert_check.cu")
    subprocess.run([B._nvcc()] + B.NVCC_FLAGS + [src, "-o", exe], check=True,
                   capture_output=True)
    r = subprocess.run([exe], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr


def test_default_stream_is_the_current_one(S):
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert S._stream(None) == side.cuda_stream == S._stream(side)
    assert S._stream(None) == torch.cuda.current_stream().cuda_stream
