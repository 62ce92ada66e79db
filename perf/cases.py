"""Performance cases: the work that a program using this library has it do,
through the public binding, from the smallest grids to the largest.

A case is a dict of plain values.  Five kinds of call sequence stand for the
library's uses:

  scenario  a forward run: set the state, record gauges, take CFL steps, with
            an adjoint-weighted flag pass after every 10 steps when the run
            has an adjoint (solved beforehand, as a server keeps it, or
            inside the pass, as a plain run does)
  adjoint   a whole adjoint solve with its snapshots, then the flag pass (with
            its m output) that the forward run starts with
  flags     one flag pass of a running forward state against stored snapshots
  patches   batched uneven patches: set, step every level, read back
  amr       a coarse grid with ringed patches: set, hierarchy steps, read back

Fields are formed on the GPU from the seed alone with the scales of the basin
workloads: a 4000 m basin with a tanh shelf and seamounts, and a metre-scale
Gaussian source at rest (`reach` 0) or a train of outgoing waves whose front
has covered `reach` times the domain's width (beyond it the ocean is exactly
at rest, as ahead of a tsunami).
"""
import math
import random

import numpy as np
import torch

from paper_1605_05320_gb300 import swadj as S

DEV = "cuda"
G = 9.81
CFL = 0.75
DRY = 1e-3
FLAG_EVERY = 10          # forward steps between flag passes


def _case(kind, name=None, **kw):
    c = dict(kind=kind, ndim=2, nx=0, ny=0, dx=1e3, fp64=False, order=2, walls=False, steps=0,
             reach=0.0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # The 1D ocean with a step shelf (2000 cells, FP64): every call is a
        # few microseconds, so launches and latency are all there is.
        _case("scenario", "ocean_1d", ndim=1, nx=2000, ny=1, dx=400.0, fp64=True, steps=200,
              gauges=2, adj_n=2000, every=10),
        # A small request to the serving loop: 512^2 over the 2048 km basin,
        # flagged against the resident 2048^2 adjoint.
        _case("scenario", "request_512", nx=512, ny=512, dx=4e3, steps=100, gauges=16,
              adj_n=2048, every=14),
        # The basin workload just after its source is released: most of the
        # ocean is still at rest.
        _case("scenario", "basin_2048", nx=2048, ny=2048, steps=40, gauges=2),
        # The same grid late in a run: waves in every cell.
        _case("scenario", "basin_2048_late", nx=2048, ny=2048, steps=40, gauges=2, reach=1.0),
        # The precision study's grid: 4096^2 half way through, 16 gauges,
        # flagged against a coarser adjoint.
        _case("scenario", "study_4096", nx=4096, ny=4096, steps=20, reach=0.5, gauges=16,
              adj_n=1024, every=20),
        # The adjoint solve of the basin workload, a snapshot every 20 steps.
        _case("adjoint", "adjoint_2048", nx=2048, ny=2048, reach=0.35, t_steps=2000, every=20),
        # One flag pass of the basin workload, half way through its run.
        _case("flags", "flags_2048", nx=2048, ny=2048, reach=0.35, t_steps=2000, every=20,
              adj_n=2048, at=0.4, bracket=False, want_m=False),
        # Uneven patches on three levels, sides 16 to 256, about half of them
        # holding waves.
        _case("patches", "patches", count=480, levels=3, side_lo=16, side_hi=256, ratio=4,
              steps=60, nx=2048, ny=2048, reach=0.35),
        # Two-level mesh refinement on the basin: 64 patches at ratio 4 over
        # the source, 10 coarse steps.
        _case("amr", "amr_2048", nx=2048, ny=2048, steps=10, ratio=4, tiles=8, side=32,
              levels=1),
        # The unsplit update with transverse waves.
        _case("scenario", "unsplit_2048", nx=2048, ny=2048, steps=10, reach=0.5, gauges=2,
              ctu=True),
        # The plain per-grid FP64 form: adjoint solve and forward run.
        _case("scenario", "plain_f64_512", nx=512, ny=512, dx=4e3, fp64=True, steps=60,
              gauges=2, adj_n=512, every=5, reach=0.3, solve=True),
        # Inundation in FP64: waves running up a beach with islands, between
        # walls, odd sizes.
        _case("scenario", "runup_f64", nx=511, ny=350, dx=50.0, fp64=True, steps=40, gauges=4,
              wetdry=True, walls=True, reach=1.0),
    ]


def _spread(rng, lo, hi):
    """A whole number between lo and hi, even over its logarithm."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["ocean", "basin", "basin", "basin", "served", "unsplit", "plain", "runup",
                       "adjoint", "adjoint", "flags", "patches", "amr"])
    order = rng.choice([2, 2, 2, 1])
    walls = rng.random() < 0.3
    reach = rng.choice([0.0, round(rng.uniform(0.1, 1.0), 2)])
    if kind == "ocean":
        n = _spread(rng, 100, 8000)
        return _case("scenario", ndim=1, nx=n, ny=1, dx=800e3 / n, fp64=rng.random() < 0.7,
                     steps=10 * rng.randint(5, 30), gauges=rng.randint(0, 4), order=order,
                     walls=walls, **(dict(adj_n=n, every=10) if rng.random() < 0.5 else {}))
    if kind in ("adjoint", "flags"):
        nx, ny = _spread(rng, 64, 2048), _spread(rng, 64, 2048)
        if kind == "flags":
            nx = 4 * ((nx + 3) // 4) if rng.random() < 0.6 else nx
            return _case("flags", nx=nx, ny=ny, reach=round(rng.uniform(0.1, 1.0), 2), dx=1e3,
                         t_steps=rng.randint(200, 1000), every=rng.randint(10, 20),
                         adj_n=nx if rng.random() < 0.6 else max(64, nx // 4),
                         at=round(rng.uniform(0.0, 0.7), 2), bracket=rng.random() < 0.3,
                         want_m=rng.random() < 0.3)
        f64 = rng.random() < 0.3
        if f64:
            nx, ny = min(nx, 700), min(ny, 700)
        return _case("adjoint", nx=nx, ny=ny, fp64=f64, t_steps=rng.randint(50, 150 if f64 else 1500),
                     every=rng.randint(5, 25), order=order, walls=walls,
                     reach=round(rng.uniform(0.1, 1.0), 2))
    if kind == "patches":
        return _case("patches", count=_spread(rng, 8, 480), levels=rng.randint(1, 3), side_lo=16,
                     side_hi=rng.randint(64, 256), ratio=rng.choice([2, 4]), order=order,
                     steps=2 * rng.randint(5, 30), nx=2048, ny=2048, reach=reach)
    if kind == "amr":
        n = _spread(rng, 256, 2048)
        return _case("amr", nx=n, ny=n, steps=rng.randint(2, 8), ratio=rng.choice([2, 3, 4]),
                     tiles=rng.randint(1, 6), side=rng.randint(8, 24), levels=rng.choice([1, 1, 2]))
    nx, ny = _spread(rng, 64, 4096), _spread(rng, 64, 4096)
    if kind == "served":
        n = rng.choice([512, 1024, 2048])
        return _case("scenario", nx=n, ny=n, dx=2048e3 / n, steps=20, gauges=16, reach=reach,
                     adj_n=rng.choice([512, 1024]), every=rng.randint(10, 20))
    if kind == "basin":
        return _case("scenario", nx=nx, ny=ny, dx=round(rng.uniform(500.0, 4e3)),
                     steps=rng.randint(4, 20), reach=reach, gauges=rng.choice([0, 2, 16]),
                     order=order, walls=walls)
    if kind == "unsplit":
        nx, ny = min(nx, 2048), min(ny, 2048)
        f64 = rng.random() < 0.25
        if f64:
            nx, ny = min(nx, 500), min(ny, 500)
        return _case("scenario", nx=nx, ny=ny, fp64=f64, steps=rng.randint(4, 10), reach=reach,
                     gauges=2, ctu=True, order=order)
    if kind == "runup":
        nx, ny = min(nx, 1500), min(ny, 1200)
        f64 = rng.random() < 0.4
        if f64:
            nx, ny = min(nx, 400), min(ny, 400)
        return _case("scenario", nx=nx, ny=ny, dx=50.0, fp64=f64, steps=rng.randint(10, 40),
                     gauges=2, wetdry=True, walls=True, reach=1.0, order=order)
    nx, ny = min(nx, 600), min(ny, 600)
    return _case("scenario", nx=nx, ny=ny, dx=4e3, fp64=True, steps=10 * rng.randint(1, 5),
                 gauges=2, reach=reach, order=order, walls=walls,
                 **(dict(adj_n=nx, every=5, solve=True) if rng.random() < 0.5 else {}))


# ------------------------------------------------------------------ inputs
def _centres(nx, ny, dx):
    x = (torch.arange(nx, dtype=torch.float64, device=DEV) + 0.5) * dx
    y = (torch.arange(ny, dtype=torch.float64, device=DEV) + 0.5) * dx
    return x.repeat(ny), y.repeat_interleave(nx)


class Ocean:
    """The seeded bottom, waves and target of a case as functions of (x, y)."""

    def __init__(self, c, seed):
        r = random.Random(seed)
        self.c = c
        self.L, self.Ly = c["nx"] * c["dx"], c["ny"] * c["dx"]
        self.amp, self.wid = r.uniform(0.1, 2.0), r.uniform(10e3, 60e3)
        if c["kind"] == "amr":   # the source the patches sit on
            self.src = (0.35 * self.L + r.uniform(0.0, 20e3), 0.5 * self.Ly)
        else:
            self.src = (r.uniform(0.2, 0.6) * self.L, r.uniform(0.2, 0.8) * self.Ly)
        self.lam = max(self.wid, 12 * c["dx"])
        self.target = (0.85 * self.L, r.uniform(0.4, 0.6) * self.Ly)
        self.tw = max(10e3, 3 * c["dx"])
        self.mounts = [(r.uniform(0, 0.78) * self.L, r.uniform(0, 1) * self.Ly,
                        r.uniform(500, 2000), r.uniform(10e3, 50e3)) for _ in range(20)]
        self.gauges = [(r.uniform(0.1, 0.9) * self.L, r.uniform(0.1, 0.9) * self.Ly)
                       for _ in range(c.get("gauges", 0))]

    def bottom(self, x, y):
        c = self.c
        if c.get("wetdry"):   # a beach with islands
            B = -2.0 + 3.0 * x / self.L + 0.2 * torch.cos(y / 90)
            for (mx, my, a, _) in self.mounts[:3]:
                B += a / 700 * torch.exp(-((x - mx) ** 2 + (y - my) ** 2) / (0.06 * self.L) ** 2)
            return B
        if c["ndim"] == 1:
            return torch.where(x < 0.875 * self.L, -4000.0, -200.0).to(torch.float64)
        B = -4000.0 + 1950.0 * (1.0 + torch.tanh((x - 0.85 * self.L) / 30e3))
        for (mx, my, a, w) in self.mounts:
            B += a * torch.exp(-((x - mx) ** 2 + (y - my) ** 2) / (w * w))
        return B.clamp_(max=-50.0)

    def state(self, x, y, B):
        """(eta, hu, hv)."""
        c = self.c
        if c["ndim"] == 1:
            y = torch.full_like(x, self.src[1])
        X, Y = x - self.src[0], y - self.src[1]
        r2 = X * X + Y * Y
        if c.get("wetdry"):
            eta = 0.4 * torch.cos(r2.sqrt() / (8 * c["dx"])) * torch.exp(-r2 / (0.5 * self.L) ** 2)
            h = (eta - B).clamp_(min=0.0)
            dry = h <= 0.0
            m = torch.where(dry, 0.0, 0.3 * eta * (G * h).sqrt() / (r2.sqrt() + c["dx"]))
            return torch.where(dry, B, eta), m * X, m * Y
        if c["reach"] == 0.0:
            eta = self.amp * torch.exp(-r2 / (self.lam * self.lam))
            eta = torch.where(eta < 1e-12, 0.0, eta)
            return eta, torch.zeros_like(eta), torch.zeros_like(eta)
        R = 1.5 * c["reach"] * max(self.L, self.Ly)
        env = (1.0 - r2 / (R * R)).clamp_(min=0.0)
        rr = r2.sqrt()
        eta = self.amp * env * env * torch.cos(6.0 * rr / self.lam) / (1.0 + rr / self.lam).sqrt()
        m = eta * (G * -B).sqrt() / (rr + c["dx"])
        return eta, m * X, m * Y if c["ndim"] == 2 else torch.zeros_like(eta)

    def phi(self, x, y):
        if self.c["ndim"] == 1:
            y = torch.full_like(x, self.target[1])
        e = torch.exp(-((x - self.target[0]) ** 2 + (y - self.target[1]) ** 2) / self.tw ** 2)
        return torch.where(e < 1e-30, 0.0, e)


def _np(t):
    return t.cpu().numpy()


def _desc(c, nx=None, ny=None, dx=None, fp64=None):
    w = 1 if c["walls"] else 0
    fp64 = c["fp64"] if fp64 is None else fp64
    return S.make_desc(c["ndim"], nx or c["nx"], ny or c["ny"], 0.0, 0.0, dx or c["dx"],
                       (dx or c["dx"]) if c["ndim"] == 2 else 1.0,
                       precision=S.SWA_FP64 if fp64 else S.SWA_FP32, order=c["order"],
                       bc=(w, w, w, w), cfl=_cfl(c), dry_tol=DRY)


def _cfl(c):
    return 0.5 if c.get("wetdry") else CFL


def _t_f(c):
    """The adjoint's final time: t_steps basin CFL steps, else a plain run's
    own steps, else the time waves take to cross most of the domain."""
    t_steps = c.get("t_steps", c["steps"])
    if c["kind"] == "scenario" and not c.get("solve"):
        t_steps = 3.5 * c["nx"] if c["ndim"] == 1 else 2000 * c["nx"] / 2048
    return max(t_steps, 20) * CFL * c["dx"] / math.sqrt(G * 4000.0)


def _adjoint_grid(c):
    """(nx, ny, dx) of the case's adjoint grid: adj_n columns over the domain."""
    n = c.get("adj_n", c["nx"])
    if n == c["nx"]:
        return c["nx"], c["ny"], c["dx"]
    dx = c["nx"] * c["dx"] / n
    return n, max(2, int(round(c["ny"] * c["dx"] / dx))), dx


def _make_adjoint(c, oc):
    nx, ny, dx = _adjoint_grid(c)
    x, y = _centres(nx, ny, dx)
    phi = torch.zeros((c["ndim"] + 1, nx * ny), dtype=torch.float64, device=DEV)
    phi[0] = oc.phi(x, y)
    adj = S.Adjoint(_desc(c, nx, ny, dx), _np(oc.bottom(x, y)), _np(phi), _t_f(c))
    store = S.SnapStore(adj, adj.info()[0] // c["every"] + 3,
                        S.SWA_FP64 if c["fp64"] else S.SWA_FP32)
    return adj, store, phi


# ------------------------------------------------------------ preparation
def prepare(case, seed):
    c, oc = case, Ocean(case, seed)
    S.load()
    if c["kind"] in ("patches", "amr"):
        return _prepare_patches(c, oc)
    x, y = _centres(c["nx"], c["ny"], c["dx"])
    B = oc.bottom(x, y)
    st = dict(c=c, q=oc.state(x, y, B), t_f=_t_f(c), t_s=0.32 * _t_f(c), tol=1e-3)
    n = c["nx"] * c["ny"]
    st["g"] = g = S.Grid(_desc(c), _np(B))
    if c.get("ctu"):
        g.set_scheme(S.SWA_SCHEME_CTU)
    if c.get("wetdry"):
        g.set_wetdry(True)
    if c.get("adj_n") or c["kind"] == "adjoint":
        st["adj"], st["store"], st["phi"] = _make_adjoint(c, oc)
        if c["kind"] != "adjoint" and not c.get("solve"):
            st["store"].run_adjoint(c["every"])
        passes = max(1, c["steps"] // FLAG_EVERY)
        st["flags"] = torch.zeros(n, dtype=torch.uint8, device=DEV)
        st["counts"] = torch.zeros(passes, dtype=torch.int64, device=DEV)
        if c["kind"] == "adjoint" or c.get("want_m"):
            st["m"] = torch.zeros(n, dtype=torch.float32, device=DEV)
    if c["kind"] != "scenario":
        g.set_state(*st["q"], c.get("at", 0.0) * st["t_f"])
    if oc.gauges:
        st["xy"] = torch.tensor(oc.gauges, dtype=torch.float64, device=DEV)
        st["series"] = torch.zeros((c["steps"], len(oc.gauges)), dtype=torch.float64,
                                   device=DEV)
    return st


def _layout(c):
    """Patch descriptors (level, x_lo, y_lo, nx, ny, dx, dy), the case's own."""
    L, dx = c["nx"] * c["dx"], c["dx"]
    if c["kind"] == "patches":
        r, out = random.Random(c["count"] * 1000 + c["side_hi"]), []
        for k in range(c["count"]):
            lev = 1 + k % c["levels"]
            nx, ny = r.randint(c["side_lo"], c["side_hi"]), r.randint(c["side_lo"], c["side_hi"])
            d = dx / c["ratio"] ** (lev - 1)
            out.append((lev, r.uniform(0, L - nx * d), r.uniform(0, L - ny * d), nx, ny, d, d))
        return out
    out, rt = [], c["ratio"]
    tiles, side, d, n = c["tiles"], c["side"], dx, c["nx"]
    cx, cy = int(0.35 * n), n // 2
    for lev in range(1, c["levels"] + 1):
        df = d / rt
        for b in range(tiles):
            for a in range(tiles):
                i, j = cx - tiles * side // 2 + a * side, cy - tiles * side // 2 + b * side
                out.append((lev, i * d - 2 * df, j * d - 2 * df, side * rt + 4, side * rt + 4,
                            df, df))
        cx, cy, d, tiles = cx * rt, cy * rt, df, max(1, tiles // 2)
    return out


def _patch_centres(descs):
    """Flat (x, y) of every patch's cells, patch by patch, and the offsets."""
    xs, ys, off = [], [], [0]
    for (_, x0, y0, nx, ny, dx, dy) in descs:
        x = x0 + (torch.arange(nx, dtype=torch.float64) + 0.5) * dx
        y = y0 + (torch.arange(ny, dtype=torch.float64) + 0.5) * dy
        xs.append(x.repeat(ny))
        ys.append(y.repeat_interleave(nx))
        off.append(off[-1] + nx * ny)
    return torch.cat(xs).to(DEV), torch.cat(ys).to(DEV), off


def _prepare_patches(c, oc):
    descs = _layout(c)
    x, y, off = _patch_centres(descs)
    B = oc.bottom(x, y)
    q = oc.state(x, y, B)
    st = dict(c=c, descs=descs, off=off, pq=[[f[a:b] for f in q] for a, b in zip(off, off[1:])])
    Bn = _np(B)
    common = _desc(c, fp64=False)
    st["ps"] = S.PatchSet(descs, [Bn[a:b] for a, b in zip(off, off[1:])], common)
    out = torch.empty((3, off[-1]), dtype=torch.float64, device=DEV)
    st["pout"], st["pslices"] = out, [[f[a:b] for f in out] for a, b in zip(off, off[1:])]
    if c["kind"] == "amr":
        x, y = _centres(c["nx"], c["ny"], c["dx"])
        Bc = oc.bottom(x, y)
        st["q"] = oc.state(x, y, Bc)
        st["g"] = S.Grid(_desc(c), _np(Bc))
        levels = list(range(1, c["levels"] + 1))
        st["amr"] = S.Amr(st["g"], st["ps"], levels, [c["ratio"]] * c["levels"])
        st["dt"] = 0.9 * CFL * c["dx"] / math.sqrt(G * float(-Bc.min()))
    return st


# -------------------------------------------------------------------- runs
def _state(g):
    """The grid's state arrays, in the precision it keeps them, as views of
    its workspace: (h, hu, hv) in FP64, (eta, hu, hv) in FP32."""
    dt, size = ((torch.float64, 8) if g.desc.precision == S.SWA_FP64 else (torch.float32, 4))
    base, out = g.ws.data_ptr(), []
    for p in S.swa_grid_arrays(g.h)[:g.desc.ndim + 1]:
        out.append(g.ws[p - base:p - base + g.n * size].view(dt))
    return out


def run(st):
    return {"scenario": _run_scenario, "adjoint": _run_adjoint, "flags": _run_flags,
            "patches": _run_patches, "amr": _run_amr}[st["c"]["kind"]](st)


def _flag(st, k=0):
    mode = S.SWA_FLAG_BRACKET if st["c"].get("bracket") else S.SWA_FLAG_INTERP
    S.swa_flag_cells(st["g"].h, st["store"].h, st["t_s"], st["t_f"], st["tol"], mode,
                     st["flags"], st.get("m"), st["counts"][k])


def _run_scenario(st):
    c, g = st["c"], st["g"]
    out = {}
    if c.get("solve"):
        S.swa_set_adjoint_state(st["adj"].h, st["phi"], S.SWA_DEVICE)
        S.swa_snapstore_clear(st["store"].h)
        st["store"].run_adjoint(c["every"])
        out["adjoint"] = torch.empty_like(st["phi"])
        S.swa_get_adjoint_state(st["adj"].h, out["adjoint"], S.SWA_DEVICE)
    g.set_state(*st["q"], 0.0)
    if "series" in st:
        S.swa_grid_record_gauges(g.h, st["xy"].shape[0], st["xy"], st["series"], None,
                                 c["steps"])
    if "store" in st:
        for k in range(c["steps"] // FLAG_EVERY):
            g.step(FLAG_EVERY, 1e300)
            _flag(st, k)
        out["flags"], out["counts"] = st["flags"], st["counts"]
    else:
        g.step(c["steps"], 1e300)
    out["state"] = _state(g)
    if "series" in st:   # the record is kept in the grid's own precision
        out["series"] = st["series"] if c["fp64"] else st["series"].float()
    return out


def _run_adjoint(st):
    adj, store = st["adj"], st["store"]
    S.swa_set_adjoint_state(adj.h, st["phi"], S.SWA_DEVICE)
    S.swa_snapstore_clear(store.h)
    store.run_adjoint(st["c"]["every"])
    q = torch.empty_like(st["phi"])
    S.swa_get_adjoint_state(adj.h, q, S.SWA_DEVICE)
    # the window of the whole run, [0, t_f]
    S.swa_flag_cells(st["g"].h, store.h, 0.0, st["t_f"], st["tol"], S.SWA_FLAG_INTERP,
                     st["flags"], st["m"], st["counts"])
    return {"adjoint": q if st["c"]["fp64"] else q.float(), "m": st["m"], "flags": st["flags"],
            "count": st["counts"]}


def _run_flags(st):
    _flag(st)
    out = {"flags": st["flags"], "count": st["counts"]}
    if "m" in st:
        out["m"] = st["m"]
    return out


def _set_patches(st):
    ps = st["ps"]
    for k, q in enumerate(st["pq"]):
        ps.set_state(k, *q)
    for lev in ps.levels:
        ps.start(lev, 0.0)


def _read_patches(st):
    for k, (eta, hu, hv) in enumerate(st["pslices"]):
        S.swa_patches_get_state(st["ps"].h, k, None, hu, hv, eta, S.SWA_DEVICE)
    return st["pout"].float()   # patches are FP32


def _run_patches(st):
    _set_patches(st)
    for lev in st["ps"].levels:
        st["ps"].step(lev, st["c"]["steps"])
    return {"patches": _read_patches(st)}


def _run_amr(st):
    st["g"].set_state(*st["q"], 0.0)
    _set_patches(st)
    t = 0.0
    for _ in range(st["c"]["steps"]):
        st["amr"].step(t, st["dt"])
        t = t + st["dt"]
    return {"state": _state(st["g"]), "patches": _read_patches(st)}


# -------------------------------------------------------------------- work
def work(case):
    """Bytes and operations of one pass.  A step of a grid reads its state and
    bottom once and writes its state once, and so does an adjoint step; a
    flag pass reads the state and bottom and writes a byte per cell; the
    state set is read in FP64 and stored.  Operations: those of the scheme
    per cell-update, counted in the source."""
    c = case
    esz = 8 if c["fp64"] else 4
    comp = c["ndim"] + 1
    n = c["nx"] * c["ny"]
    step_b = (2 * comp + 1) * esz
    ops = (320 if c["ndim"] == 2 else 160) if c["fp64"] else (218 if c["ndim"] == 2 else 110)
    if c.get("ctu"):
        ops *= 2
    set_b = comp * (8 + esz)
    b = f = 0.0
    if c["kind"] in ("patches", "amr"):
        ncoarse = 0
        counts = {}
        if c["kind"] == "patches":
            mean = 0.5 * (c["side_lo"] + c["side_hi"])
            cells, updates = c["count"] * mean * mean, c["count"] * mean * mean * c["steps"]
        else:
            ncoarse, cells, updates, sub = n, 0, 0, 1
            for (lev, _, _, px, py, _, _) in _layout(c):
                counts[lev] = counts.get(lev, 0) + px * py
            for lev in sorted(counts):
                sub *= c["ratio"]
                cells += counts[lev]
                updates += counts[lev] * sub * c["steps"]
            updates += n * c["steps"]
        b = (cells + ncoarse) * (set_b + 12) + updates * step_b
        return {"bytes": b, "flops": updates * ops}
    if c["kind"] == "adjoint" or c.get("solve"):
        nx, ny, dx = _adjoint_grid(c)
        na = nx * ny
        steps = _t_f(c) * math.sqrt(G * 4000.0) / dx / CFL
        b += na * (steps * step_b + steps / c["every"] * comp * esz + 2 * comp * 8)
        f += na * steps * 210
    if c["kind"] != "scenario":
        snaps = 1 if c["kind"] == "flags" else _t_f(c) * math.sqrt(G * 4000.0) / c["dx"] / CFL / c["every"]
        reads = snaps if (c["kind"] == "adjoint" or c.get("want_m")) else 0
        return {"bytes": b + n * (4 * esz + 2 + reads * comp * esz), "flops": f + n * 6}
    b += n * (set_b + c["steps"] * step_b)
    if c.get("adj_n"):
        b += n * (comp * esz + esz + 1) * (c["steps"] // FLAG_EVERY)
    return {"bytes": b, "flops": f + n * c["steps"] * ops}


# ------------------------------------------------- the same in 64 bits, plain
def _mirror(n, wall):
    """Indices of cells -2 .. n + 1 (copied or mirrored) and the sign of their
    normal momentum."""
    i = torch.arange(-2, n + 2, device=DEV)
    s = torch.ones(n + 4, dtype=torch.float64, device=DEV)
    if wall:
        s = torch.where((i < 0) | (i >= n), -1.0, s)
        i = torch.where(i < 0, -1 - i, torch.where(i >= n, 2 * n - 1 - i, i))
    return i.clamp(0, n - 1), s


def _roe(h, mn, mt, eta):
    """Waves [(speed, Z)] of the edges between neighbours along the last axis,
    and (u, v, c) of their Roe states."""
    a, b = slice(None, -1), slice(1, None)
    un, ut, sq = mn / h, mt / h, h.sqrt()
    hb = 0.5 * (h[..., a] + h[..., b])
    den = sq[..., a] + sq[..., b]
    u = (sq[..., a] * un[..., a] + sq[..., b] * un[..., b]) / den
    v = (sq[..., a] * ut[..., a] + sq[..., b] * ut[..., b]) / den
    ch = (G * hb).sqrt()
    s1, s3 = u - ch, u + ch
    d1 = mn[..., b] - mn[..., a]
    d2 = mn[..., b] * un[..., b] - mn[..., a] * un[..., a] + G * hb * (eta[..., b] - eta[..., a])
    d3 = mn[..., b] * ut[..., b] - mn[..., a] * ut[..., a]
    b1, b3 = (s3 * d1 - d2) / (2 * ch), (d2 - s1 * d1) / (2 * ch)
    z = torch.zeros_like(b1)
    return [(s1, (b1, b1 * s1, b1 * v)), (u, (z, z, d3 - v * d1)),
            (s3, (b3, b3 * s3, b3 * v))], (u, v, ch)


def _split(waves, nu, order):
    """Of the inner edges: fluctuations to the left and right and the limited
    correction, three components each."""
    m = slice(1, -1)
    left, right, F = ([0.0] * 3 for _ in range(3))
    for s, Z in waves:
        sm = s[..., m]
        wr = torch.where(sm > 0, 1.0, torch.where(sm < 0, 0.0, 0.5))
        zm = [z[..., m] for z in Z]
        zz = sum(z * z for z in zm)
        up = [torch.where(sm > 0, z[..., :-2], z[..., 2:]) for z in Z]
        th = torch.where(zz != 0, sum(p * q for p, q in zip(up, zm)) / torch.where(zz != 0, zz, 1.0), 0.0)
        phi = torch.minimum(torch.minimum(0.5 * (1 + th), 2 * th), torch.full_like(th, 2.0)).clamp_(min=0)
        k = 0.5 * torch.sign(sm) * (1 - nu * sm.abs()) * phi if order == 2 else 0.0 * sm
        for j in range(3):
            left[j] = left[j] + (1 - wr) * zm[j]
            right[j] = right[j] + wr * zm[j]
            F[j] = F[j] + k * zm[j]
    return left, right, F


def _shore(h, mn, mt, eta, B, edge, left, right):
    """Replaces the fluctuations of the marked edges by the hydrostatic
    reconstruction with an HLL flux."""
    a, b = slice(1, -2), slice(2, -1)
    Bm = torch.maximum(B[..., a], B[..., b])
    side = []
    for k in (a, b):
        wet = h[..., k] > DRY
        u = torch.where(wet, mn[..., k] / h[..., k], 0.0)
        v = torch.where(wet, mt[..., k] / h[..., k], 0.0)
        hs = (eta[..., k] - Bm).clamp(min=0)
        ps, p = 0.5 * G * hs * hs, 0.5 * G * h[..., k] ** 2
        side.append(dict(u=u, c=(G * hs).sqrt(), Q=(hs, hs * u, hs * v), S=p - ps,
                         F=(hs * u, hs * u * u + ps, hs * u * v),
                         f=(mn[..., k], mn[..., k] * u + p, mn[..., k] * v)))
    A, D = side
    sl = torch.minimum(A["u"] - A["c"], D["u"] - D["c"])
    sr = torch.maximum(A["u"] + A["c"], D["u"] + D["c"])
    any_wet = (A["Q"][0] > 0) | (D["Q"][0] > 0)
    for j in range(3):
        mid = (sr * A["F"][j] - sl * D["F"][j] + sl * sr * (D["Q"][j] - A["Q"][j])) / torch.where(sr > sl, sr - sl, 1.0)
        F = torch.where(sl >= 0, A["F"][j], torch.where(sr <= 0, D["F"][j], mid))
        F = torch.where(any_wet, F, 0.0)
        left[j] = torch.where(edge, F + (A["S"] if j == 1 else 0) - A["f"][j], left[j])
        right[j] = torch.where(edge, D["f"][j] - F - (D["S"] if j == 1 else 0), right[j])


def _sweep(h, mn, mt, B, nu, order, wetdry):
    """One sweep along the last axis of arrays with two ghost cells each side."""
    eta = h + B
    if wetdry:
        dry = h <= DRY
        hs = torch.where(dry, 1.0, h)
        u, ch = torch.where(dry, 0.0, mn / hs), (G * hs).sqrt()
        a, b = slice(None, -1), slice(1, None)
        edge = (dry[..., a] | dry[..., b]
                | ((u - ch)[..., a] < 0) & ((u - ch)[..., b] > 0)
                | ((u + ch)[..., a] < 0) & ((u + ch)[..., b] > 0))
        waves, _ = _roe(hs, torch.where(dry, 0.0, mn), torch.where(dry, 0.0, mt), eta)
        waves = [(torch.where(edge, 0.0, s), tuple(torch.where(edge, 0.0, z) for z in Z)) for s, Z in waves]
    else:
        waves, _ = _roe(h, mn, mt, eta)
    left, right, F = _split(waves, nu, order)
    if wetdry:
        _shore(h, mn, mt, eta, B, edge[..., 1:-1], left, right)
        F = [torch.where(edge[..., 1:-1], 0.0, f) for f in F]
    i = slice(2, -2)
    out = [q[..., i] - nu * (right[j][..., :-1] + left[j][..., 1:]) - nu * (F[j][..., 1:] - F[j][..., :-1])
           for j, q in enumerate((h, mn, mt))]
    if wetdry:
        dry = ~(out[0] > DRY)
        out = [out[0].clamp(min=0), torch.where(dry, 0.0, out[1]), torch.where(dry, 0.0, out[2])]
    return out


def _ctu(h, hu, hv, B, nux, nuy, order, walls):
    """One unsplit step with transverse waves of a (ny, nx) grid."""
    ny, nx = h.shape
    ix, sx = _mirror(nx, walls)
    iy, sy = _mirror(ny, walls)
    pad = lambda q: q[iy][:, ix]
    P, U, V, E = pad(h), pad(hu) * sx, pad(hv) * sy[:, None], pad(h + B)
    T = lambda q: q.transpose(0, 1)

    def direction(h, mn, mt, eta, nu):
        waves, (u, v, c) = _roe(h, mn, mt, eta)
        lr = _split(waves, nu, order)
        full = [[0.0] * 3, [0.0] * 3]
        for s, Z in waves:
            wr = torch.where(s > 0, 1.0, torch.where(s < 0, 0.0, 0.5))
            for j in range(3):
                full[0][j] = full[0][j] + (1 - wr) * Z[j]
                full[1][j] = full[1][j] + wr * Z[j]

        def trans(a):
            beta = (((v + c) * a[0] - a[2]) / (2 * c), a[1] - u * a[0], (a[2] - (v - c) * a[0]) / (2 * c))
            vec = ((1.0, u, v - c), (0.0, 1.0, 0.0), (1.0, u, v + c))
            dn, up = [0.0] * 3, [0.0] * 3
            for s, b, r in zip((v - c, v, v + c), beta, vec):
                for j in range(3):
                    dn[j] = dn[j] + torch.clamp(s, max=0) * b * r[j]
                    up[j] = up[j] + torch.clamp(s, min=0) * b * r[j]
            return dn, up
        (ldn, lup), (rdn, rup) = trans(full[0]), trans(full[1])
        # per cell (without the outermost): its low edge's right-going and its
        # high edge's left-going fluctuation, in the other direction's frame
        o = (0, 2, 1)
        up = [rup[k][..., :-1] + lup[k][..., 1:] for k in o]
        dn = [rdn[k][..., :-1] + ldn[k][..., 1:] for k in o]
        return lr, up, dn

    (xl, xr, xF), yup, ydn = direction(P, U, V, E, nux)
    (yl, yr, yF), xup, xdn = direction(T(P), T(V), T(U), T(E), nuy)
    out = []
    comp = (0, 2, 1)
    for j in range(3):
        # x-edges of the interior rows; xup, xdn are (x, y) with y inner cells
        tx = lambda q: T(q)[2 - 1:-1, :]                      # rows 2 .. ny + 1 of the padded grid
        Fx = xF[j][2:-2] - 0.5 * nuy * (tx(xup[j])[:, 1:-2] + tx(xdn[j])[:, 2:-1])
        dq = -nux * (xr[j][2:-2][:, :-1] + xl[j][2:-2][:, 1:]) - nux * (Fx[:, 1:] - Fx[:, :-1])
        k = comp[j]
        yu, yd = yup[k][:, 1:-1], ydn[k][:, 1:-1]             # columns 2 .. nx + 1
        Fy = T(yF[k])[:, 2:-2] - 0.5 * nux * (yu[1:-2] + yd[2:-1])
        dq = dq - nuy * (T(yr[k])[:-1, 2:-2] + T(yl[k])[1:, 2:-2]) - nuy * (Fy[1:] - Fy[:-1])
        out.append((h, hu, hv)[j] + dq)
    return out


def _smax(h, hu, hv, dx, dy, wetdry):
    hs = torch.where(h > DRY, h, 1.0) if wetdry else h
    c = (G * hs).sqrt()
    s = (hu.abs() / hs + c) / dx
    if dy:
        s = torch.maximum(s, (hv.abs() / hs + c) / dy)
    return float((torch.where(h > DRY, s, 0.0) if wetdry else s).max())


def _gauge(eta, c, xy):
    """Bilinear eta at the gauges, clamped to the outermost cell centres."""
    row = []
    for (x, y) in xy:
        fx = min(max(x / c["dx"] - 0.5, 0.0), c["nx"] - 1.0)
        i = min(int(fx), c["nx"] - 2)
        ax = fx - i
        if c["ndim"] == 1:
            row.append((1 - ax) * eta[0, i] + ax * eta[0, i + 1])
            continue
        fy = min(max(y / c["dx"] - 0.5, 0.0), c["ny"] - 1.0)
        j = min(int(fy), c["ny"] - 2)
        ay = fy - j
        row.append((1 - ay) * ((1 - ax) * eta[j, i] + ax * eta[j, i + 1])
                   + ay * ((1 - ax) * eta[j + 1, i] + ax * eta[j + 1, i + 1]))
    return torch.stack(row)


def _forward(c, oc):
    """The state after the case's steps and the gauge series, in 64 bits."""
    nx, ny, dx = c["nx"], c["ny"], c["dx"]
    x, y = _centres(nx, ny, dx)
    B = oc.bottom(x, y)
    eta, hu, hv = (q.view(ny, nx) for q in oc.state(x, y, B))
    B = B.view(ny, nx)
    h = eta - B
    two_d, wd = c["ndim"] == 2, bool(c.get("wetdry"))
    ix, sx = _mirror(nx, c["walls"])
    iy, sy = _mirror(ny, c["walls"])
    BX, BY = B[:, ix], B[iy].T
    series = []
    for _ in range(c["steps"]):
        if oc.gauges:
            series.append(_gauge(h + B, c, oc.gauges))
        dt = _cfl(c) / _smax(h, hu, hv, dx, dx if two_d else 0.0, wd)
        nu = dt / dx
        if c.get("ctu"):
            h, hu, hv = _ctu(h, hu, hv, B, nu, nu, c["order"], c["walls"])
            continue
        h, hu, hv = _sweep(h[:, ix], hu[:, ix] * sx, hv[:, ix], BX, nu, c["order"], wd)
        if two_d:
            ht, hvt, hut = _sweep(h[iy].T, (hv[iy] * sy[:, None]).T, hu[iy].T, BY, nu, c["order"], wd)
            h, hu, hv = ht.T, hut.T, hvt.T
    state = [(h if c["fp64"] else h + B).reshape(-1), hu.reshape(-1), hv.reshape(-1)]
    return state[:c["ndim"] + 1], torch.stack(series) if series else None


def _adjoint_sweep(e, m, ch, nu, order):
    """One adjoint sweep along the last axis (two ghost cells each side; no
    cell is dry)."""
    a, b = slice(None, -1), slice(1, None)
    gh = ch * ch
    d1, d2 = gh[..., a] * m[..., a] - gh[..., b] * m[..., b], e[..., a] - e[..., b]
    cl, cr = ch[..., a], ch[..., b]
    b1, b2 = (d1 + cr * d2) / (cl + cr), (cl * d2 - d1) / (cl + cr)
    i = slice(1, -1)
    F = [0.0, 0.0]
    if order == 2:
        def part(bb, cc, sign, up):
            Z = (bb[..., i] * cc[..., i] * sign, bb[..., i])
            U = (bb[..., up] * cc[..., up] * sign, bb[..., up])
            zz = Z[0] * Z[0] + Z[1] * Z[1]
            th = torch.where(zz != 0, (U[0] * Z[0] + U[1] * Z[1]) / torch.where(zz != 0, zz, 1.0), 0.0)
            phi = torch.minimum(torch.minimum(0.5 * (1 + th), 2 * th), torch.full_like(th, 2.0)).clamp_(min=0)
            k = -0.5 * sign * (1 - nu * cc[..., i]) * phi
            return k * Z[0], k * Z[1]
        p, q = part(b1, cl, 1.0, slice(2, None)), part(b2, cr, -1.0, slice(None, -2))
        F = [p[0] + q[0], p[1] + q[1]]
    left = [b1[..., i] * cl[..., i] + F[0], b1[..., i] + F[1]]
    right = [-b2[..., i] * cr[..., i] - F[0], b2[..., i] - F[1]]
    j = slice(2, -2)
    return [q[..., j] - nu * (right[k][..., :-1] + left[k][..., 1:]) for k, q in enumerate((e, m))]


def _backward(c, oc, q=None):
    """The adjoint state at the end of its solve, and max |q^ . q| over its
    snapshots for the forward state q."""
    nx, ny, dx = _adjoint_grid(c)
    x, y = _centres(nx, ny, dx)
    ch = (G * -oc.bottom(x, y)).sqrt().view(ny, nx)
    e = oc.phi(x, y).view(ny, nx)
    mu, ga = torch.zeros_like(e), torch.zeros_like(e)
    N = max(1, math.ceil(_t_f(c) * float((ch / dx).max()) / _cfl(c)))
    nu = _t_f(c) / N / dx
    ix, sx = _mirror(nx, c["walls"])
    iy, sy = _mirror(ny, c["walls"])
    CX, CY = ch[:, ix], ch[iy].T.contiguous()
    best = None
    for k in range(N + 1):
        if q is not None and (k % c["every"] == 0 or k == N):
            d = (e * q[0] + mu * q[1] + ga * q[2]).abs()
            best = d if best is None else torch.maximum(best, d)
        if k == N:
            break
        if c["ndim"] == 2:
            et, gt = _adjoint_sweep(e[iy].T, (ga[iy] * sy[:, None]).T, CY, nu, c["order"])
            e, ga = et.T, gt.T
        e, mu = _adjoint_sweep(e[:, ix], mu[:, ix] * sx, CX, nu, c["order"])
    out = torch.stack([v.reshape(-1) for v in (e, mu, ga)[:c["ndim"] + 1]])
    return out, None if best is None else best.reshape(-1)


def _patches(c, oc):
    """Every patch after its level's steps: each cell's stencils gathered from
    the flat arrays of all patches."""
    descs = _layout(c)
    x, y, off = _patch_centres(descs)
    B = oc.bottom(x, y)
    eta, hu, hv = oc.state(x, y, B)
    out = torch.empty((3, off[-1]), dtype=torch.float64, device=DEV)
    for lev in sorted({d[0] for d in descs}):
        cells, sx, sy, n = [], [], [], 0
        for k, (l, _, _, nx, ny, dx, _) in enumerate(descs):
            if l != lev:
                continue
            ix, _ = _mirror(nx, False)
            iy, _ = _mirror(ny, False)
            i, j = torch.arange(nx, device=DEV), torch.arange(ny, device=DEV)
            w = torch.arange(5, device=DEV)
            sx.append((n + j[:, None, None] * nx + ix[i[:, None] + w][None]).reshape(-1, 5))
            sy.append((n + iy[j[:, None] + w][:, None] * nx + i[None, :, None]).reshape(-1, 5))
            cells.append(torch.arange(off[k], off[k + 1], device=DEV))
            n, d = n + nx * ny, dx
        cells, sx, sy = torch.cat(cells), torch.cat(sx), torch.cat(sy)
        b = B[cells]
        h, u, v = (eta - B)[cells], hu[cells], hv[cells]
        bx, by = b[sx], b[sy]
        for _ in range(c["steps"]):
            nu = CFL / _smax(h, u, v, d, d, False) / d
            h, u, v = (q[:, 0] for q in _sweep(h[sx], u[sx], v[sx], bx, nu, c["order"], False))
            h, v, u = (q[:, 0] for q in _sweep(h[sy], v[sy], u[sy], by, nu, c["order"], False))
        out[0, cells], out[1, cells], out[2, cells] = h + b, u, v
    return out


def exact(case, seed):
    """What run() returns, in 64 bits with plain torch: the states, gauges and
    m.  Flags are bytes and counts; the refinement hierarchy's glue (fills,
    subcycling, refluxing) has no short plain form."""
    c, oc = case, Ocean(case, seed)
    if c["kind"] == "amr" or (c["kind"] == "flags"):
        return None
    if c["kind"] == "patches":
        return {"patches": _patches(c, oc)}
    if c["kind"] == "adjoint":
        x, y = _centres(c["nx"], c["ny"], c["dx"])
        q = [v.view(c["ny"], c["nx"]) for v in oc.state(x, y, oc.bottom(x, y))]
        a, m = _backward(c, oc, q)
        return {"adjoint": a, "m": m, "flags": None, "count": None}
    out = {}
    if c.get("solve"):
        out["adjoint"] = _backward(c, oc)[0]
    if c.get("adj_n"):
        out["flags"] = out["counts"] = None
    out["state"], series = _forward(c, oc)
    if series is not None:
        out["series"] = series
    return out
