"""The workloads this library is timed on, through its public entry points.

A case is a dict of plain values.  Kinds:

  solve   one 2D phase-space solve: upload of the initial f, a number of time
          steps with the remaps that fall into them, and the reads of f and
          of the last remap's f_ini (FP64 solves also read the pixel masses
          and the force); with "emap" > 0 the E_map criterion may remap sooner
  batch   many independent uneven solves advanced together for one remap cycle
  init    a new initial condition: upload, spline coefficients, element reset
  solve4d the 4D phase-space solve, as "solve"

Every pass starts again from the initial f, so that passes on one state do
the same work and give the same outputs.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1705_03750_gb300 import inputs as I
from paper_1705_03750_gb300 import inputs4d as I4
from paper_1705_03750_gb300 import vlamet as V
from paper_1705_03750_gb300 import vlamet4d as V4


def _solve(name, nx, nv, prec, steps, n_s, ic="halos", dt=0.002, emap=0.0):
    c = {"kind": "solve", "nx": nx, "nv": nv, "s": 4 if max(nx, nv) <= 128 else 8, "precision": prec, "steps": steps,
         "n_s": n_s, "ic": ic, "dt": dt, "emap": emap}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the paper's first test, a 128 x 128 isothermal sheet in FP64: the
        # smallest grid in use, a cycle of 20 short steps and its remap
        _solve("sheet_128_f64", 128, 128, "f64", 20, 20, ic="sheet", dt=0.005),
        # a small ragged grid with odd sides in FP64
        _solve("halos_301x217_f64", 301, 217, "f64", 20, 20),
        # a typical served request: 512 x 512, FP32-mixed, one remap cycle
        _solve("halos_512_f32", 512, 512, "f32", 25, 25),
        # an ordinary solve whose sides are odd and differ
        _solve("halos_1531x997_f32", 1531, 997, "f32", 25, 25),
        # a remap cycle of the benchmark's configuration, in both precisions
        _solve("halos_4096_f32", 4096, 4096, "f32", 25, 25),
        _solve("halos_4096_f64", 4096, 4096, "f64", 25, 25),
        # the largest configured 2D grid
        _solve("halos_8192_f32", 8192, 8192, "f32", 25, 25),
        # a served request with coarse x under fine v, which the E_map
        # criterion remaps every few steps
        _solve("emap_576x2048_f32", 576, 2048, "f32", 25, 25, emap=0.5),
        # many uneven solves in one group (sides 64 ... 512), one remap cycle
        {"name": "batch_48_f32", "kind": "batch", "solves": 48, "side_lo": 64, "side_hi": 512, "precision": "f32",
         "n_s": 20, "emap": 0.5},
        # a new initial condition on the benchmark's grid
        {"name": "init_4096_f64", "kind": "init", "nx": 4096, "nv": 4096, "s": 8, "precision": "f64"},
        # 4D phase space: a small ragged grid, and the configured 64^4 workload
        {"name": "phase4d_20x24x22x18", "kind": "solve4d", "n0": 20, "n1": 24, "n2": 22, "n3": 18, "s": 4,
         "steps": 10, "n_s": 10},
        {"name": "phase4d_64", "kind": "solve4d", "n0": 64, "n1": 64, "n2": 64, "n3": 64, "s": 4, "steps": 10,
         "n_s": 10},
    ]


def _side(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "solve", "batch", "init", "solve4d"])
    if kind == "solve":
        prec = rng.choice(["f32", "f32", "f64"])
        nx = _side(rng, 96, 4096)
        nv = min(4096, max(96, int(round(nx * math.exp(rng.uniform(-1.2, 1.2))))))
        small = max(nx, nv) <= 128
        # grids much finer in v than in x are run with the E_map criterion
        emap = 0.5 if nv > 1.5 * nx else 0.0
        return _solve(None, nx, nv, prec, rng.choice([20, 25]), rng.choice([20, 25]),
                      ic=rng.choice(["halos", "halos", "sheet"]), dt=0.005 if small else 0.002, emap=emap)
    if kind == "batch":
        return {"kind": "batch", "solves": rng.randint(8, 48), "side_lo": 64, "side_hi": rng.randint(200, 700),
                "precision": rng.choice(["f32", "f32", "f64"]), "n_s": 20, "emap": 0.5}
    if kind == "init":
        return {"kind": "init", "nx": _side(rng, 96, 4096), "nv": _side(rng, 96, 4096), "s": 8,
                "precision": rng.choice(["f32", "f64"])}
    n = _side(rng, 14, 48)
    n0, n1, n2, n3 = (max(12, n + rng.randint(-3, 3)) for _ in range(4))
    return {"kind": "solve4d", "n0": n0, "n1": n1, "n2": n2, "n3": n3, "s": 4, "steps": 10, "n_s": 10}


# ---- inputs --------------------------------------------------------------

def _axis(lo, hi, n):
    return torch.linspace(lo, hi, n, dtype=torch.float64, device="cuda")


def _halos_f(h, x, v):
    f = torch.zeros(x.numel(), v.numel(), dtype=torch.float64, device=x.device)
    for k in range(h.m.size):
        gx = h.m[k] / (2.0 * math.pi * h.sx[k] * h.sv[k]) * torch.exp(-0.5 * ((x - h.xc[k]) / h.sx[k]) ** 2)
        f.addr_(gx, torch.exp(-0.5 * ((v - h.vc[k]) / h.sv[k]) ** 2))
    return f


def _sheet_f(sigma, x, v):
    x0 = sigma * sigma / math.pi
    amp = 1.0 / (2.0 * x0) / (math.sqrt(2.0 * math.pi) * sigma)
    return amp * torch.outer(torch.cosh(x / x0) ** -2, torch.exp(-0.5 * (v / sigma) ** 2))


def _config(nx, nv, s, prec, dt, n_s, v_hi=1.5, emap=0.0):
    p = V.VM_FP32_MIXED if prec == "f32" else V.VM_FP64
    return V.Config(nx, nv, -1.0, 1.0, -v_hi, v_hi, s, dt, n_s, 1.0, p, emap_remap=emap)


def _solver(cfg, f0, force):
    """A solver, its device f0 and the buffers its results are read into."""
    t = torch.float32 if cfg.precision == V.VM_FP32_MIXED else torch.float64
    d = {"solver": V.Solver(cfg), "f0": f0, "dtype": np.float32 if t == torch.float32 else np.float64,
         "f": torch.empty(cfg.nx, cfg.nv, dtype=t, device="cuda"),
         "fini": torch.empty(cfg.nx, cfg.nv, dtype=t, device="cuda")}
    d["force"] = {k: torch.empty(cfg.nx, dtype=torch.float64, device="cuda") for k in ("M", "a", "da", "d2a")} \
        if force else None
    return d


def _prepare_solve(c, seed):
    sheet = c["ic"] == "sheet"
    # the sheet's dispersion and box, or the halos, are the seed's
    sigma = float(np.random.default_rng(seed).uniform(0.3, 0.7)) if sheet else 0.0
    v_hi = 5.0 * sigma if sheet else 1.5
    cfg = _config(c["nx"], c["nv"], c["s"], c["precision"], c["dt"], c["n_s"], v_hi, c["emap"])
    x, v = _axis(-1.0, 1.0, c["nx"]), _axis(-v_hi, v_hi, c["nv"])
    f0 = _sheet_f(sigma, x, v) if sheet else _halos_f(I.draw_halos(seed, 16), x, v)
    return _solver(cfg, f0, c["precision"] == "f64")


def _members(c, seed):
    """Sides and kind of each solve of a batch (the case's own), and the
    sheets' dispersions and the halos' numbers (the seed's)."""
    r = np.random.default_rng([c["solves"], c["side_lo"], c["side_hi"]])
    sides = np.exp(r.uniform(math.log(c["side_lo"]), math.log(c["side_hi"]), (c["solves"], 2))).round().astype(int)
    sheet = r.uniform(size=c["solves"]) < 0.5
    r = np.random.default_rng(seed)
    return sides, sheet, r.uniform(0.3, 0.7, c["solves"]), r.integers(4, 17, c["solves"])


def _prepare_batch(c, seed):
    sides, sheet, sigma, nh = _members(c, seed)
    parts = []
    for q in range(c["solves"]):
        nx, nv = int(sides[q, 0]), int(sides[q, 1])
        v_hi = 5.0 * float(sigma[q]) if sheet[q] else 1.5
        x, v = _axis(-1.0, 1.0, nx), _axis(-v_hi, v_hi, nv)
        f0 = _sheet_f(float(sigma[q]), x, v) if sheet[q] else _halos_f(I.draw_halos(seed * 1000 + q, int(nh[q])), x, v)
        cfg = _config(nx, nv, 4 if max(nx, nv) <= 128 else 8, c["precision"], 0.005 if sheet[q] else 0.002, c["n_s"],
                      v_hi, c["emap"])
        p = _solver(cfg, f0, False)
        p["solver"].set_f(f0)
        parts.append(p)
    return {"parts": parts, "batch": V.Batch([p["solver"] for p in parts])}


def _prepare_init(c, seed):
    cfg = _config(c["nx"], c["nv"], c["s"], c["precision"], 0.002, 25)
    f0 = _halos_f(I.draw_halos(seed, 16), _axis(-1.0, 1.0, c["nx"]), _axis(-1.5, 1.5, c["nv"]))
    return _solver(cfg, f0, False)


def _prepare_4d(c, seed):
    n = (c["n0"], c["n1"], c["n2"], c["n3"])
    rc = I4.HALOS4D_64.with_(n=n, s=c["s"], n_s=c["n_s"], seed=seed)
    h = I4.draw_halos4d(seed, rc.halos)
    ax = [_axis(rc.lo[a], rc.hi[a], n[a]) for a in range(4)]
    f0 = torch.zeros(n, dtype=torch.float64, device="cuda")
    for k in range(rc.halos):
        ex, ey = (torch.exp(-0.5 * ((ax[a] - h["cx"][k, a]) / h["sx"][k]) ** 2) for a in range(2))
        eu, ew = (torch.exp(-0.5 * ((ax[2 + a] - h["cv"][k, a]) / h["sv"][k]) ** 2) for a in range(2))
        amp = h["m"][k] / ((2.0 * math.pi) ** 2 * h["sx"][k] ** 2 * h["sv"][k] ** 2)
        f0 += amp * torch.einsum("ij,kl->ijkl", torch.outer(ex, ey), torch.outer(eu, ew))
    return {"solver": V4.Solver4D(V4.config(rc)), "f0": f0, "f": torch.empty_like(f0), "fini": torch.empty_like(f0)}


def prepare(case, seed):
    kind = case["kind"]
    fn = {"solve": _prepare_solve, "batch": _prepare_batch, "init": _prepare_init, "solve4d": _prepare_4d}[kind]
    return dict(fn(case, seed), case=case)


# ---- one pass ------------------------------------------------------------

def _run_solve(st):
    s, c = st["solver"], st["case"]
    s.set_f(st["f0"])
    s.step(c["steps"])
    out = {"f": s.read_f(st["dtype"], out=st["f"]), "fini": s.read_fini(st["dtype"], out=st["fini"])}
    if st["force"] is not None:
        out.update(s.density_force(st["force"]))
    return out


def _run_batch(st):
    for p in st["parts"]:
        p["solver"].set_f(p["f0"])
    st["batch"].step(st["case"]["n_s"])
    # one result per solve: f of the last step
    return {"f%02d" % q: p["solver"].read_f(p["dtype"], out=p["f"]) for q, p in enumerate(st["parts"])}


def _run_init(st):
    s = st["solver"]
    s.set_f(st["f0"])
    return {"f": s.read_f(st["dtype"], out=st["f"]), "eta": s.read_eta(st["dtype"], out=st["fini"])}


def _run_4d(st):
    s = st["solver"]
    s.set_f(st["f0"])
    s.step(st["case"]["steps"])
    return {"f": s.read_f(out=st["f"]), "fini": s.read_fini(out=st["fini"])}


def run(state):
    return {"solve": _run_solve, "batch": _run_batch, "init": _run_init, "solve4d": _run_4d}[state["case"]["kind"]](state)


# ---- what a pass cannot do without ---------------------------------------

def _work_2d(nx, nv, s, steps, n_s, b):
    n, ne = nx * nv, (nx / s + 3) * (nv / s + 3)
    remaps = steps // n_s
    # upload and coefficients; per step the read of f_ini, the write of f and
    # the elements; per remap the read of eta, the writes of f_ini and eta
    byts = n * (8 + 3 * b) + steps * (2 * b * n + 2 * 96 * ne) + remaps * (3 * b * n + 96 * ne) + 2 * b * n
    # per site the inverse map (30) and the six-point value (25); per remap
    # the blend over five elements (200) and the spline (60), twice two sweeps
    return byts, n * (steps * 55.0 + remaps * 280.0 + 20.0)


def work(case):
    kind = case["kind"]
    b = 4 if case.get("precision") == "f32" else 8
    if kind == "solve":
        by, fl = _work_2d(case["nx"], case["nv"], case["s"], case["steps"], case["n_s"], b)
    elif kind == "batch":
        # the mean member: sides log-uniform
        r = math.log(case["side_hi"] / case["side_lo"])
        side = (case["side_hi"] - case["side_lo"]) / r
        by, fl = (case["solves"] * w for w in _work_2d(side, side, 8, case["n_s"], case["n_s"], b))
    elif kind == "init":
        n = case["nx"] * case["nv"]
        by, fl = n * (8 + 4 * b), n * 20.0
    else:
        n = case["n0"] * case["n1"] * case["n2"] * case["n3"]
        ne = math.prod(case["n%d" % a] / case["s"] + 3 for a in range(4))
        st, rm = case["steps"], case["steps"] // case["n_s"]
        by = n * 32 + st * (16 * n + 960 * ne) + rm * (24 * n + 480 * ne)
        fl = n * (st * 305.0 + rm * 1500.0)
    return {"bytes": float(by), "flops": float(fl)}


# ---- the same in 64 bits, without this library ----------------------------

def _spline_lines(a):
    """Coefficients of the cubic B-spline through the columns' values with
    zero slope at both ends: (1, 4, 1)/6 rows, (4, 2)/6 and (2, 4)/6 at the ends."""
    n = a.shape[0]
    y, cp = np.empty_like(a), np.empty(n)
    for i in range(n):
        sub = 0.0 if i == 0 else (2.0 if i == n - 1 else 1.0)
        sup = 0.0 if i == n - 1 else (2.0 if i == 0 else 1.0)
        den = 4.0 - (sub * cp[i - 1] if i else 0.0)
        cp[i] = sup / den
        y[i] = (6.0 * a[i] - (sub * y[i - 1] if i else 0.0)) / den
    for i in range(n - 2, -1, -1):
        y[i] -= cp[i] * y[i + 1]
    return y


def exact(case, seed):
    if case["kind"] != "init":
        return None  # the influence map of a whole solve has no short form in plain torch or numpy
    f0 = _halos_f(I.draw_halos(seed, 16), _axis(-1.0, 1.0, case["nx"]), _axis(-1.5, 1.5, case["nv"])).cpu().numpy()
    eta = _spline_lines(np.ascontiguousarray(_spline_lines(np.ascontiguousarray(f0.T)).T))
    return {"f": f0, "eta": eta}
