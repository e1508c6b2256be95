"""The work a program has this package do, as cases that can be timed and compared.

A case names one pass through the public entry points: a whole uncertainty-quantification call on host
buffers (``run_uq_host``), a batch of lattice-Boltzmann runs on device buffers (``run_batch``, periodic
or channel), or one of the statistics layers on fields that are already on the device (``project``,
``stats``, ``w1_speed``).  Sizes are those of ``workloads.py``, ``bench.py`` and the tests, with shorter
time loops where a full one would take longer than a second or two.

The lattices' initial fields come from the uncertain inputs; ``prepare`` draws the bounds of those inputs
(or the Monte Carlo seed) from the seed.  ``exact`` restates the method in FP64 with plain torch and numpy.
"""
from __future__ import annotations

import math
import random
from dataclasses import replace

import numpy as np
import torch

from paper_2508_13867_gb300 import ensemble, workloads
from paper_2508_13867_gb300 import uqlb as U

DEV = "cuda:0"


def listed() -> list[dict]:
    return [
        # the benchmark's workload end to end: 5^4 collocation samples of the 4-D Taylor-Green set-up
        # through one C call with host outputs (Algorithm 1)
        dict(name="uq_gpc4d_256", kind="uq", nx=256, ny=256, steps=2000, dim=4, pts=5, order=4, storage="f32"),
        # the plain small case: one uncertain viscosity, 5 samples of 64 x 64 in FP64; latency and launches
        dict(name="uq_gpc1d_64_f64", kind="uq", nx=64, ny=64, steps=1000, dim=1, pts=5, order=4, storage="f64"),
        # a block of the 512 x 512 Monte Carlo ensemble: runs, fields on the device, mean and variance
        dict(name="mc4d_512", kind="tgv", nx=512, ny=512, steps=400, samples=96, storage="f32", stats=True, every=0),
        # the paper's perturbed vortex at resolution 128: odd lattices of 127 x 127, energy series
        dict(name="paper4d_127", kind="pert", nx=127, ny=127, steps=600, samples=128, storage="f32", stats=True,
             every=100),
        # 16-bit fixed-point populations on the 4-D set-up
        dict(name="mc4d_256_fx16", kind="tgv", nx=256, ny=256, steps=300, samples=128, storage="fx16", stats=True,
             every=0),
        # a batch of unlike samples (Taylor-Green of three sizes, channels of many) in BF16, run as groups
        dict(name="uneven_bf16", kind="uneven", n_tgv=128, n_cyl=32, storage="bf16"),
        # the cylinder collocation study on the drag coefficient, with its steady-state test
        dict(name="cylinder_gpc_f32", kind="channel", nd=20, steps=4000, samples=9, storage="f32", steady=True,
             bc="halfway", inout="face", gpc=True),
        # the method comparison's Monte Carlo arm on the cylinder in FP64
        dict(name="cylinder_mc_f64", kind="channel", nd=20, steps=400, samples=64, storage="f64", steady=False,
             bc="halfway", inout="face", gpc=False),
        # coefficients, mean and variance of the benchmark's fields (tensor grid)
        dict(name="project_gpc4d_256", kind="project", dim=4, pts=5, order=4, quad="gl", fields=2 * 256 * 256 + 1,
             dtype="f32"),
        # coefficients on the 137-point sparse grid, fields of the paper's resolution 256 (odd count)
        dict(name="project_smolyak_255", kind="project", dim=4, pts=3, order=3, quad="smolyak",
             fields=2 * 255 * 255 + 1, dtype="f32"),
        # Monte Carlo mean and variance of a large ensemble's fields
        dict(name="stats_mc_512", kind="stats", samples=1024, fields=2 * 512 * 512 + 1, dtype="f32"),
        # distance of two resolutions' speed distributions (statistical solutions), n = 128 against 256
        dict(name="w1_128_256", kind="w1", sa=128, na=127 * 127, sb=256, nb=255 * 255, dtype="f32", bins=1 << 20),
    ]


def _log(rng: random.Random, lo: float, hi: float) -> int:
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random) -> dict:
    kind = rng.choice(["uq", "tgv", "tgv", "pert", "channel", "channel", "project", "stats", "w1", "uneven"])
    if kind == "uq":
        n, storage = _log(rng, 48, 384), rng.choice(["f32", "f32", "f64"])
        dim, pts, order = rng.choice([(1, 5, 4), (2, 5, 4), (3, 4, 3), (4, 3, 2)])
        most = 3e9 if storage == "f64" else 3e10
        steps = max(20, int(min(_log(rng, 100, 2000), most / (n * n * pts ** dim))))
        return dict(kind="uq", nx=n, ny=n, steps=steps, dim=dim, pts=pts, order=order, storage=storage)
    if kind in ("tgv", "pert"):
        nx = _log(rng, 32, 640)
        ny = nx if kind == "pert" or rng.random() < 0.7 else _log(rng, 32, 640)
        storage = rng.choice(["f32", "f32", "f32", "f16", "bf16", "fx16"])
        samples = max(1, min(_log(rng, 4, 512), int(6e7 / (nx * ny))))
        steps = max(10, int(min(_log(rng, 50, 1500), 2e10 / (nx * ny * samples))))
        return dict(kind=kind, nx=nx, ny=ny, steps=steps, samples=samples, storage=storage, stats=samples > 1,
                    every=rng.choice([0, 0, 50]))
    if kind == "channel":
        nd = rng.randint(8, 30)
        storage = rng.choice(["f32", "f32", "fx16", "f64", "f64"])
        bc, inout = rng.choice([("halfway", "face")] * 3 + [("bouzidi", "face"), ("bouzidi", "interpolated")])
        samples = _log(rng, 3, 64)
        steps = max(20, int(min(_log(rng, 200, 4000), (4e8 if storage == "f64" else 2e9) / (90 * nd * nd * samples))))
        return dict(kind="channel", nd=nd, steps=steps, samples=samples, storage=storage, steady=False, bc=bc,
                    inout=inout, gpc=False)
    if kind == "project":
        dim, pts, order, quad = rng.choice([(1, 9, 8, "gl"), (2, 7, 5, "gl"), (3, 5, 4, "gl"), (4, 5, 4, "gl"),
                                            (4, 3, 2, "gl"), (4, 3, 3, "smolyak"), (3, 3, 3, "smolyak")])
        n = _log(rng, 24, 400)
        return dict(kind="project", dim=dim, pts=pts, order=order, quad=quad, fields=2 * n * n + 1,
                    dtype=rng.choice(["f32", "f32", "f64"]))
    if kind == "stats":
        n = _log(rng, 24, 512)
        return dict(kind="stats", samples=max(2, min(_log(rng, 16, 4096), int(6e8 / (2 * n * n)))),
                    fields=2 * n * n + 1, dtype=rng.choice(["f32", "f32", "f64"]))
    if kind == "w1":
        n = _log(rng, 16, 256)
        m = rng.choice([n, max(8, n // 2)])
        return dict(kind="w1", sa=m, na=(m - 1) ** 2, sb=n, nb=(n - 1) ** 2, dtype=rng.choice(["f32", "f32", "f64"]),
                    bins=1 << rng.choice([12, 16, 20]))
    return dict(kind="uneven", n_tgv=_log(rng, 8, 96), n_cyl=rng.randint(2, 24), storage=rng.choice(["bf16", "f32", "fx16"]))


# ---- inputs ------------------------------------------------------------------------------------------

_PARAMS = ["nu", "u0", "zeta2", "zeta3"]


def _bounds(rng: random.Random, dim: int) -> list[tuple[float, float]]:
    """Bounds of the uncertain inputs: the 4-D workload's, each end moved by up to a tenth of the width."""
    out = []
    for lo, hi in workloads.TGV4D_BOUNDS[:dim]:
        w = 0.1 * (hi - lo)
        out.append((lo + w * rng.random(), hi - w * rng.random()))
    return out


def _workload(case: dict, rng: random.Random) -> workloads.Workload:
    """The workload of a uq, tgv or pert case."""
    if case["kind"] == "pert":
        n = case["nx"] + 1
        ma, re = workloads.tgv_paper4d_params(n)
        p = U.uqlb_unit_converter(n, ma, re)
        w = workloads.tgv_paper4d(n, p["tau"], p["u_lattice"], case["steps"], n_samples=case["samples"],
                                  seed=rng.randrange(1 << 31), storage=case["storage"])
        return replace(w, qoi_every=case["every"])
    base = replace(workloads.tgv(case["nx"], case["steps"]), ny=case["ny"])
    if case["kind"] == "uq":
        return workloads.Workload("uq", base, _bounds(rng, case["dim"]), _PARAMS[:case["dim"]], "gpc",
                                  pts_per_dim=case["pts"], order=case["order"], storage=case["storage"])
    return workloads.Workload("mc", base, _bounds(rng, 4), _PARAMS, "mc", n_mc=case["samples"],
                              seed=rng.randrange(1 << 31), storage=case["storage"], qoi_every=case["every"])


def _channel(case: dict, rng: random.Random) -> workloads.Workload:
    mid = 0.04 * (1.0 + 0.02 * (rng.random() - 0.5))
    spread = 0.1 if case["gpc"] else 0.2
    base = workloads.channel(case["nd"], steps=case["steps"], steady_tol=1e-8 if case["steady"] else 0.0,
                             bc=case["bc"], inout=case["inout"])
    base.steady_checks = 1 if case["storage"] == "f64" else 5
    bounds = [((1.0 - spread) * mid, (1.0 + spread) * mid)]
    if case["gpc"]:
        return workloads.Workload("cylinder", base, bounds, ["u0"], "gpc", pts_per_dim=case["samples"],
                                  order=case["samples"] - 1, storage=case["storage"], qoi_every=100)
    return workloads.Workload("cylinder", base, bounds, ["u0"], "mc", n_mc=case["samples"], seed=rng.randrange(1 << 31),
                              storage=case["storage"], qoi_every=100)


def _fields(samples: int, fields: int, dtype: str, seed: int) -> torch.Tensor:
    """Field rows as runs leave them: a few smooth modes whose amplitudes vary with the sample, plus
    small-scale differences."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    t = torch.float64 if dtype == "f64" else torch.float32
    x = torch.linspace(0.0, 6.0 * math.pi, fields, device=DEV, dtype=torch.float32)
    modes = torch.stack([torch.sin(x), torch.sin(2.0 * x + 0.3), torch.cos(3.0 * x)])
    amp = 0.01 * (torch.tensor([1.0, 0.1, 0.1], device=DEV) *
                  (1.0 + 0.2 * torch.randn((samples, 3), device=DEV, generator=g)))
    m = torch.empty((samples, fields), device=DEV, dtype=t)
    for s in range(0, samples, 64):
        blk = amp[s:s + 64] @ modes
        m[s:s + 64] = blk + 1e-5 * torch.randn(blk.shape, device=DEV, generator=g)
    return m


def prepare(case: dict, seed: int) -> dict:
    rng = random.Random(seed)
    kind = case["kind"]
    ens = ensemble.Ensemble(0)
    st = {"case": case, "ens": ens}
    if kind in ("uq", "tgv", "pert", "channel"):
        w = _channel(case, rng) if kind == "channel" else _workload(case, rng)
        ens.setup(w)
        st["w"] = w
        if kind != "uq":
            st["samples"] = ens.ensemble_samples(w)
            st["out"] = {}
    elif kind == "uneven":
        specs = workloads.uneven_batch(seed=rng.randrange(1 << 31), n_tgv=case["n_tgv"], n_cyl=case["n_cyl"])
        st["samples"] = [ensemble.sample_struct(replace(s, steps=min(s.steps, 2000))) for s in specs]
        st["out"] = {}
    elif kind == "project":
        ens.set_inputs(_bounds(rng, case["dim"]))
        ens.init_gpc(case["order"], case["pts"], quad=U.UQLB_QUAD_CLENSHAW_CURTIS_SMOLYAK
                     if case["quad"] == "smolyak" else U.UQLB_QUAD_GAUSS_LEGENDRE_TENSOR)
        st["m"] = _fields(ens.num_samples, case["fields"], case["dtype"], seed)
        st["coeffs"] = torch.empty((ens.num_terms, case["fields"]), dtype=torch.float64, device=DEV)
    elif kind == "stats":
        ens.set_inputs(_bounds(rng, 1))
        ens.init_mc(case["samples"], seed)
        st["m"] = _fields(case["samples"], case["fields"], case["dtype"], seed)
    else:
        st["a"] = _fields(case["sa"], 2 * case["na"] + 1, case["dtype"], seed)
        st["b"] = _fields(case["sb"], 2 * case["nb"] + 1, case["dtype"], seed + 1000003)
    return st


# ---- one pass ----------------------------------------------------------------------------------------

def run(state: dict):
    case, ens = state["case"], state["ens"]
    kind = case["kind"]
    if kind == "uq":
        mean, var, _, _ = ens.run_uq_host(state["w"], fields_dtype="f64" if case["storage"] == "f64" else "f32")
        return {"mean": mean, "var": var}
    if kind in ("tgv", "pert"):
        res = ens.run_batch(state["samples"], storage=case["storage"], qoi_every=case["every"],
                            series=case["every"] > 0, out=state["out"])
        out = {"fields": res["fields"], "qoi": res["qoi"]}
        if case["every"]:
            out["series"] = res["series"]
        if case["stats"]:
            out["mean"], out["var"] = ens.stats(res["fields"])
        return out
    if kind == "channel":
        res = ens.run_batch(state["samples"], storage=case["storage"], qoi_every=100, series=True,
                            fields_dtype="f64" if case["storage"] == "f64" else "f32", out=state["out"])
        cd = res["qoi"][:, U.UQLB_QOI_CD:U.UQLB_QOI_CD + 1]
        out = {"fields": res["fields"], "qoi": res["qoi"], "series": res["series"]}
        out["cd_mean"], out["cd_var"] = ens.stats(ens.project(cd) if case["gpc"] else cd)
        return out
    if kind == "uneven":
        return {"qoi": ens.run_batch(state["samples"], storage=case["storage"], fields=False, out=state["out"])["qoi"]}
    if kind == "project":
        c = ens.project(state["m"], state["coeffs"])
        mean, var = ens.stats(c)
        return {"coeffs": c, "mean": mean, "var": var}
    if kind == "stats":
        mean, var = ens.stats(state["m"])
        return {"mean": mean, "var": var}
    dist, bound, (ia, ib) = ens.w1_speed(state["a"], case["na"], state["b"], case["nb"], bins=case["bins"])
    return {"distance": dist, "bound": bound, "nonfinite_a": ia, "nonfinite_b": ib}


def _uneven_nodes(case: dict) -> float:
    """Expected node updates of an uneven batch: the mean over its random sizes and step counts."""
    tgv = sum(n * n * min(1300.0 * (n / 256.0) ** 2 if n > 128 else 500.0, 2000.0) for n in (128, 256, 512)) / 3.0
    return case["n_tgv"] * tgv + case["n_cyl"] * 90.2 * 30.0 ** 2 * 2000.0


def work(case: dict) -> dict:
    """What a pass cannot do without: about 100 operations per node update of the BGK step, every input
    read once and every output written once (the lattices are neither)."""
    kind = case["kind"]
    if kind in ("uq", "tgv", "pert"):
        nodes = case["nx"] * case["ny"]
        s = case["pts"] ** case["dim"] if kind == "uq" else case["samples"]
        fields = 2 * nodes + 1
        eb = 8 if case["storage"] == "f64" else 4
        k = math.comb(case["dim"] + case["order"], case["order"]) if kind == "uq" else 2
        out = 2 * fields * 8 + (0 if kind == "uq" else s * (fields * eb + 64))
        return {"bytes": 128.0 * s + out, "flops": 100.0 * nodes * s * case["steps"] + 2.0 * k * s * fields}
    if kind == "channel":
        nodes = 22 * case["nd"] * ((41 * case["nd"]) // 10)
        eb = 8 if case["storage"] == "f64" else 4
        s = case["samples"]
        return {"bytes": s * (128.0 + eb * (2 * nodes + 1) + 64 + 8 * (case["steps"] // 100)),
                "flops": 100.0 * nodes * s * case["steps"]}
    if kind == "uneven":
        return {"bytes": 192.0 * (case["n_tgv"] + case["n_cyl"]), "flops": 100.0 * _uneven_nodes(case)}
    eb = 8 if case.get("dtype") == "f64" else 4
    if kind == "project":
        if case["quad"] == "gl":
            s, flops = case["pts"] ** case["dim"], 0.0
            rows = s
            for d in range(case["dim"]):  # one input at a time, the last first
                terms = math.comb(d + 1 + case["order"], case["order"])
                rows //= case["pts"]
                flops += 2.0 * rows * terms * case["pts"]
        else:
            s = {3: 69, 4: 137}[case["dim"]]
            flops = 2.0 * s * math.comb(case["dim"] + case["order"], case["order"])
        k = math.comb(case["dim"] + case["order"], case["order"])
        f = case["fields"]
        return {"bytes": f * (s * eb + (k + 2) * 8.0), "flops": f * (flops + 2.0 * k)}
    if kind == "stats":
        return {"bytes": case["fields"] * (case["samples"] * eb + 16.0), "flops": 4.0 * case["fields"] * case["samples"]}
    n = case["sa"] * case["na"] + case["sb"] * case["nb"]
    return {"bytes": n * 2.0 * eb + 32, "flops": 5.0 * n}


# ---- the same numbers in FP64 with torch and numpy ------------------------------------------------------

_CX = [0, 1, 0, -1, 0, 1, -1, -1, 1]
_CY = [0, 0, 1, 0, -1, 1, 1, -1, -1]
_OPP = [0, 3, 4, 1, 2, 7, 8, 5, 6]
_W = [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4


def _moments(g):
    drho = g.sum(0)
    jx = g[1] - g[3] + g[5] - g[6] - g[7] + g[8]
    jy = g[2] - g[4] + g[5] + g[6] - g[7] - g[8]
    return drho, jx, jy, jx / (1.0 + drho), jy / (1.0 + drho)


def _equilibrium(i, drho, rho, ux, uy, uu):
    """f_i^eq - w_i."""
    if i == 0:
        return _W[0] * (drho - 1.5 * rho * uu)
    cu = _CX[i] * ux + _CY[i] * uy
    return _W[i] * (drho + rho * (3.0 * cu + 4.5 * cu * cu - 1.5 * uu))


def _start(rho, u, v):
    g = torch.empty((9,) + tuple(u.shape), dtype=torch.float64, device=DEV)
    uu = u * u + v * v
    for i in range(9):
        g[i] = _equilibrium(i, rho - 1.0, rho, u, v, uu)
    return g


def _relaxed(g, omega):
    """Post-collision populations and the velocity they were relaxed to."""
    drho, jx, jy, ux, uy = _moments(g)
    rho = 1.0 + drho
    uu = ux * ux + uy * uy
    return [g[i] + omega * (_equilibrium(i, drho, rho, ux, uy, uu) - g[i]) for i in range(9)], ux, uy


def _grid(nx, ny):
    y, x = torch.meshgrid(torch.arange(ny, dtype=torch.float64, device=DEV),
                          torch.arange(nx, dtype=torch.float64, device=DEV), indexing="ij")
    return x, y


def _column(values):
    return torch.tensor(values, dtype=torch.float64, device=DEV).reshape(-1, 1, 1)


def _tgv_start(samples):
    s0 = samples[0]
    x, y = _grid(s0.nx, s0.ny)
    u0 = _column([s.u0 for s in samples])
    if s0.kind == workloads.TGV_PERTURBED:
        x, y = 2.0 * math.pi * x / s0.nx, 2.0 * math.pi * y / s0.ny
        kx, ky = (torch.sin(4.0 * x), torch.cos(4.0 * x)), (torch.sin(4.0 * y), torch.cos(4.0 * y))
        eps = sum(_column([s.pert[2 * i + j] for s in samples]) * kx[i] * ky[j] for i in range(2) for j in range(2))
        a = u0 + 0.25 * eps
        u, v = -a * torch.cos(2.0 * x) * torch.sin(2.0 * y), a * torch.sin(2.0 * x) * torch.cos(2.0 * y)
        return 1.0 - 0.75 * a * a * (torch.cos(4.0 * x) + torch.cos(4.0 * y)), u, v
    kx, ky = 2.0 * math.pi / s0.nx, 2.0 * math.pi / s0.ny
    u = v = 0.0
    for m, a in ((1, u0), (2, _column([s.amp2 for s in samples])), (3, _column([s.amp3 for s in samples]))):
        u = u + a * torch.sin(m * kx * x) * torch.cos(m * ky * y)
        v = v - a * torch.cos(m * kx * x) * torch.sin(m * ky * y)
    return 1.0 + 0.75 * u0 * u0 * (torch.cos(2.0 * kx * x) + torch.cos(2.0 * ky * y)), u, v


def _rows(samples, g, solid=None):
    """Field rows [u, v, K] and the scalar columns of the state g."""
    drho, jx, jy, ux, uy = _moments(g)
    rho = 1.0 + drho
    if solid is not None:
        ux, uy, rho = (torch.where(solid, torch.zeros_like(a), a) for a in (ux, uy, rho))
    k = torch.tensor([2.0 / (s.nx * s.ny * s.u_ref ** 2) if s.u_ref > 0 else 0.0 for s in samples],
                     dtype=torch.float64, device=DEV) * (ux * ux + uy * uy).sum((1, 2))
    n = len(samples)
    qoi = torch.zeros((n, U.UQLB_QOI_COLS), dtype=torch.float64, device=DEV)
    qoi[:, U.UQLB_QOI_K] = k
    qoi[:, U.UQLB_QOI_MASS] = rho.sum((1, 2))
    qoi[:, U.UQLB_QOI_MOMX] = (rho * ux).sum((1, 2))
    qoi[:, U.UQLB_QOI_MOMY] = (rho * uy).sum((1, 2))
    return torch.cat([ux.reshape(n, -1), uy.reshape(n, -1), k[:, None]], 1), qoi


def _run_tgv(samples, steps, every=0):
    fields, qois, series = [], [], []
    per = max(1, int(4e6 / (samples[0].nx * samples[0].ny)))
    for b in range(0, len(samples), per):
        part = samples[b:b + per]
        omega = _column([1.0 / (3.0 * s.nu + 0.5) for s in part])
        g = _start(*_tgv_start(part))
        ks = [_rows(part, g)[1][:, U.UQLB_QOI_K]] if every else []
        for t in range(steps):
            post, _, _ = _relaxed(g, omega)
            for i in range(9):
                g[i] = torch.roll(post[i], (_CY[i], _CX[i]), (1, 2))
            if every and (t + 1) % every == 0:
                ks.append(_rows(part, g)[1][:, U.UQLB_QOI_K])
        f, q = _rows(part, g)
        q[:, U.UQLB_QOI_STEPS] = steps
        fields.append(f)
        qois.append(q)
        series += [torch.stack(ks, 1)] if every else []
    return torch.cat(fields), torch.cat(qois), torch.cat(series) if every else None


def _run_channel(samples, steps, every):
    """Halfway walls and staircase obstacle, moving-wall inlet, anti-bounce-back outlet; drag every
    `every` steps."""
    s0 = samples[0]
    nx, ny, n = s0.nx, s0.ny, len(samples)
    x, y = _grid(nx, ny)
    solid = (x + 0.5 - s0.cyl_cx) ** 2 + (y + 0.5 - s0.cyl_cy) ** 2 < s0.cyl_r ** 2
    omega = _column([1.0 / (3.0 * s.nu + 0.5) for s in samples])
    u0 = torch.tensor([s.u0 for s in samples], dtype=torch.float64, device=DEV)
    norm = 2.0 / (u0 * u0 * 2.0 * s0.cyl_r)
    g = torch.zeros((9, n, ny, nx), dtype=torch.float64, device=DEV)
    back, wall, profile = [None] * 9, [None] * 9, [None] * 9
    h = torch.arange(ny, dtype=torch.float64, device=DEV) + 0.5
    for i in range(1, 9):
        sx, sy = x - _CX[i], y - _CY[i]
        out_y = (sy < 0) | (sy >= ny)
        inside = ~out_y & (sx >= 0) & (sx < nx)
        src = torch.roll(solid, (_CY[i], _CX[i]), (0, 1))
        back[i] = out_y | (inside & src)            # halfway bounce-back
        wall[i] = (inside & src & ~solid).nonzero(as_tuple=True)  # fluid nodes with the obstacle behind -c_i
        hy = h - 0.5 * _CY[i]
        profile[i] = torch.where(out_y[:, 0], torch.zeros_like(hy), 4.0 * 1.5 * hy * (ny - hy) / (ny * ny))
    row = torch.arange(ny, device=DEV)
    series = torch.full((n, steps // every + 1), float("nan"), dtype=torch.float64, device=DEV)
    cd = cl = torch.zeros(n, dtype=torch.float64, device=DEV)
    for t in range(steps):
        post, ux, uy = _relaxed(g, omega)
        if (t + 1) % every == 0 or t + 1 == steps:
            fx = fy = 0.0
            for i in range(1, 9):  # the link along c_o = -c_i carries 2 c_o f*_o
                o = _OPP[i]
                tot = (post[o][:, wall[i][0], wall[i][1]] + _W[o]).sum(1)
                fx, fy = fx + 2.0 * _CX[o] * tot, fy + 2.0 * _CY[o] * tot
            cd, cl = fx * norm, fy * norm
            if (t + 1) % every == 0:
                series[:, (t + 1) // every - 1] = cd
        ramp = 0.5 * (1.0 - math.cos(math.pi * t / s0.ramp_steps)) if t < s0.ramp_steps else 1.0
        uxo, uyo = ux[:, :, -1], uy[:, :, -1]
        uu = uxo * uxo + uyo * uyo
        g[0] = post[0]
        for i in range(1, 9):
            o = _OPP[i]
            g[i] = torch.where(back[i], post[o], torch.roll(post[i], (_CY[i], _CX[i]), (1, 2)))
            ok = (row - _CY[i] >= 0) & (row - _CY[i] < ny)
            if _CX[i] == 1:
                v = post[o][:, :, 0] + 6.0 * _W[i] * ramp * u0[:, None] * profile[i]
                g[i][:, :, 0] = torch.where(ok, v, post[o][:, :, 0])
            elif _CX[i] == -1:
                cu = _CX[i] * uxo + _CY[i] * uyo
                v = -post[o][:, :, -1] + 2.0 * _W[i] * (4.5 * cu * cu - 1.5 * uu)
                g[i][:, :, -1] = torch.where(ok, v, post[o][:, :, -1])
        g[:, :, solid] = 0.0
    f, q = _rows(samples, g, solid)
    q[:, U.UQLB_QOI_CD], q[:, U.UQLB_QOI_CL], q[:, U.UQLB_QOI_STEPS] = cd, cl, steps
    return f, q, series


def _gpc_basis(dim, order, pts):
    """Points' weights a[s] and basis Phi[k, s] of the tensor Gauss-Legendre grid, total degree."""
    x, w = np.polynomial.legendre.leggauss(pts)
    phi = np.stack([math.sqrt(2 * p + 1) * np.polynomial.legendre.Legendre.basis(p)(x) for p in range(order + 1)])
    at = np.stack(np.meshgrid(*[np.arange(pts)] * dim, indexing="ij"), -1).reshape(-1, dim)
    alpha = U.uqlb_multi_indices(dim, order)
    a = np.prod(0.5 * w[at], axis=1)
    return a, np.prod([phi[alpha[:, d]][:, at[:, d]] for d in range(dim)], axis=0)


def _coefficients(weights, m):
    """weights [K, S] times the rows of m, in FP64."""
    w = torch.as_tensor(weights, dtype=torch.float64, device=DEV)
    out = torch.empty((w.shape[0], m.shape[1]), dtype=torch.float64, device=DEV)
    for f in range(0, m.shape[1], 1 << 16):
        out[:, f:f + (1 << 16)] = w @ m[:, f:f + (1 << 16)].double()
    return out


def _mean_var(m, ddof=1):
    mean = torch.empty(m.shape[1], dtype=torch.float64, device=DEV)
    var = torch.empty_like(mean)
    for f in range(0, m.shape[1], 1 << 15):
        d = m[:, f:f + (1 << 15)].double()
        mean[f:f + (1 << 15)] = d.mean(0)
        var[f:f + (1 << 15)] = ((d - d.mean(0)) ** 2).sum(0) / (m.shape[0] - ddof)
    return mean, var


def exact(case: dict, seed: int):
    kind = case["kind"]
    if kind == "uneven":
        return None
    rng = random.Random(seed)
    ens = ensemble.Ensemble(0)
    if kind in ("uq", "tgv", "pert"):
        s = case["pts"] ** case["dim"] if kind == "uq" else case["samples"]
        if case["nx"] * case["ny"] * s * case["steps"] > 1.1e10:  # about 20 s
            return None
        w = _workload(case, rng)
        ens.setup(w)
        samples = ens.ensemble_samples(w)
        f, q, series = _run_tgv(samples, case["steps"], case.get("every", 0))
        if kind == "uq":
            a, phi = _gpc_basis(case["dim"], case["order"], case["pts"])
            c = _coefficients(a * phi, f)
            return {"mean": c[0].cpu().numpy(), "var": (c[1:] ** 2).sum(0).cpu().numpy()}
        out = {"fields": f, "qoi": q}
        if case["every"]:
            out["series"] = series
        if case["stats"]:
            out["mean"], out["var"] = _mean_var(f)
        return out
    if kind == "channel":
        if (case["bc"], case["inout"]) != ("halfway", "face"):
            return None
        w = _channel(case, rng)
        ens.setup(w)
        f, q, series = _run_channel(ens.ensemble_samples(w), case["steps"], 100)
        cd = q[:, U.UQLB_QOI_CD:U.UQLB_QOI_CD + 1]
        out = {"fields": f, "qoi": q, "series": series}
        if case["gpc"]:
            a, phi = _gpc_basis(1, case["samples"] - 1, case["samples"])
            c = _coefficients(a * phi, cd)
            out["cd_mean"], out["cd_var"] = c[0], (c[1:] ** 2).sum(0)
        else:
            out["cd_mean"], out["cd_var"] = _mean_var(cd)
        return out
    if kind == "project":
        st = prepare(case, seed)
        if case["quad"] == "gl":
            a, phi = _gpc_basis(case["dim"], case["order"], case["pts"])
        else:  # the sparse grid itself is an input: its points and weights
            _, xi, a = st["ens"].samples()
            alpha = U.uqlb_multi_indices(case["dim"], case["order"])
            one = np.stack([math.sqrt(2 * p + 1) * np.polynomial.legendre.Legendre.basis(p)(xi)
                            for p in range(case["order"] + 1)])
            phi = np.prod([one[alpha[:, d], :, d] for d in range(case["dim"])], axis=0)
        c = _coefficients(a * phi, st["m"])
        return {"coeffs": c, "mean": c[0], "var": (c[1:] ** 2).sum(0)}
    st = prepare(case, seed)
    if kind == "stats":
        mean, var = _mean_var(st["m"])
        return {"mean": mean, "var": var}
    speeds = []
    for m, nodes in ((st["a"], case["na"]), (st["b"], case["nb"])):
        u, v = m[:, :nodes].double(), m[:, nodes:2 * nodes].double()
        speeds.append(torch.sqrt(u * u + v * v).reshape(-1))
    vmax = max(float(s.max()) for s in speeds)
    bins = case["bins"]
    cdf = [torch.bincount((s * (bins / vmax)).long().clamp(0, bins - 1), minlength=bins).double().cumsum(0) / s.numel()
           for s in speeds]
    h = vmax / bins
    return {"distance": float((cdf[0] - cdf[1]).abs().sum() * h), "bound": h, "nonfinite_a": 0, "nonfinite_b": 0}
