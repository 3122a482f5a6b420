"""The solver's measured work: time steps of the workloads that its users run.

A case is a plain dict; ``kind`` says which workload it is:

* ``column``  one soil column (1-d) in FP64 through ``Solver.step``;
* ``plane``   a 2-d field: the Gardner infiltration, the strip infiltration or
  the two-layer field;
* ``field``   a 3-d heterogeneous drainage;
* ``columns`` a batch of soil columns through ``Columns.run``;
* ``served``  a mix of resident requests stepped together through ``Batcher``;
* ``laws``    water content and conductivity of a resident state
  (``richards_soil_eval`` on device arrays).

A pass hands the initial state to the solver (or the batch), takes ``steps``
time steps and reads the state back into a device array: the loop of a user's
program, from the same start every time.  Everything a program sets up once --
the contexts with their soil, boundary conditions and sink -- is prepared.
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_2606_04292_gb300 import richards as R
from paper_2606_04292_gb300 import workloads as W


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the paper's Celia column: the smallest problem, one thread block,
        # stepped in FP64 as in the temporal studies
        dict(name="column_celia_128", kind="column", soil="celia", n=128, dt=10.0, steps=2),
        # the layered column (three laws), odd and finer than the paper's
        dict(name="column_layered_777", kind="column", soil="composite", n=777, dt=10.0, steps=1),
        # the paper's 2-d Gardner infiltration, 128^2, mixed precision
        dict(name="plane_gardner_128", kind="plane", soil="gardner", n=128, precision=2, tol=1e-10, dt=0.1, steps=2),
        # strip infiltration on the odd 513^2 grid, W(2,2) on the three finest
        # levels, as the benchmark's mixed run of it
        dict(name="plane_strip_513", kind="plane", soil="strip", n=513, precision=2, tol=1e-10, dt=60.0, steps=2),
        # the same workload in plain FP64 at the served 257^2
        dict(name="plane_strip_fp64_257", kind="plane", soil="strip", n=257, precision=0, tol=1e-8, dt=60.0, steps=1),
        # the two-layer field with its full-multigrid start and 10 + 10 sweeps
        dict(name="plane_layered_256", kind="plane", soil="two_layer", n=256, precision=2, tol=1e-10, dt=0.01,
             steps=2),
        # the benchmark's headline: 256^3 drainage, FP64 outer layer
        dict(name="field_256", kind="field", n0=256, n1=256, n2=256, precision=2, tol=1e-8, dt=300.0, steps=2),
        # a ragged field of about 10^6 cells: no axis nests
        dict(name="field_ragged", kind="field", n0=117, n1=93, n2=101, precision=2, tol=1e-9, dt=300.0, steps=2),
        # drainage in plain FP64
        dict(name="field_fp64_96", kind="field", n0=96, n1=96, n2=96, precision=0, tol=1e-8, dt=300.0, steps=1),
        # batched root-uptake columns of 64 to 1024 cells
        dict(name="columns_4096", kind="columns", ncol=4096, nmin=64, nmax=1024, precision=2, tol=1e-11, dt=600.0,
             steps=4),
        # served requests: a mix of sizes, laws and dimensions in one batcher
        dict(name="served_8", kind="served", requests=8, size2d=257, size3d=65, tol=1e-10, steps=1),
        # theta and K of a 128^3 state for water accounting, FP64 laws
        dict(name="laws_128", kind="laws", n0=128, n1=128, n2=128, soil="vangenuchten"),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["column", "plane", "plane", "field", "field", "columns", "served", "laws"])
    if kind == "column":
        return dict(kind=kind, soil=rng.choice(["celia", "composite"]), n=_logint(rng, 32, 2048),
                    dt=round(rng.uniform(2.0, 10.0), 3), steps=1)
    if kind == "plane":
        soil = rng.choice(["gardner", "strip", "two_layer"])
        prec = rng.choice([0, 2])
        lo, hi = {"gardner": (64, 385), "strip": (65, 641), "two_layer": (64, 320)}[soil]
        if prec == 0:
            hi = 257
        dt = {"gardner": 0.1, "strip": 60.0, "two_layer": 0.01}[soil] * rng.uniform(0.5, 1.0)
        return dict(kind=kind, soil=soil, n=_logint(rng, lo, hi), precision=prec, tol=1e-8 if prec == 0 else 1e-10,
                    dt=round(dt, 6), steps=1)
    if kind == "field":
        prec = rng.choice([0, 2, 2])
        hi = 80 if prec == 0 else 224
        n = [_logint(rng, 24, hi) for _ in range(3)]
        if prec and rng.random() < 0.5:                  # even sizes: nested levels, colour-split parameters
            n = [max(32, 16 * (m // 16)) for m in n]
        return dict(kind=kind, n0=n[0], n1=n[1], n2=n[2], precision=prec, tol=1e-8 if prec == 0 else 1e-9,
                    dt=round(rng.uniform(100.0, 300.0), 2), steps=1)
    if kind == "columns":
        nmin = _logint(rng, 16, 128)
        return dict(kind=kind, ncol=_logint(rng, 8, 3000), nmin=nmin, nmax=_logint(rng, nmin, 1500), precision=2,
                    tol=1e-11, dt=round(rng.uniform(200.0, 600.0), 2), steps=rng.randint(1, 3))
    if kind == "served":
        return dict(kind=kind, requests=rng.randint(2, 8), size2d=_logint(rng, 65, 257), size3d=_logint(rng, 17, 65),
                    tol=1e-10, steps=1)
    return dict(kind="laws", n0=_logint(rng, 16, 200), n1=_logint(rng, 16, 200), n2=_logint(rng, 16, 200),
                soil=rng.choice(["haverkamp", "gardner", "vangenuchten", "layers"]))


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _uniform(g, n, lo, hi):
    return lo + (hi - lo) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64)


def _smooth(g, shape, corr):
    """A standardised Gaussian field, correlated over ``corr`` cells."""
    F = torch.fft.rfftn(torch.randn(shape, generator=g, device="cuda", dtype=torch.float64))
    s = corr / math.sqrt(2.0)
    f = [torch.fft.fftfreq(m, device="cuda", dtype=torch.float64) for m in shape[:-1]]
    f.append(torch.fft.rfftfreq(shape[-1], device="cuda", dtype=torch.float64))
    for d, x in enumerate(f):
        F *= torch.exp(-2.0 * math.pi ** 2 * s * s * x * x).reshape([-1 if k == d else 1 for k in range(len(shape))])
    G = torch.fft.irfftn(F, s=shape)
    return (G - G.mean()) / G.std()


def _host(t):
    """Pinned host copy as a numpy array: what a program hands in from."""
    p = torch.empty(t.numel(), dtype=torch.float64, pin_memory=True)
    p.copy_(t.reshape(-1))
    return p.numpy()


def _column_problem(c, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    make = W.celia_1d if c["soil"] == "celia" else W.celia_composite_1d
    prob = make(n=c["n"], dt=c["dt"], precision=0)
    top = -20.7 * rng.uniform(0.9, 1.1)
    dry = -61.5 * rng.uniform(0.95, 1.05)
    prob["bc"]["value"][0], prob["bc"]["value"][1] = dry, top
    # past the first steps: a smooth wetting front down from the top
    z = (np.arange(c["n"]) + 0.5) / c["n"]
    prob["psi0"] = dry + (top - dry) * np.exp(-(1.0 - z) / rng.uniform(0.1, 0.2))
    return prob


def _plane_problem(c, seed):
    g = _gen(seed)
    n, soil = c["n"], c["soil"]
    kw = dict(precision=c["precision"], tol=c["tol"])
    if soil == "gardner":
        prob = W.gardner_2d(n=n, dt=c["dt"], **kw)
        psi = -10.0 + 0.05 * _smooth(g, (n, n), 6.0)
    elif soil == "strip":
        prob = W.strip_2d(n=n, dt=c["dt"], cycle_gamma=2, gamma_levels=3, **kw)
        psi = -10.0 + 0.05 * _smooth(g, (n, n), 6.0)
    else:
        prob = W.two_layer_2d(n=n, dt=c["dt"], **kw)
        z = (torch.arange(n, device="cuda", dtype=torch.float64) + 0.5) * (100.0 / n)
        psi = -z[:, None].expand(n, n) * (1.0 + 0.01 * _smooth(g, (n, n), 8.0))
    prob["psi0"] = _host(psi)
    return prob


def _field_problem(c, seed):
    g = _gen(seed)
    n = (c["n0"], c["n1"], c["n2"])
    N = n[0] * n[1] * n[2]
    prob = W.drainage_3d(n=16, dt=c["dt"], precision=c["precision"], tol=c["tol"])
    prob["n"] = n
    Ks = torch.exp(math.log(1e-5) + _smooth(g, n[::-1], 8.0)).reshape(-1)
    prob["soil"].update(Ks_field=_host(Ks), p1_field=_host(_uniform(g, N, 2.0, 5.0)),
                        p2_field=_host(_uniform(g, N, 1.5, 2.5)))
    # a field some hours into its drainage: drier with height
    z = (torch.arange(n[2], device="cuda", dtype=torch.float64) + 0.5) / n[2]
    psi = -0.1 - 0.4 * z[:, None, None] + 0.02 * _smooth(g, n[::-1], 8.0)
    prob["psi0"] = _host(psi)
    prob["psi_prev"] = _host(psi + 0.004 * z[:, None, None])
    return prob


def _columns_problems(c, seed):
    """Soils from the seed, lengths from the case alone."""
    probs = W.columns(ncol=c["ncol"], seed=seed, dt=c["dt"], nmin=c["nmin"], nmax=c["nmax"], precision=c["precision"],
                      tol=c["tol"], max_outer=40)
    lengths = np.random.Generator(np.random.PCG64(5)).integers(c["nmin"], c["nmax"] + 1, c["ncol"])
    for p, n in zip(probs, lengths.tolist()):
        p["n"] = (n, 1, 1)                               # wetter towards the bottom
        p["psi0"] = -1.0 + 0.3 * np.sin(np.arange(n) / n * 3.0)
    return probs


def _served_problems(c, seed):
    """Requests of the serving trace (soil, sink, heads from the seed) in a fixed order of sizes."""
    sizes = [(2, c["size2d"]), (3, c["size3d"]), (2, c["size2d"] // 2 + 1)]
    trace = W.serving_trace(seed=seed, sizes2d=(sizes[0][1], sizes[2][1]), sizes3d=(sizes[1][1],), max_requests=96)
    out = []
    for k in range(c["requests"]):
        want = sizes[k % 3]
        at = next(i for i, p in enumerate(trace) if (p["dim"], p["n"][0]) == want)
        out.append(W.with_opts(trace.pop(at), precision=2, tol=c["tol"]))
    return out


def _laws_problem(c, seed):
    g = _gen(seed)
    n = (c["n0"], c["n1"], c["n2"])
    N = n[0] * n[1] * n[2]
    prob = W.drainage_3d(n=16, precision=0)
    prob["n"] = n
    s = c["soil"]
    if s == "layers":
        prob["soil"] = dict(W.test_materials()[0])
        prob = W.with_materials(prob, W.test_materials(), W.material_pattern(prob, "layers", 3, seed))
    else:
        m = {"haverkamp": W.HAVERKAMP, "gardner": W.GARDNER, "vangenuchten": W.VANGENUCHTEN}[s]
        t = {k["model"]: k for k in W.test_materials()}[m]
        soil = dict(t, Ks_field=_host(1e-5 * torch.exp(torch.randn(N, generator=g, device="cuda",
                                                                   dtype=torch.float64))),
                    p1_field=None, p2_field=None)
        if m == W.VANGENUCHTEN:
            soil.update(p1_field=_host(_uniform(g, N, 2.0, 5.0)), p2_field=_host(_uniform(g, N, 1.5, 2.5)))
        elif m == W.GARDNER:
            soil.update(p1_field=_host(_uniform(g, N, 1.0, 5.0)))
        prob["soil"] = soil
    # heads from saturation to -30 m, most of them above -1 m
    prob["psi0"] = _host(0.02 - torch.exp(_uniform(g, N, -6.0, math.log(30.0))))
    return prob


def _solver(prob):
    stream = torch.cuda.Stream()
    return dict(solver=R.Solver(prob, stream=stream.cuda_stream), stream=stream, prob=prob,
                out=torch.empty(W.ncells(prob), dtype=torch.float64, device="cuda"))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "columns":
        probs = _columns_problems(case, seed)
        stream = torch.cuda.Stream()
        cols = R.Columns(probs, stream=stream.cuda_stream)
        return dict(case=case, cols=cols, stream=stream,
                    psi0=_host(torch.from_numpy(np.concatenate([p["psi0"] for p in probs]))),
                    out=torch.empty(cols.N, dtype=torch.float64, device="cuda"))
    if kind == "served":
        probs = _served_problems(case, seed)
        stream = torch.cuda.Stream()
        return dict(case=case, stream=stream, units=[_solver(p) for p in probs],
                    batcher=R.Batcher(max_contexts=len(probs), stream=stream.cuda_stream))
    if kind == "laws":
        st = _solver(_laws_problem(case, seed))
        st.update(case=case, psi=torch.from_numpy(st["prob"]["psi0"]).cuda(),
                  K=torch.empty_like(st["out"]))
        return st
    make = {"column": _column_problem, "plane": _plane_problem, "field": _field_problem}[kind]
    st = _solver(make(case, seed))
    st["case"] = case
    return st


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------
def _ptr(t):
    return C.cast(C.c_void_p(t.data_ptr()), C.POINTER(C.c_double))


def run(state):
    kind, steps = state["case"]["kind"], state["case"].get("steps", 1)
    if kind == "columns":
        cols = state["cols"]
        cols.set_state(state["psi0"])
        st = cols.run(state["case"]["dt"], steps, 1)
        if st != R.RICH_OK:
            raise R.RichardsError(st, "a column failed")
        R.lib().richards_columns_get_state(cols.h, _ptr(state["out"]), 1)
        return state["out"]
    if kind == "served":
        units = state["units"]
        for u in units:
            u["solver"].set_state(u["prob"]["psi0"])
        solvers = [u["solver"] for u in units]
        for _ in range(steps):
            sts, _info = state["batcher"].step(solvers, [u["prob"]["dt"] for u in units],
                                               [u["prob"]["scheme"] for u in units])
            for st in sts:
                if st != R.RICH_OK:
                    raise R.RichardsError(st, "a request failed")
        for u in units:
            u["solver"].state_to_device(u["out"].data_ptr())
        return [u["out"] for u in units]
    if kind == "laws":
        st = R.lib().richards_soil_eval(state["solver"].h, _ptr(state["psi"]), _ptr(state["out"]), _ptr(state["K"]),
                                        0, 1)
        if st != R.RICH_OK:
            raise R.RichardsError(st, "richards_soil_eval failed")
        return [state["out"], state["K"]]
    solver, prob = state["solver"], state["prob"]
    solver.set_state(prob["psi0"], prob.get("psi_prev"))
    for _ in range(steps):
        solver.step()
    solver.state_to_device(state["out"].data_ptr())
    return state["out"]


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------
def work(case):
    """Bytes: each step reads psi^n and psi^{n-1} and the per-cell soil fields
    and writes psi^{n+1} (FP64).  Flops: per cell and step one evaluation of
    the laws at the old, lagged and new state and one multigrid cycle of four
    half-sweeps and a defect on the finest level (about 150 per law pair and
    60 per stencil visit)."""
    kind, steps = case["kind"], case.get("steps", 1)
    fields = 0
    if kind == "column":
        cells = case["n"]
    elif kind == "plane":
        cells = case["n"] ** 2
    elif kind == "columns":
        cells = int(case["ncol"] * 0.5 * (case["nmin"] + case["nmax"]))
    elif kind == "served":
        size = [case["size2d"] ** 2, case["size3d"] ** 3, (case["size2d"] // 2 + 1) ** 2]
        cells = sum(size[k % 3] for k in range(case["requests"]))
    else:
        cells = case["n0"] * case["n1"] * case["n2"]
        fields = 3
    if kind == "laws":
        fields = {"vangenuchten": 3, "gardner": 2, "haverkamp": 1, "layers": 0.125}[case["soil"]]
        return {"bytes": cells * 8 * (3 + fields), "flops": cells * 150}
    return {"bytes": steps * cells * 8 * (3 + fields), "flops": steps * cells * (3 * 150 + 5 * 60)}


# ---------------------------------------------------------------------------
# The same results in plain FP64 torch: Newton on the whole system
# ---------------------------------------------------------------------------
def _theta_K(mat, psi, want):
    """Table 1: theta, d theta/d psi and K at psi (saturated for psi >= 0)."""
    ts, tr, Ks, p1, p2, p3, p4, model = (mat[k] for k in ("theta_s", "theta_r", "Ks", "p1", "p2", "p3", "p4",
                                                           "model"))
    dry = psi < 0
    h = torch.where(dry, -psi, torch.ones_like(psi))
    if model == W.HAVERKAMP:
        u, v = h ** p2, h ** p4
        th, dth = tr + p1 * (ts - tr) / (p1 + u), p1 * (ts - tr) * p2 * (u / h) / (p1 + u) ** 2
        K = Ks * p3 / (p3 + v)
    elif model == W.GARDNER:
        e = torch.exp(-p1 * h)
        th, dth, K = tr + (ts - tr) * e, p1 * (ts - tr) * e, Ks * e
    else:
        m = 1 - 1 / p2
        t = (p1 * h) ** p2
        l1 = torch.log1p(t)
        Se = torch.exp(-m * l1)
        th, dth = tr + (ts - tr) * Se, (ts - tr) * m * p2 * (t / h) * Se / (1 + t)
        K = Ks * torch.exp(-p3 * m * l1) * torch.expm1(-m * torch.log1p(1 / t)) ** 2
    if want == "K":
        return torch.where(dry, K, Ks + torch.zeros_like(K))
    return torch.where(dry, th, ts + torch.zeros_like(th)), torch.where(dry, dth, torch.zeros_like(dth))


def _laws(sys, psi, want):
    if sys["index"] is None:
        return _theta_K(sys["mats"][0], psi, want)
    parts = [_theta_K(m, psi, want) for m in sys["mats"]]
    if want == "K":
        return sum(torch.where(sys["index"] == k, p, 0.0) for k, p in enumerate(parts))
    return tuple(sum(torch.where(sys["index"] == k, p[j], 0.0) for k, p in enumerate(parts)) for j in range(2))


def _sys_of(prob, dev):
    """The discrete problem's arrays, axis a on tensor dimension -1 - a."""
    dim, n = prob["dim"], prob["n"][:prob["dim"]]
    shape = tuple(n[::-1])
    put = lambda a: torch.as_tensor(np.array(a, dtype=np.float64), device=dev).reshape(shape)
    soil = prob["soil"]
    index = None
    if soil.get("materials"):
        mats = soil["materials"]
        index = torch.as_tensor(np.array(soil["material_index"]), device=dev).reshape(shape)
    else:
        mats = [dict(soil)]
        for k, f in (("Ks", "Ks_field"), ("p1", "p1_field"), ("p2", "p2_field")):
            if soil.get(f) is not None:
                mats[0][k] = put(soil[f])
    h = [prob["L"][a] / n[a] for a in range(dim)]
    faces = []                                            # (axis, side, kind, Dirichlet mask, value)
    for a in range(dim):
        fshape = tuple(1 if d == a else n[d] for d in range(dim))[::-1]
        for side in range(2):
            f = 2 * a + side
            b = prob["bc"]
            field = lambda x: torch.as_tensor(np.array(x, dtype=np.float64), device=dev).reshape(fshape)
            val = field(b["value_field"][f]) if b["value_field"][f] is not None else \
                torch.full(fshape, float(b["value"][f]), device=dev, dtype=torch.float64)
            mask = field(b["mask_field"][f]) != 0 if b["mask_field"][f] is not None else \
                torch.ones(fshape, device=dev, dtype=torch.bool)
            faces.append((a, side, b["kind"][f], mask, val))
    smax = torch.zeros(shape, device=dev, dtype=torch.float64)
    k = prob["sink"]
    if k["enabled"]:
        nv, v = n[dim - 1], dim - 1
        depth = torch.from_numpy(prob["L"][v] * (2.0 * (nv - 1 - np.arange(nv)) + 1.0) / (2.0 * nv)).to(dev)
        Z = k["root_decay"] * (1 - math.exp(-k["root_depth"] / k["root_decay"]))
        s = torch.where(depth <= k["root_depth"], k["Tp"] * torch.exp(-depth / k["root_decay"]) / Z, 0.0)
        smax += s.reshape([-1] + [1] * (dim - 1))
    return dict(dim=dim, mats=mats, index=index, h=h, faces=faces, smax=smax, sink=k, valid=None)


def _sink(sys, psi):
    k, s = sys["sink"], sys["smax"]
    if not k["enabled"]:
        return torch.zeros_like(psi), torch.zeros_like(psi)
    up, dn = (k["h1"] - psi) / (k["h1"] - k["h2"]), (psi - k["h4"]) / (k["h3"] - k["h4"])
    a = torch.where(psi >= k["h2"], up, torch.where(psi >= k["h3"], torch.ones_like(psi), dn))
    out = (psi >= k["h1"]) | (psi < k["h4"])
    da = torch.where(psi >= k["h2"], -1 / (k["h1"] - k["h2"]), torch.where(psi >= k["h3"], 0.0, 1 / (k["h3"] - k["h4"])))
    return torch.where(out, 0.0, a) * s, torch.where(out, 0.0, da) * s


def _end(t, a, side):
    return t.narrow(-1 - a, t.shape[-1 - a] - 1 if side else 0, 1)


def _assemble(sys, star):
    """Face conductances, Dirichlet diagonal and the gravity and boundary part of g."""
    K = _laws(sys, star, "K")
    g, db, links = torch.zeros_like(star), torch.zeros_like(star), []
    v = sys["dim"] - 1
    for a in range(sys["dim"]):
        h, n = sys["h"][a], star.shape[-1 - a]
        Kf = 0.5 * (K.narrow(-1 - a, 0, n - 1) + K.narrow(-1 - a, 1, n - 1))
        if sys["valid"] is not None:
            Kf = Kf * sys["valid"].narrow(-1 - a, 1, n - 1)
        links.append(Kf / (h * h))
        if a == v:
            g.narrow(-1 - a, 0, n - 1).add_(Kf / h)
            g.narrow(-1 - a, 1, n - 1).sub_(Kf / h)
    if sys["valid"] is not None:                          # columns: free drainage below, no flux above
        g[:, :1] -= K[:, :1] / sys["h"][0]
        return links, db, g
    for a, side, kind, mask, val in sys["faces"]:
        h, Ki = sys["h"][a], _end(K, a, side)
        if kind == W.DIRICHLET:
            full = torch.zeros_like(star)
            _end(full, a, side).copy_(val.expand_as(Ki))
            kb = torch.where(mask, 0.5 * (Ki + _end(_laws(sys, full, "K"), a, side)), 0.0)
            dz = (0.5 if side else -0.5) * h if a == v else 0.0
            _end(db, a, side).add_(2 * kb / (h * h))
            _end(g, a, side).add_(2 * kb / (h * h) * (val + dz))
        elif kind == W.FLUX:
            _end(g, a, side).add_(val / h)
        elif kind == W.FREE_DRAINAGE:
            _end(g, a, side).sub_(Ki / h)
    return links, db, g


def _flux(links, x):
    out = torch.zeros_like(x)
    for a, m in enumerate(links):
        n = x.shape[-1 - a]
        q = m * (x.narrow(-1 - a, 1, n - 1) - x.narrow(-1 - a, 0, n - 1))
        out.narrow(-1 - a, 0, n - 1).sub_(q)
        out.narrow(-1 - a, 1, n - 1).add_(q)
    return out


def _linear(links, D, r):
    """(diag(D) + M) x = r: the Thomas algorithm in 1-d, else Jacobi-preconditioned CG."""
    diag = D.clone()
    for a, m in enumerate(links):
        n = D.shape[-1 - a]
        diag.narrow(-1 - a, 0, n - 1).add_(m)
        diag.narrow(-1 - a, 1, n - 1).add_(m)
    if len(links) == 1:
        b, c, d = (t.cpu().numpy().reshape(-1, t.shape[-1]).T.copy() for t in (diag, -links[0], r))
        for i in range(1, len(b)):
            w = c[i - 1] / b[i - 1]
            b[i] -= w * c[i - 1]
            d[i] -= w * d[i - 1]
        d[-1] /= b[-1]
        for i in range(len(b) - 2, -1, -1):
            d[i] = (d[i] - c[i] * d[i + 1]) / b[i]
        return torch.from_numpy(np.ascontiguousarray(d.T)).to(r.device).reshape(r.shape)
    x, res = torch.zeros_like(r), r.clone()
    z = res / diag
    p, rz = z.clone(), (res * z).sum()
    stop = 1e-6 * res.abs().max()
    for k in range(20000):
        q = D * p + _flux(links, p)
        al = rz / (p * q).sum()
        x += al * p
        res -= al * q
        if k % 20 == 19 and res.abs().max() <= stop:
            break
        z = res / diag
        new = (res * z).sum()
        p = z + (new / rz) * p
        rz = new
    return x


def _solve_step(sys, psi, prev, dt, scheme, lag, opts):
    a = 1 / dt if scheme == 1 else 1.5 / dt
    th = _laws(sys, psi, "theta")[0]
    star = psi if scheme == 1 or lag else 2 * psi - prev
    hist = th / dt if scheme == 1 else (4 * th - _laws(sys, prev, "theta")[0]) / (2 * dt)
    links, db, g = _assemble(sys, star)
    g = g + hist
    x = psi.clone()

    def defect(x):
        t, dt_ = _laws(sys, x, "theta")
        S, dS = _sink(sys, x)
        r = g - (a * t + S + db * x + _flux(links, x))
        return (r if sys["valid"] is None else r * sys["valid"]), a * dt_ + dS + db

    r, D = defect(x)
    best = r.abs().max().item()
    for _ in range(60):
        if sys["valid"] is not None:
            D = torch.where(sys["valid"] > 0, D, torch.ones_like(D))
        dx = _linear(links, D, r)
        s = 1.0
        while True:
            y = x + s * dx
            ry, Dy = defect(y)
            now = ry.abs().max().item()
            if now < best or s < 1e-3:
                break
            s *= 0.5
        if not now < best:
            break
        fall, (x, r, D), best = now / best, (y, ry, Dy), now
        if fall > 0.5 and best / a < 1e-15:
            break
    return x


def exact(case, seed):
    kind, steps = case["kind"], case.get("steps", 1)
    if kind == "laws":
        prob = _laws_problem(case, seed)
        sys = _sys_of(prob, "cuda")
        psi = torch.as_tensor(np.array(prob["psi0"]), device="cuda").reshape(sys["smax"].shape)
        return [_laws(sys, psi, "theta")[0].reshape(-1), _laws(sys, psi, "K").reshape(-1)]
    if kind == "columns":
        probs = _columns_problems(case, seed)
        n = np.array([p["n"][0] for p in probs])
        if steps * int(n.max()) > 4200:
            return None
        col = lambda f: torch.tensor([f(p) for p in probs], dtype=torch.float64).reshape(-1, 1)
        i = torch.arange(int(n.max()))[None, :]
        valid = (i < torch.from_numpy(n)[:, None]).double()
        h = col(lambda p: p["L"][0] / p["n"][0])
        k = probs[0]["sink"]
        nn = torch.from_numpy(n)[:, None]
        depth = col(lambda p: p["L"][0]) * (2 * (nn - 1 - i) + 1).double() / (2 * nn).double()
        Z = k["root_decay"] * (1 - math.exp(-k["root_depth"] / k["root_decay"]))
        smax = torch.where((depth <= k["root_depth"]) & (valid > 0), k["Tp"] * torch.exp(-depth / k["root_decay"]) / Z,
                           0.0)
        mat = {q: col(lambda p, q=q: p["soil"][q]) for q in ("theta_s", "theta_r", "Ks", "p1", "p2", "p3", "p4")}
        sys = dict(dim=1, mats=[dict(mat, model=W.VANGENUCHTEN)], index=None, h=[h], smax=smax, sink=k, valid=valid)
        psi = torch.full(valid.shape, -1.0, dtype=torch.float64)
        for r, p in enumerate(probs):
            psi[r, :n[r]] = torch.from_numpy(p["psi0"])
        for _ in range(steps):
            psi = _solve_step(sys, psi, None, case["dt"], 1, 0, probs[0]["opts"])
        return psi[valid > 0]
    make = {"column": _column_problem, "plane": _plane_problem, "field": _field_problem}
    probs = _served_problems(case, seed) if kind == "served" else [make[kind](case, seed)]
    if sum(W.ncells(p) for p in probs) * steps > 2_400_000:
        return None
    out = []
    for prob in probs:
        sys = _sys_of(prob, "cpu" if kind == "column" else "cuda")
        put = lambda t: torch.as_tensor(np.array(t), device=sys["smax"].device).reshape(sys["smax"].shape)
        psi, prev = put(prob["psi0"]), None if prob.get("psi_prev") is None else put(prob["psi_prev"])
        for _ in range(steps):
            scheme = 2 if prob["scheme"] == 2 and prev is not None else 1
            psi, prev = _solve_step(sys, psi, prev, prob["dt"], scheme, prob["opts"]["bdf2_lag"], prob["opts"]), psi
        out.append(psi.reshape(-1))
    return out if kind == "served" else out[0]
