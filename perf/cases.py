"""The work this framework is measured on: what its users have it do, through its public calls.

A case is one pass of a job: rewrite the state of a box (from a velocity field, or from the
populations of a saved state), advance it some time steps, and read the result back (moments,
diagnostics, populations, spectrum). Everything stays on the GPU except the scalars that the
diagnostics return. A pass starts by rewriting the state, so every pass does the same work.

Results read from a box are handed on in the precision of its storage (a snapshot of an FP16
run is kept in FP16), FP64 results in FP64.
"""
import math

import torch

from paper_1507_02518_gb300 import lb, workloads

DEV = "cuda"
F64 = dict(dtype=torch.float64, device=DEV)
KEPT = {"f64": torch.float64, "f32": torch.float32, "f16": torch.float16}
SIZE = {"f64": 8, "f32": 4, "f16": 2}
# diagnostics whose value is not a difference of nearly equal sums
SCALARS = ("mass", "kinetic_energy", "enstrophy", "dissipation", "dudx2")
COUNTS = ("step", "nodes", "nonfinite_count")


def _box(name, n, storage, scheme, steps, begin, reads, **more):
    c = {"name": name, "kind": "run", "nx": n, "ny": n, "nz": n, "nu": 1e-3, "storage": storage,
         "scheme": scheme, "variant": "d+t+q", "gamma": "estimate", "flow": "modes",
         "steps": steps, "begin": begin, "reads": reads, "diag": 2}
    c.update(more)
    return c


def listed():
    return [
        # the reference workload of the method in FP64: a Taylor-Green vortex on 32^3, a few
        # steps at a time with diagnostics, as a parity or teaching run does
        _box("tg32_f64_pull", 32, "f64", "pull", 20, "field", "state", flow="tg"),
        # a small box stepped and monitored every 50 steps: launches and read-backs count
        _box("monitor32_f32_aa", 32, "f32", "aa", 50, "state", "moments"),
        # a box with odd edges (rows that are no multiple of anything), resumed from a saved
        # state and saved again; the smallest shear part
        _box("ragged_f32_aa", 151, "f32", "aa", 20, "state", "state", ny=89, nz=67,
             variant="d", diag=0),
        # the paper's Kida run A (N = 100, FP64): consistent initial state by the density
        # pre-solve, steps, 8th-order statistics
        _box("table2_kida100_f64_aa", 100, "f64", "aa", 20, "presolve", "moments", flow="kida",
             nu=100 * 0.05 / 6000.0, iters=32, diag=8),
        # isotropic turbulence on 256^3 in FP32, the headline run: resumed, 50 steps to the
        # next diagnostics, a snapshot
        _box("hit256_f32_pull", 256, "f32", "pull", 50, "state", "moments", flow="hit",
             nu=2e-4),
        # the same box in FP64: resumed, a few steps, saved
        _box("hit256_f64_pull", 256, "f64", "pull", 3, "state", "state", flow="hit", nu=2e-4,
             diag=0),
        # a large box in half-precision storage, in place (Kida vortex, 512^3), from its
        # initial velocity field to the first snapshot
        _box("kida512_f16_aa", 512, "f16", "aa", 20, "field", "moments", flow="kida", nu=5e-5),
        # an ensemble of boxes of uneven sizes and viscosities stepped together
        {"name": "ensemble24_f32_pull", "kind": "ensemble", "nbox": 24, "boxes": 20150702,
         "storage": "f32", "scheme": "pull", "variant": "d+t+q", "gamma": "estimate",
         "steps": 20},
        # the central-moment form of the method, resumed and saved
        _box("central192_f32_pull", 192, "f32", "pull", 20, "state", "state", flow="hit",
             nu=5e-4, variant="cd+ct+cq"),
        # the exact stabilizer per node and its distance from the estimate, in FP64
        _box("exact96_f64_pull", 96, "f64", "pull", 2, "state", "state", flow="hit",
             nu=5e-4, gamma="exact", gap=True, diag=0),
        # statistics of a decaying-turbulence run at a report time: 8th-order diagnostics and
        # the energy spectrum, no steps
        _box("spectra256_f32", 256, "f32", "pull", 0, "kept", "spectrum", flow="hit", nu=2e-4,
             diag=8),
        # the start of a run from a velocity field, saved after ten steps: the first steps from
        # equilibrium take the FP64 re-collision
        _box("start256_f32_aa", 256, "f32", "aa", 10, "field", "state", flow="hit", nu=2e-4),
    ]


def draw(rng):
    """A case of the ranges above: every storage and scheme, the shear parts and stabilizers
    in use, edges from 16 to 384 (odd ones among them), from a field, a state or a pre-solve."""
    def edge(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    pick = rng.random()
    storage = rng.choice(["f32", "f32", "f64", "f16"])
    scheme = rng.choice(["pull", "aa"])
    nu = math.exp(rng.uniform(math.log(5e-5), math.log(2e-3)))
    if pick < 0.10:
        return {"kind": "ensemble", "nbox": rng.randint(3, 24), "boxes": rng.randint(1, 10 ** 6),
                "storage": rng.choice(["f32", "f16"]), "scheme": scheme, "variant": "d+t+q",
                "gamma": "estimate", "steps": rng.randint(2, 30)}
    if pick < 0.20:
        c = _box("", edge(48, 288), rng.choice(["f32", "f64"]), scheme, 0, "kept", "spectrum",
                 nu=nu, diag=rng.choice([2, 8]))
    elif pick < 0.30:
        c = _box("", edge(24, 128), rng.choice(["f32", "f64"]), scheme, rng.randint(1, 3),
                 "state", "moments", nu=nu, gamma="exact", gap=True, diag=0)
    elif pick < 0.42:
        c = _box("", edge(24, 160), rng.choice(["f32", "f64"]), scheme, rng.randint(1, 20),
                 "presolve", "moments", nu=nu, flow="kida", iters=rng.choice([16, 32, 64]),
                 diag=rng.choice([2, 8]))
    else:
        c = _box("", edge(16, 384), storage, scheme, rng.randint(1, 40),
                 rng.choice(["field", "state", "state"]), rng.choice(["moments", "state"]),
                 nu=nu, variant=rng.choice(["d+t+q", "d+t+q", "d", "d+t", "cd+ct+cq"]),
                 gamma=rng.choice(["estimate", "estimate", "estimate", "lbgk"]),
                 diag=rng.choice([0, 2, 8]))
        if rng.random() < 0.5:  # a box with three different edges
            c["ny"], c["nz"] = edge(16, 288), edge(16, 288)
        limit = 1.0e9 if storage != "f64" else 5e7  # node updates of the largest listed case
        c["steps"] = max(1, min(c["steps"], int(limit / (c["nx"] * c["ny"] * c["nz"]))))
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _modes(nx, ny, nz, count, kmax, gen):
    """Solenoidal Fourier modes as (integer wave vector, amplitude, phase)."""
    out = []
    while len(out) < count:
        k = [int(v) for v in torch.randint(-kmax, kmax + 1, (3,), generator=gen)]
        k = [v if 4 * abs(v) <= n else 0 for v, n in zip(k, (nx, ny, nz))]
        if k == [0, 0, 0] or sum(v * v for v in k) > kmax * kmax:
            continue
        q = [2 * math.pi * v / n for v, n in zip(k, (nx, ny, nz))]
        a = [float(v) for v in torch.randn(3, generator=gen, dtype=torch.float64)]
        s = sum(x * y for x, y in zip(a, q)) / sum(x * x for x in q)
        ph = 2 * math.pi * float(torch.rand((), generator=gen, dtype=torch.float64))
        out.append((q, [x - s * y for x, y in zip(a, q)], ph))
    return out


def _mode_field(nx, ny, nz, urms, gen, count=16):
    """A smooth solenoidal velocity field of a few random large-scale modes."""
    x = torch.arange(nx, **F64).view(1, 1, nx)
    y = torch.arange(ny, **F64).view(1, ny, 1)
    z = torch.arange(nz, **F64).view(nz, 1, 1)
    u = torch.zeros((3, nz, ny, nx), **F64)
    for q, a, ph in _modes(nx, ny, nz, count, 4, gen):
        c = torch.cos(q[0] * x + q[1] * y + (q[2] * z + ph))
        for k in range(3):
            u[k].add_(c, alpha=a[k])
    u *= urms / math.sqrt(float(u.square().mean()))
    return u


def _field(case, seed):
    """u [3, nz, ny, nx] (density 1) of the case's flow."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    gen = torch.Generator().manual_seed(int(seed))
    flow = case["flow"]
    if flow == "hit":
        return workloads.random_spectrum_device(nx, 4.0, 0.04, seed, DEV)[1]
    if flow == "kida":  # the vortex with a small disturbance
        u = workloads.kida_device(nx, 0.05, DEV)[1]
        return u.add_(_mode_field(nx, ny, nz, 1e-3, gen, 4))
    if flow == "tg":
        u = torch.as_tensor(workloads.taylor_green(nx, 0.05)[1], **F64)
        return u.add_(_mode_field(nx, ny, nz, 1e-3, gen, 4))
    return _mode_field(nx, ny, nz, 0.04, gen)


def _roll(a, axis, k):
    """a shifted so that place x holds a(x + k) along x (0), y (1) or z (2)."""
    return torch.roll(a, -k, dims=a.dim() - 1 - axis)


def _state(case, u, seed):
    """Populations f [27, nz, ny, nx] of a flow under way at velocity u: equilibrium, the
    non-equilibrium part that the velocity gradients give, small higher moments."""
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 7)
    rho = 1.0 + 0.5 * (float((u * u).sum(0).mean()) - (u * u).sum(0))
    tau = 3.0 * case["nu"] + 0.5
    S = {}
    for a in range(3):
        for b in range(a, 3):
            S[a, b] = 0.25 * (_roll(u[a], b, 1) - _roll(u[a], b, -1)
                              + _roll(u[b], a, 1) - _roll(u[b], a, -1))
    ax = _axes(u)
    f = torch.empty((27,) + tuple(u.shape[1:]), **F64)
    for i, v in _velocities():
        f[i] = _feq(ax, v)
        neq = sum((v[a] * v[a] - 1.0 / 3.0) * S[a, a] for a in range(3))
        neq = neq + sum(2.0 * v[a] * v[b] * S[a, b] for a in range(3) for b in range(a + 1, 3)
                        if v[a] * v[b])
        noise = torch.randn(u.shape[1:], generator=gen, **F64)
        f[i] = rho * (f[i] - 3.0 * tau * _weight(v) * neq) + 5e-5 * _weight(v) * noise
    return f


# ---------------------------------------------------------------- the passes
def prepare(case, seed):
    s = {"case": case}
    if case["kind"] == "ensemble":
        boxes = workloads.batch_boxes(case["nbox"], case["boxes"])
        s["batch"] = lb.Batch(boxes, case["variant"], case["gamma"], case["storage"],
                              case["scheme"])
        s["f"], s["rho"], s["u"] = [], [], []
        for k, b in enumerate(boxes):
            c, n = {"nu": b["nu"]}, b["n"]
            gen = torch.Generator().manual_seed(int(seed) * 1000 + k)
            u = _mode_field(n, n, n, b["urms"], gen)
            s["f"].append(_state(c, u, int(seed) * 1000 + k))
            s["u"].append(torch.empty((3, n, n, n), **F64))
            s["rho"].append(torch.empty((n, n, n), **F64))
        return s
    lat = lb.Lattice(case["nx"], case["ny"], case["nz"], nu=case["nu"], variant=case["variant"],
                     gamma=case["gamma"], storage=case["storage"], scheme=case["scheme"])
    s["lat"] = lat
    if case["diag"]:
        lat.set_diag_order(case["diag"])
    u = _field(case, seed)
    if case["begin"] in ("state", "kept"):
        s["f"] = _state(case, u, seed)
    else:
        s["u0"] = u.contiguous()
    if case["reads"] == "state":
        s["out"] = torch.empty((27,) + lat.shape, **F64)
    else:
        s["rho"], s["u"] = torch.empty(lat.shape, **F64), torch.empty((3,) + lat.shape, **F64)
    if case["begin"] == "kept":
        lb.lb_set_populations(lat.ctx, s.pop("f").data_ptr(), True)
    return s


def _scalars(d, gamma=False):
    return {k: d[k] for k in SCALARS + COUNTS + (("gamma_mean",) if gamma else ())}


def run(s):
    case = s["case"]
    keep = KEPT[case["storage"]]
    if case["kind"] == "ensemble":
        batch = s["batch"]
        for k, f in enumerate(s["f"]):
            box = batch.box(k)
            lb.lb_set_time(box, 0)
            lb.lb_set_populations(box, f.data_ptr(), True)
        batch.step(case["steps"])
        ds = batch.diagnostics()
        for k in range(case["nbox"]):
            lb.lb_moments(batch.box(k), s["rho"][k].data_ptr(), s["u"][k].data_ptr(), True)
        return {"u": torch.cat([u.flatten() for u in s["u"]]).to(keep),
                "rho": torch.cat([r.flatten() for r in s["rho"]]).to(keep),
                "diag": {k: torch.tensor([d[k] for d in ds])
                         for k in SCALARS + COUNTS + ("gamma_mean",)}}
    lat, out = s["lat"], {}
    if case["begin"] == "state":
        lb.lb_set_time(lat.ctx, 0)
        lb.lb_set_populations(lat.ctx, s["f"].data_ptr(), True)
    elif case["begin"] == "field":
        lat.init_field(None, s["u0"])
    elif case["begin"] == "presolve":
        out["iters"], _ = lat.presolve(s["u0"], max_iters=case["iters"], tol=-1.0)
    if case["steps"]:
        lat.step(case["steps"])
    if case["diag"]:
        out["diag"] = _scalars(lat.diagnostics(), case["steps"] > 0)
    if case.get("gap"):
        g = lat.stabilizer_gap()
        out["gap"] = {k: g[k] for k in ("nodes", "mean_abs", "mean_estimate", "mean_exact")}
    if case["reads"] == "state":
        lb.lb_get_populations(lat.ctx, s["out"].data_ptr(), True)
        out["f"] = s["out"].to(keep)
        return out
    if case["reads"] == "spectrum":
        out["E"] = lat.spectrum()
    lb.lb_moments(lat.ctx, s["rho"].data_ptr(), s["u"].data_ptr(), True)
    out["rho"], out["u"] = s["rho"].to(keep), s["u"].to(keep)
    return out


def work(case):
    """Bytes: every input and output once, and the populations read and written once a step
    (a step of the boxes measured here does not stay on the chip). Operations: those of the
    moments, the equilibrium, the entropic products and the relaxation per node."""
    if case["kind"] == "ensemble":
        P = sum(b["n"] ** 3 for b in workloads.batch_boxes(case["nbox"], case["boxes"]))
    else:
        P = case["nx"] * case["ny"] * case["nz"]
    v = 27 * SIZE[case["storage"]]
    begin = case.get("begin", "state")
    reads = case.get("reads", "moments")
    nbytes = case["steps"] * 2 * v * P
    nbytes += {"state": 27 * 8 + v, "field": 24 + v, "kept": 0, "presolve": 24 + v}[begin] * P
    nbytes += case.get("iters", 0) * 2 * v * P
    nbytes += (27 * 8 + v if reads == "state" else 32 + v) * P
    if case.get("diag", 2):
        nbytes += v * P
    if case.get("gap"):
        nbytes += v * P
    flops = case["steps"] * 600 * P + case.get("iters", 0) * 250 * P + 100 * P
    if case["gamma"] == "exact":
        flops += (case["steps"] + 1) * 3 * 27 * 20 * P
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits
def _velocities():
    return [(i, (i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1)) for i in range(27)]


def _weight(v):
    return math.prod(2.0 / 3.0 if c == 0 else 1.0 / 6.0 for c in v)


def _axes(u):
    """Per axis the three factors of the product-form equilibrium (velocities -1, 0, +1)."""
    out = []
    for a in range(3):
        R = torch.sqrt(1.0 + 3.0 * u[a] * u[a])
        out.append([(2.0 * R - 1.0 - 3.0 * u[a]) / 6.0, 2.0 * (2.0 - R) / 3.0,
                    (2.0 * R - 1.0 + 3.0 * u[a]) / 6.0])
    return out


def _feq(ax, v):
    return ax[0][v[0] + 1] * ax[1][v[1] + 1] * ax[2][v[2] + 1]


def _moments(f):
    rho = sum(f[i] for i in range(27))
    j = [sum(v[a] * f[i] for i, v in _velocities() if v[a]) for a in range(3)]
    return rho, torch.stack([j[a] / rho for a in range(3)])


def _shear(dev, u, case):
    """Delta s of the deviations f - f_eq: the moments of the shear part, transformed back
    axis by axis (about u for the central-moment variants)."""
    var = case["variant"]
    central, with_t, with_q = var.startswith("c"), "t" in var, "q" in var

    def m(p, q, r):
        return sum((v[0] ** p) * (v[1] ** q) * (v[2] ** r) * dev[i] for i, v in _velocities()
                   if (v[0] or not p) and (v[1] or not q) and (v[2] or not r))
    M = {k: m(*k) for k in ((2, 0, 0), (0, 2, 0), (0, 0, 2), (1, 1, 0), (1, 0, 1), (0, 1, 1))}
    if with_q:
        for k in ((1, 2, 0), (1, 0, 2), (2, 1, 0), (0, 1, 2), (2, 0, 1), (0, 2, 1)):
            M[k] = m(*k)
            if central:  # rho and u are conserved: lower moments of dev vanish
                one, two = k.index(1), k.index(2)
                e2 = tuple(2 if a == two else 0 for a in range(3))
                e11 = tuple(1 if a in (one, two) else 0 for a in range(3))
                M[k] = M[k] - 2.0 * u[two] * M[e11] - u[one] * M[e2]
        M[1, 1, 1] = m(1, 1, 1)
        if central:
            M[1, 1, 1] = M[1, 1, 1] - u[0] * M[0, 1, 1] - u[1] * M[1, 0, 1] - u[2] * M[1, 1, 0]
    if not with_t:
        tr = (M[2, 0, 0] + M[0, 2, 0] + M[0, 0, 2]) / 3.0
        for k in ((2, 0, 0), (0, 2, 0), (0, 0, 2)):
            M[k] = M[k] - tr

    def coef(a, v, p):  # 1D inverse: the weight of moment p in the population of velocity v
        w = u[a] if central else 0.0
        if v == 0:
            return (1.0 - w * w, -2.0 * w, -1.0)[p]
        return (w * (w + v) / 2.0, v / 2.0 + w, 0.5)[p]
    ds = []
    for _, v in _velocities():
        acc = 0.0
        for k, val in M.items():
            cs = [coef(a, v[a], k[a]) for a in range(3)]
            if any(isinstance(c, float) and c == 0.0 for c in cs):
                continue
            acc = acc + cs[0] * cs[1] * cs[2] * val
        ds.append(acc if torch.is_tensor(acc) else torch.zeros_like(u[0]))
    return ds


def _gammas(f, case, exact):
    """(ds, dh, gamma estimate, gamma) of the collision of f."""
    beta = 1.0 / (6.0 * case["nu"] + 1.0)
    rho, u = _moments(f)
    ax = _axes(u)
    eq = [rho * _feq(ax, v) for _, v in _velocities()]
    dev = [f[i] - eq[i] for i in range(27)]
    ds = _shear(dev, u, case)
    dh = [dev[i] - ds[i] for i in range(27)]
    if case["gamma"] == "lbgk":
        two = torch.full_like(rho, 2.0)
        return beta, ds, dh, two, two
    num = sum(ds[i] * dh[i] / eq[i] for i in range(27))
    den = sum(dh[i] * dh[i] / eq[i] for i in range(27))
    est = torch.where(den > 1e-300, 1.0 / beta - (2.0 - 1.0 / beta) * num / den, 2.0)
    if not exact:
        return beta, ds, dh, est, est
    g = est.clone()
    for _ in range(12):
        val = der = 0.0
        for i in range(27):
            x = ((1.0 - beta * g) * dh[i] - (2.0 * beta - 1.0) * ds[i]) / eq[i]
            val = val + dh[i] * torch.log1p(x)
            der = der - beta * dh[i] * dh[i] / (eq[i] * (1.0 + x))
        g = g - val / der
    return beta, ds, dh, est, g


def _steps(f, case, n):
    """n time steps on the list f of 27 planes, in place; the mean gamma of the last one."""
    nz = f[0].shape[0]
    chunk = max(1, int(2 ** 24 // (f[0].shape[1] * f[0].shape[2])))
    mean = 0.0
    for step in range(n):
        total = 0.0
        for z in range(0, nz, chunk):
            part = [p[z:z + chunk] for p in f]
            beta, ds, dh, _, g = _gammas(part, case, case["gamma"] == "exact")
            for i in range(27):
                part[i] -= beta * (2.0 * ds[i] + g * dh[i])
            total += float(g.sum())
            del ds, dh, g
        mean = total / f[0].numel()
        for i, v in _velocities():
            if v != (0, 0, 0):
                f[i].copy_(torch.roll(f[i], (v[2], v[1], v[0]), dims=(0, 1, 2)))
    return mean


def _exact_diag(rho, u, case, gamma, steps):
    order = case.get("diag", 2)
    cs = (0.5,) if order == 2 else (4.0 / 5.0, -1.0 / 5.0, 4.0 / 105.0, -1.0 / 280.0)
    G = [[sum(c * (_roll(u[a], b, k + 1) - _roll(u[a], b, -k - 1)) for k, c in enumerate(cs))
          for b in range(3)] for a in range(3)]
    curl = (G[2][1] - G[1][2], G[0][2] - G[2][0], G[1][0] - G[0][1])
    d = {"mass": float(rho.sum()),
         "kinetic_energy": 0.5 * sum(float((u[a] - u[a].mean()).square().mean())
                                     for a in range(3)),
         "enstrophy": 0.5 * sum(float(c.square().mean()) for c in curl),
         "dissipation": 0.5 * case["nu"] * sum(float((G[a][b] + G[b][a]).square().mean())
                                               for a in range(3) for b in range(3)),
         "dudx2": float(G[0][0].square().mean()), "step": steps, "nodes": rho.numel(),
         "nonfinite_count": 0}
    if gamma is not None:
        d["gamma_mean"] = gamma
    return d


def _exact_presolve(u, iters):
    """The pre-solve at its default relaxation: f <- S f_eq(rho(f), u) (beta_pre = 1/2)."""
    ax = _axes(u)
    f = [_feq(ax, v).clone() for _, v in _velocities()]
    for _ in range(iters):
        rho = sum(f)
        for i, v in _velocities():
            f[i] = torch.roll(rho * _feq(ax, v), (v[2], v[1], v[0]), dims=(0, 1, 2))
    return f


def _exact_spectrum(u):
    n = u.shape[-1]
    k = torch.fft.fftfreq(n, d=1.0 / n, **F64)
    kr = torch.fft.rfftfreq(n, d=1.0 / n, **F64)
    K2 = k.view(n, 1, 1) ** 2 + k.view(1, n, 1) ** 2 + kr.view(1, 1, -1) ** 2
    shell = torch.round(torch.sqrt(K2)).to(torch.int64)
    w = torch.full((1, 1, kr.numel()), 2.0, **F64)
    w[..., 0] = 1.0
    if n % 2 == 0:
        w[..., -1] = 1.0
    nb = int(math.sqrt(3.0) * n / 2.0) + 2
    E = torch.zeros(nb, **F64)
    for a in range(3):
        e = 0.5 * w * (torch.fft.rfftn(u[a]) / float(n) ** 3).abs().square()
        E.index_add_(0, shell.flatten(), e.flatten())
    E[0] = 0.0
    return E.cpu().numpy()


def exact(case, seed):
    if case["kind"] == "ensemble":
        boxes = workloads.batch_boxes(case["nbox"], case["boxes"])
        us, rs, ds = [], [], []
        for k, b in enumerate(boxes):
            c = dict(case, nu=b["nu"])
            gen = torch.Generator().manual_seed(int(seed) * 1000 + k)
            u = _mode_field(b["n"], b["n"], b["n"], b["urms"], gen)
            f = list(_state(c, u, int(seed) * 1000 + k))
            mean = _steps(f, c, case["steps"])
            rho, u = _moments(f)
            us.append(u.flatten())
            rs.append(rho.flatten())
            ds.append(_exact_diag(rho, u, c, mean, case["steps"]))
        return {"u": torch.cat(us), "rho": torch.cat(rs),
                "diag": {k: torch.tensor([d[k] for d in ds], dtype=torch.float64)
                         if k in SCALARS + ("gamma_mean",) else torch.tensor([d[k] for d in ds])
                         for k in SCALARS + COUNTS + ("gamma_mean",)}}
    u = _field(case, seed)
    out = {}
    if case["begin"] in ("state", "kept"):
        f = list(_state(case, u, seed))
    elif case["begin"] == "field":
        ax = _axes(u)
        f = [_feq(ax, v).clone() for _, v in _velocities()]
        del ax
    else:
        out["iters"] = case["iters"]
        f = _exact_presolve(u, case["iters"])
    del u
    mean = _steps(f, case, case["steps"])
    if case.get("gap"):
        _, _, _, est, g = _gammas(f, case, True)
        out["gap"] = {"nodes": est.numel(), "mean_abs": float((est - g).abs().mean()),
                      "mean_estimate": float(est.mean()), "mean_exact": float(g.mean())}
    if case["reads"] == "state":
        if case["diag"]:
            out["diag"] = _exact_diag(*_moments(f), case, mean, case["steps"])
        out["f"] = torch.stack(f)
        return out
    rho, u = _moments(f)
    del f
    if case["diag"]:
        out["diag"] = _exact_diag(rho, u, case, mean if case["steps"] else None, case["steps"])
    if case["reads"] == "spectrum":
        out["E"] = _exact_spectrum(u)
    out["rho"], out["u"] = rho, u
    return out
