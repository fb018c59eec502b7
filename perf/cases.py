"""The calls by which the framework's speed is measured.

Each case is one thing a user of the stochastic-collocation LBM path has it do
through its public entry points (`sclbm.Ensemble`, `sclbm.InflowLoss`): advance
an ensemble and reduce it, reduce 121 samples to gPC coefficients, bound a
profile by quantiles, average in time, export a flow field with its vortices,
differentiate a run.  Sizes and physics are those of `workloads.py` and of the
smoke run, or smaller and larger members of the same families; geometry, wind
and probes are drawn from the seed.  `exact` restates what a call computes in
64-bit torch and numpy, from the definitions alone.
"""
import math

import numpy as np
import torch

from paper_2508_18202_gb300 import sclbm as S

VEL, OUT, BB, FS = S.SC_BC_VELOCITY, S.SC_BC_OUTFLOW, S.SC_BC_BOUNCE_BACK, S.SC_BC_FREE_SLIP
FACES = {"urban": [VEL, OUT, VEL, VEL, BB, FS],       # inlet, outlet, wind on the sides, ground, sky
         "channel": [VEL, OUT, BB, BB, BB, BB],
         "disk": [VEL, VEL, VEL, VEL, BB, FS]}        # the paper's cylinder: wind on the whole mantle
RULES = {"gl": S.SC_Q_GL, "cc": S.SC_Q_CC_SMOLYAK, "gh": S.SC_Q_GH}
PRECISIONS = {"fp64": S.SC_P_FP64_PLAIN, "fp32": S.SC_P_FP32_SHIFT, "bf16": S.SC_P_BF16_STORE,
              "fp16": S.SC_P_FP16_STORE}
BYTES = {"fp64": 8, "fp32": 4, "bf16": 2, "fp16": 2}
L2_BYTES = 129e6        # an ensemble smaller than this stays on the chip between time levels
FLOPS_PER_UPDATE = 300  # collision of one cell (BGK + Smagorinsky; the regularized one about 500)

_BASE = dict(kind="run", faces="urban", prec="fp32", coll="bgk", c_smag=0.14, tau0=0.50096, rule="cc", inputs=2,
             level=3, nodes=0, degree=2, ramp=100, warm=200, steps=20, series=False, exact=True)


def _case(name, **over):
    return dict(_BASE, name=name, **over)


def listed():
    return [
        # the smallest whole call: the smoke run's ensemble (odd sizes, 3 samples), stepped and reduced; an
        # interactive check, a unit test, one iterate of an outer loop
        _case("small_urban", nx=45, ny=21, nz=14, rule="gl", inputs=1, tau0=0.56, ramp=4, warm=25, steps=25),
        # the reference precision on the channel with a cube: validation runs are made this way
        _case("channel_fp64", nx=48, ny=24, nz=24, faces="channel", prec="fp64", c_smag=0.0, tau0=0.6, rule="gl",
              inputs=1, level=5, degree=4, ramp=0, warm=50, steps=100),
        # the ordinary ensemble: the urban LES block, 13 Smolyak samples, between two output times
        _case("les_fp32", nx=256, ny=128, nz=64, exact=False),
        # the same ensemble in the storage that halves its memory
        _case("les_bf16", nx=256, ny=128, nz=64, prec="bf16", exact=False),
        # uneven districts advanced together in one handle, each reduced by itself
        _case("batched_uneven", nx=128, ny=64, nz=48, nx2=192, ny2=96, nz2=64, level2=4, nx3=320, ny3=160, nz3=64,
              level3=2, warm=100, exact=False),
        # the largest: one wave of the large ensemble (12 of its 69 samples, 16.8 M cells each)
        _case("large_wave", nx=512, ny=256, nz=128, tau0=0.50192, inputs=3, level=4, nodes=12, ramp=20, warm=40,
              steps=8, exact=False),
        # the paper's model: circular domain, regularized collision, Gaussian inputs, hourly wind that turns
        _case("disk_series", nx=120, ny=120, nz=40, faces="disk", coll="rr", c_smag=0.25, tau0=0.5000013, rule="gh",
              level=5, degree=5, ramp=10, warm=60, steps=16, series=True),
        # the paper's reduction: 121 samples to mean, spread and 21 Hermite coefficients, at an odd level
        _case("gpc_121", kind="moments", nx=96, ny=96, nz=40, faces="disk", coll="rr", c_smag=0.25, tau0=0.5000013,
              rule="gh", level=11, degree=5, ramp=8, warm=61, steps=0),
        # the running time average of |u|, sampled between steps and reduced over the samples
        _case("time_average", kind="average", nx=192, ny=96, nz=64, warm=50, steps=3),
        # one sample's velocity and vortices for a figure
        _case("vortices", kind="fields", nx=256, ny=128, nz=64, rule="gl", inputs=1, ramp=20, warm=60, steps=0),
        # confidence bounds of probe columns and a layer's patch from the gPC surrogate
        _case("quantile_bands", kind="quantiles", nx=64, ny=64, nz=16, rule="gh", level=3, degree=5, cells=4096,
              samples=4096),
        # one gradient of the probe misfit for the assimilation of the inflow
        _case("adjoint", kind="adjoint", nx=128, ny=64, nz=48, rule="gl", inputs=1, level=1, degree=-1, c_smag=0.0,
              tau0=0.6, ramp=0, warm=0, steps=300, probes=16),
    ]


def draw(rng):
    def size(lo, hi, odd=True):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return max(lo, n if odd and rng.random() < 0.5 else n // 8 * 8)

    kind = rng.choice(["run", "run", "run", "run", "disk", "moments", "average", "fields", "quantiles", "adjoint"])
    c = dict(_BASE)
    if kind == "run":
        prec = rng.choice(["fp32", "fp32", "bf16", "fp16", "fp64"])
        top = (128, 64, 40) if prec == "fp64" else (384, 192, 80)
        c.update(nx=size(32, top[0]), ny=size(20, top[1]), nz=size(12, top[2]), prec=prec, level=rng.choice([2, 3, 3]),
                 inputs=rng.choice([1, 2, 2, 3]), rule=rng.choice(["cc", "gl"]), warm=2 * rng.randint(10, 40), ramp=15,
                 coll=rng.choice(["bgk", "bgk", "bgk", "rr"]), tau0=rng.choice([0.50096, 0.51, 0.56]),
                 series=rng.random() < 0.2, faces=rng.choice(["urban", "urban", "channel"]))
        if rng.random() < 0.25 and prec != "fp64":
            c.update(nx2=size(32, 160), ny2=size(20, 96), nz2=c["nz"], level2=2)
        updates = 7e7 if prec == "fp64" else 1.4e9  # no more work than the largest listed case
        c["steps"] = 2 * max(4, min(rng.randint(4, 25), int(updates / 2 / _cells(c))))
    elif kind in ("disk", "moments"):
        n = size(48, 200)
        c.update(kind="run" if kind == "disk" else "moments", nx=n, ny=n, nz=size(14, 48), faces="disk", coll="rr",
                 c_smag=0.25, rule="gh", level=rng.choice([3, 5, 7] if kind == "disk" else [3, 5, 7, 11]),
                 degree=rng.choice([2, 3, 5]), ramp=8, warm=rng.randint(20, 60), steps=16 if kind == "disk" else 0,
                 series=kind == "disk", prec=rng.choice(["fp32", "fp32", "bf16"]))
    elif kind == "average":
        c.update(kind="average", nx=size(64, 256), ny=size(32, 128), nz=size(16, 64), warm=rng.randint(10, 30),
                 steps=rng.randint(1, 6), prec=rng.choice(["fp32", "fp32", "fp16"]))
    elif kind == "fields":
        c.update(kind="fields", nx=size(64, 512), ny=size(32, 256), nz=size(16, 96), rule="gl", inputs=1, ramp=20,
                 warm=rng.randint(20, 60), steps=0, prec=rng.choice(["fp32", "fp32", "bf16"]))
    elif kind == "quantiles":
        c.update(kind="quantiles", nx=64, ny=64, nz=16, rule=rng.choice(["gh", "gl"]), degree=rng.choice([2, 3, 5]),
                 cells=size(40, 8000), samples=size(200, 8192))
    else:
        c.update(kind="adjoint", nx=size(48, 160), ny=size(24, 80), nz=size(16, 56), rule="gl", inputs=1, level=1,
                 degree=-1, c_smag=0.0, tau0=rng.choice([0.56, 0.6, 0.8]), ramp=0, warm=0,
                 steps=rng.randint(40, 400), probes=rng.choice([1, 4, 16, 40]))
    cells = _cells(c) * max(1, c.get("steps", 0) + c.get("warm", 0))
    c["exact"] = c["kind"] == "quantiles" or cells < 2.5e9
    return c


# ------------------------------------------------------------ the problem of a case
def _domains(case):
    """(nx, ny, nz, quadrature level) of each domain of a case."""
    D = [(case["nx"], case["ny"], case["nz"], case["level"])]
    for k in "23":
        if "nx" + k in case:
            D.append((case["nx" + k], case["ny" + k], case["nz" + k], case["level" + k]))
    return D


def _inputs(case):
    """Kinds and ranges of the uncertain inputs (Gaussian: mean and standard deviation)."""
    if case["rule"] == "gh":
        return [S.SC_IN_SPEED_REL, S.SC_IN_ANGLE_DEG][: case["inputs"]], [0.0, 0.0], [0.1, 6.0]
    return ([S.SC_IN_SPEED_REL, S.SC_IN_ALPHA, S.SC_IN_ANGLE_DEG][: case["inputs"]], [-0.15, 0.15, -10.0],
            [0.15, 0.35, 10.0])


def _boxes(case, seed, d, nx, ny, nz):
    """Blocks standing on the ground: footprints of 8 to 24 cells where they fit, as in the synthetic districts."""
    rng = np.random.RandomState((seed * 8 + d) % (1 << 31))
    if case["faces"] == "channel":
        x, y = nx // 4 + rng.randint(0, 3), ny // 3 + rng.randint(0, 3)
        return [[x, y, 0, x + max(2, nx // 6), y + max(2, ny // 3), max(2, nz // 2)]]
    count = 2 if case["faces"] == "disk" else max(1, round(24 * nx * ny / (256 * 128)))
    boxes = []
    for _ in range(count):
        w, l = (min(rng.randint(8, 25), max(2, n // 4)) for n in (nx, ny))
        h = min(rng.randint(10, 41), max(2, 2 * nz // 3))
        lo = (nx // 3, ny // 3) if case["faces"] == "disk" else (nx // 8, 2)
        hi = (2 * nx // 3, 2 * ny // 3) if case["faces"] == "disk" else (nx - nx // 8, ny - 2)
        x, y = rng.randint(lo[0], max(lo[0] + 1, hi[0] - w)), rng.randint(lo[1], max(lo[1] + 1, hi[1] - l))
        boxes.append([int(v) for v in (x, y, 0, min(x + w, nx - 2), min(y + l, ny - 2), h)])
    return boxes


def _wind(case, seed):
    """Nominal speed, exponent and direction of the inflow, and the hourly targets of its series."""
    rng = np.random.RandomState((seed * 8 + 7) % (1 << 31))
    u = (0.02 if case["faces"] == "disk" else 0.05) * (1 + 0.1 * rng.uniform(-1, 1))
    w = dict(u_ref=float(u), alpha=float(rng.uniform(0.2, 0.3)), angle=float(rng.uniform(-5, 5)),
             speed=1 + 0.2 * rng.uniform(-1, 1, 4096), turn=np.cumsum(rng.uniform(-20, 20, 4096)), per=16, interp=4)
    w["speed"][0], w["turn"][0] = 1.0, 0.0
    return w


def _config(case, seed):
    kinds, lo, hi = _inputs(case)
    w = _wind(case, seed)
    doms = [dict(nx=nx, ny=ny, nz=nz, boxes=_boxes(case, seed, d, nx, ny, nz), bc=FACES[case["faces"]],
                 quad_level=level, disk_radius=nx / 2 if case["faces"] == "disk" else 0.0)
            for d, (nx, ny, nz, level) in enumerate(_domains(case))]
    gauss = case["rule"] == "gh"
    return S.Config(doms, case["tau0"], case["c_smag"], w["u_ref"], w["alpha"], kinds, lo[: len(kinds)],
                    hi[: len(kinds)], RULES[case["rule"]], PRECISIONS[case["prec"]], ramp_steps=case["ramp"],
                    angle_deg=w["angle"], gpc_degree=case["degree"],
                    collision=S.SC_COLL_RR if case["coll"] == "rr" else S.SC_COLL_BGK,
                    profile=S.SC_PROFILE_LOG if gauss else S.SC_PROFILE_POWER,
                    time_average=int(case["kind"] == "average"), node_count=case["nodes"])


def _node_count(case, level):
    if case["nodes"]:
        return case["nodes"]
    if case["rule"] != "cc":
        return level ** case["inputs"]
    return len(_smolyak(case["inputs"], level)[1])


def _cells(case):
    """Cells times samples of all domains (the cells outside a disk do not count)."""
    share = math.pi / 4 if case["faces"] == "disk" else 1.0
    return sum(share * nx * ny * nz * _node_count(case, level) for nx, ny, nz, level in _domains(case))


def _terms(case):
    return math.comb(case["degree"] + case["inputs"], case["inputs"]) if case["degree"] >= 0 else 0


def _surrogate(case, seed):
    """Coefficients of a field's surrogate (falling with the degree), cells, samples and probabilities."""
    rng = np.random.RandomState(seed % (1 << 31))
    P, n = _terms(case), case["nx"] * case["ny"] * case["nz"]
    degree = np.array([sum(e) for e in _exponents(case["inputs"], case["degree"])])
    coef = rng.standard_normal((P, n)) * (0.004 * 0.3 ** degree)[:, None]
    coef[0] = 0.05 + 0.01 * rng.standard_normal(n)
    cells = np.sort(rng.choice(n, case["cells"], replace=False)).astype(np.int32)
    shape = (case["samples"], case["inputs"])
    samples = rng.standard_normal(shape) if case["rule"] == "gh" else rng.uniform(-1, 1, shape)
    return coef, cells, samples, [0.025, 0.5, 0.975]


def _columns(nx, ny):
    """Two probe columns within reach of the wind."""
    return [[nx // 2, min(8, ny // 4)], [3 * nx // 4, ny // 2]]


def _probes(case, seed):
    """Fluid probe points and the velocities measured there."""
    rng = np.random.RandomState((seed * 8 + 5) % (1 << 31))
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    solid = _flags(case, seed, 0).reshape(nz, ny, nx)
    pts = []
    while len(pts) < case["probes"]:
        x, y, z = int(rng.randint(nx // 8, nx)), int(rng.randint(0, ny)), int(rng.randint(0, nz - 2))
        if not solid[z, y, x] and [x, y, z] not in pts:
            pts.append([x, y, z])
    z = np.array(pts)[:, 2]
    target = np.zeros((case["probes"], 3))
    target[:, 0] = 0.055 * ((z + 0.5) / nz) ** 0.28 * (1 + 0.1 * rng.standard_normal(case["probes"]))
    target[:, 1] = 0.002 * rng.standard_normal(case["probes"])
    return pts, target


# ------------------------------------------------------------ what is measured
def prepare(case, seed):
    cfg = _config(case, seed)
    ens = S.Ensemble(cfg)
    s = dict(case=case, ens=ens)
    if case["kind"] == "quantiles":
        coef, s["cells"], s["samples"], s["q"] = _surrogate(case, seed)
        s["coef"] = torch.from_numpy(coef).cuda()
        return s
    if case["kind"] == "adjoint":
        points, target = _probes(case, seed)
        w = _wind(case, seed)
        s["assim"] = S.Assimilation(ens, points, target, case["steps"])
        s["theta"] = torch.tensor([w["u_ref"], w["alpha"]], dtype=torch.float32)
        s["loss"] = S.InflowLoss()
        return s
    if case["series"]:
        w = _wind(case, seed)
        ens.set_inflow_series(w["speed"], w["turn"], w["per"], w["interp"])
    ens.step(case["warm"])
    if case["kind"] == "run":
        s["probes"] = [_columns(nx, ny) for nx, ny, _, _ in _domains(case)]
    return s


def run(s):
    case, ens, kind = s["case"], s["ens"], s["case"]["kind"]
    if kind == "run":
        ens.step(case["steps"])
        return [_reduced(ens.moments(d, probes=p, gpc=True)) + [ens.velocity(d, 0)] for d, p in enumerate(s["probes"])]
    if kind == "moments":
        return _reduced(ens.moments(0, gpc=True))
    if kind == "average":
        ens.step(case["steps"])
        S.sc_lbm_average_add(ens.h)
        return _reduced(ens.average_moments(0, gpc=True)) + [ens.average_field(0, 0)]
    if kind == "fields":
        u = ens.velocity(0, 0)
        return [u, ens.qcriterion(0, u)]
    if kind == "quantiles":
        return [ens.gpc_quantiles(0, s["coef"], s["cells"], s["samples"], s["q"])]
    theta = s["theta"].clone().requires_grad_(True)
    loss = s["loss"].apply(theta, s["assim"])
    loss.backward()
    return [loss.detach(), theta.grad]


def _reduced(out):
    return [out[k] for k in ("mean", "std", "coef", "prof") if out[k] is not None]


def work(case):
    """Bytes and operations of one pass: populations in and out at each level (once for all levels where the
    ensemble stays on the chip), read once by each reduction, results written once."""
    kind, size, cells = case["kind"], BYTES[case["prec"]], _cells(case)
    if kind == "quantiles":
        n, m, P = case["cells"], case["samples"], _terms(case)
        return dict(bytes=8 * (n * P + m * P + 3 * n), flops=2 * n * m * P)
    if kind == "adjoint":
        # forward, recomputed forward and reverse sweep; the states of a segment stay on the chip
        return dict(bytes=4 * 19 * cells * (2 + 2 * math.isqrt(case["steps"])), flops=900 * cells * case["steps"])
    points = sum(nx * ny * nz for nx, ny, nz, _ in _domains(case))
    state = 19 * size * cells
    moved = state * 2 * (1 if state < L2_BYTES and case["steps"] else case["steps"])
    flops = FLOPS_PER_UPDATE * cells * case["steps"] + (40 + 2 * _terms(case)) * cells
    out = (8 * (2 + _terms(case)) + (12 if kind == "run" else 0)) * points
    if kind == "fields":
        one = case["nx"] * case["ny"] * case["nz"]
        return dict(bytes=one * (19 * size + 12 + 4), flops=100 * one)
    if kind == "average":
        return dict(bytes=moved + state + 16 * cells + out + 8 * points, flops=flops)
    return dict(bytes=moved + (state if state >= L2_BYTES or not case["steps"] else 0) + out, flops=flops)


# ------------------------------------------------------------ the same in 64 bits
C = np.array([[0, 0, 0], [1, 0, 0], [-1, 0, 0], [0, 1, 0], [0, -1, 0], [0, 0, 1], [0, 0, -1], [1, 1, 0], [-1, -1, 0],
              [1, -1, 0], [-1, 1, 0], [1, 0, 1], [-1, 0, -1], [1, 0, -1], [-1, 0, 1], [0, 1, 1], [0, -1, -1],
              [0, 1, -1], [0, -1, 1]])
OPP = [int(np.flatnonzero((C == -c).all(1))[0]) for c in C]
WEIGHTS = np.array([[1 / 3, 1 / 18, 1 / 36][int(c @ c)] for c in C])


def _flags(case, seed, d):
    """0 fluid, 1 building, 2 outside the mantle of the disk."""
    nx, ny, nz, _ = _domains(case)[d]
    f = np.zeros((nz, ny, nx), np.int8)
    for x0, y0, z0, x1, y1, z1 in _boxes(case, seed, d, nx, ny, nz):
        f[z0:z1, y0:y1, x0:x1] = 1
    if case["faces"] == "disk":
        x, y = np.arange(nx) + 0.5 - nx / 2, np.arange(ny) + 0.5 - ny / 2
        f[:, (x[None] ** 2 + y[:, None] ** 2) > (nx / 2) ** 2] = 2
    return f.reshape(-1)


def _exponents(d, degree):
    """Multi-indices of total degree <= degree, by degree, then the first exponent descending."""
    def of(d, total):
        if d == 1:
            return [(total,)]
        return [(a,) + r for a in range(total, -1, -1) for r in of(d - 1, total - a)]
    return [e for g in range(degree + 1) for e in of(d, g)]


def _basis(rule, exponents, s):
    """Orthonormal Legendre (uniform inputs) or Hermite (normal inputs) products at the points s [n][d]."""
    degree = max(sum(e) for e in exponents)
    if rule == "gh":
        one = [np.polynomial.hermite_e.hermeval(s, [0] * k + [1]) / math.sqrt(math.factorial(k))
               for k in range(degree + 1)]
    else:
        one = [math.sqrt(2 * k + 1) * np.polynomial.legendre.legval(s, [0] * k + [1]) for k in range(degree + 1)]
    return np.stack([np.prod([one[k][:, t] for t, k in enumerate(e)], axis=0) for e in exponents], axis=1)


def _clenshaw_curtis(level):
    m = 1 if level == 1 else 2 ** (level - 1) + 1
    if m == 1:
        return np.zeros(1), np.ones(1)
    k = np.arange(m)
    x = -np.cos(np.pi * k / (m - 1))
    V = np.polynomial.legendre.legvander(x, m - 1).T
    moments = np.zeros(m)
    moments[0] = 1.0
    return x, np.linalg.solve(V, moments)


def _smolyak(d, level):
    """Nodes in [-1, 1]^d and weights of the Clenshaw-Curtis sparse grid."""
    found = {}
    for flat in np.ndindex(*(level,) * d):
        lv = [i + 1 for i in flat]
        e = level + d - 1 - sum(lv)
        if not 0 <= e <= d - 1:
            continue
        rules = [_clenshaw_curtis(i) for i in lv]
        for k in np.ndindex(*(len(r[0]) for r in rules)):
            key = tuple(round(float(r[0][i]), 12) for r, i in zip(rules, k))
            w = (-1) ** e * math.comb(d - 1, e) * float(np.prod([r[1][i] for r, i in zip(rules, k)]))
            found[key] = found.get(key, 0.0) + w
    keys = sorted(found)
    return np.array(keys), np.array([found[k] for k in keys])


def _samples(case, level):
    """Standard coordinates [n][d] and weights of the collocation nodes."""
    d = case["inputs"]
    if case["rule"] == "cc":
        return _smolyak(d, level)
    x, w = np.polynomial.legendre.leggauss(level) if case["rule"] == "gl" else np.polynomial.hermite_e.hermegauss(level)
    w = w / w.sum()
    grid = np.stack(np.meshgrid(*[x] * d, indexing="ij"), -1).reshape(-1, d)
    weights = np.prod(np.stack(np.meshgrid(*[w] * d, indexing="ij"), -1).reshape(-1, d), axis=1)
    return grid, weights


def _inflow(case, seed, s, nz):
    """Inflow velocity [nz][3] of the sample with standard coordinates s."""
    kinds, lo, hi = _inputs(case)
    w = _wind(case, seed)
    xi, alpha, angle = 0.0, w["alpha"], w["angle"]
    for t, k in enumerate(kinds):
        v = lo[t] + hi[t] * s[t] if case["rule"] == "gh" else 0.5 * (lo[t] + hi[t]) + 0.5 * (hi[t] - lo[t]) * s[t]
        if k == S.SC_IN_SPEED_REL:
            xi = v
        elif k == S.SC_IN_ALPHA:
            alpha = v
        else:
            angle = v
    h = np.arange(nz) + 0.5
    shape = np.log((h + 0.1) / 0.1) / math.log((nz + 0.1) / 0.1) if case["rule"] == "gh" else (h / nz) ** alpha
    u = w["u_ref"] * (1 + xi) * shape
    t = math.radians(angle)
    return np.stack([u * math.cos(t), u * math.sin(t), 0 * u], axis=1)


def _factor(case, seed, m):
    """Turn (radians) and scale of the inflow at time level m: start-up ramp times the hourly series."""
    r = 0.5 * (1 - math.cos(math.pi * min(m, case["ramp"]) / case["ramp"])) if case["ramp"] else 1.0
    if not case["series"]:
        return 0.0, r
    w = _wind(case, seed)
    k, o = min(m // w["per"], len(w["speed"]) - 1), m % w["per"]
    if k == 0:
        return 0.0, r * w["speed"][0]
    lam = min(o, w["interp"]) / w["interp"] if m // w["per"] == k else 1.0
    at = lambda v: v[k - 1] + lam * (v[k] - v[k - 1])  # noqa: E731
    return math.radians(at(w["turn"])), r * at(w["speed"])


class _Links:
    """Where each population comes from: its source slot, and the links that add the moving-wall term."""

    def __init__(self, case, seed, d, device):
        nx, ny, nz, _ = _domains(case)[d]
        self.n, self.nz = nx * ny * nz, nz
        flags = _flags(case, seed, d)
        faces = FACES[case["faces"]]
        z, y, x = (a.reshape(-1) for a in np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij"))
        own = np.arange(self.n)
        source, moving = np.zeros((19, self.n), np.int64), np.zeros((19, self.n), bool)
        where = {tuple(c): i for i, c in enumerate(C)}
        for i, c in enumerate(C):
            p = [x - c[0], y - c[1], z - c[2]]
            out = [(p[a] < 0) | (p[a] >= n) for a, n in enumerate((nx, ny, nz))]
            face = [np.where(p[a] < 0, faces[2 * a], faces[2 * a + 1]) for a in range(3)]
            crossed = sum(o.astype(int) for o in out)
            inside = [np.clip(p[a], 0, n - 1) for a, n in enumerate((nx, ny, nz))]

            def at(cells):
                return cells[0] + nx * (cells[1] + ny * cells[2])

            def kind(k):
                return sum(((out[a] & (face[a] == k)).astype(int) for a in range(3)))

            back, src = OPP[i] * self.n + own, np.zeros(self.n, np.int64)
            to = at(inside)
            src = i * self.n + to                                        # streams from the neighbour
            bounce = (crossed == 0) & (flags[to] == 1)
            move = (crossed == 0) & (flags[to] == 2)
            bounce |= kind(BB) > 0
            move |= (crossed > 0) & (kind(BB) == 0) & (kind(VEL) > 0)
            rest = (crossed > 0) & ~bounce & ~move
            single = rest & (crossed == 1)
            # zero-gradient outlet: the transverse neighbour's population, the own one next to a building
            side = at([x, inside[1], inside[2]])
            src = np.where(single & (kind(OUT) == 1), i * self.n + np.where(flags[side] == 0, side, own), src)
            # free-slip lid: mirrored from the in-plane neighbour
            mirror = where[(c[0], c[1], -c[2])]
            plane = at([inside[0], inside[1], z])
            lid = single & (kind(FS) == 1)
            src = np.where(lid, mirror * self.n + plane, src)
            bounce |= lid & (flags[plane] == 1)
            move |= lid & (flags[plane] == 2)
            src = np.where(rest & (crossed == 2), mirror * self.n + own, src)   # outlet and lid at once
            source[i] = np.where(bounce | move, back, src)
            moving[i] = move
        self.fluid = torch.from_numpy(flags == 0).to(device)
        source[:, flags != 0] = (np.arange(19)[:, None] * self.n + own)[:, flags != 0]
        moving[:, flags != 0] = False
        self.source = torch.from_numpy(source.reshape(-1)).to(device)
        slot = np.flatnonzero(moving.reshape(-1))
        self.slot = torch.from_numpy(slot).to(device)
        self.slot_dir, self.slot_z = slot // self.n, z[slot % self.n]


def _hermite_tables(device):
    c = C.astype(float)
    eye = np.eye(3)
    H2 = np.einsum("ia,ib->iab", c, c) - eye / 3
    H3 = np.einsum("ia,ib,ig->iabg", c, c, c) - (np.einsum("ia,bg->iabg", c, eye) + np.einsum("ib,ag->iabg", c, eye)
                                                 + np.einsum("ig,ab->iabg", c, eye)) / 3
    pairs = [((0, 0, 1), (1, 2, 2)), ((0, 2, 2), (0, 1, 1)), ((1, 1, 2), (0, 0, 2))]
    rows, index = [], []
    for sign in (1, -1):
        for a, b in pairs:
            h = H3[(slice(None),) + a] + sign * H3[(slice(None),) + b]
            rows.append(h / (WEIGHTS @ h ** 2))
            index.append((a, b, sign))
    t = lambda v: torch.as_tensor(np.asarray(v), device=device)  # noqa: E731
    return t(H2.reshape(19, 9)), t(np.stack(rows, 1)), index


def _collide(f, case, tables, c, w):
    """Post-collision populations of f [..., 19, n] (float64 or complex128)."""
    rho = f.sum(-2, keepdim=True)
    u = torch.einsum("ia,...in->...an", c, f) / rho
    cu = torch.einsum("ia,...an->...in", c, u)
    usq = (u * u).sum(-2, keepdim=True)
    feq = w[:, None] * rho * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * usq)
    tau = case["tau0"]
    if not case["c_smag"] and case["coll"] == "bgk":
        return f - (f - feq) / tau
    # non-equilibrium stress against the second-order equilibrium
    pi = torch.einsum("iab,...in->...abn", torch.einsum("ia,ib->iab", c, c), f - feq)
    if case["c_smag"]:
        norm = torch.sqrt(2 * (pi * pi).sum((-3, -2)) + 1e-30)[..., None, :]
        tau = 0.5 * (tau + torch.sqrt(tau * tau + 18 * case["c_smag"] ** 2 * norm / rho))
    if case["coll"] == "bgk":
        return f - (f - feq) / tau
    H2, H3, index = tables
    keep = 1 - 1 / tau

    def third(a, b, g):
        eq = rho[..., 0, :] * u[..., a, :] * u[..., b, :] * u[..., g, :]
        ne = u[..., a, :] * pi[..., b, g, :] + u[..., b, :] * pi[..., a, g, :] + u[..., g, :] * pi[..., a, b, :]
        return eq + keep[..., 0, :] * ne

    k3 = torch.stack([third(*a) + sign * third(*b) for a, b, sign in index], -2)
    v = 4.5 * torch.einsum("ik,...kn->...in", H2, pi.flatten(-3, -2)) * keep
    return feq + w[:, None] * (v + torch.einsum("ik,...kn->...in", H3, k3))


class _Flow:
    """Populations of some samples of one domain, advanced from rest in 64 bits."""

    def __init__(self, case, seed, d, uin, links, device, dtype=torch.float64):
        self.case, self.seed, self.L = case, seed, links
        self.tables = _hermite_tables(device)
        self.c = torch.as_tensor(C, device=device).to(dtype)
        self.w = torch.as_tensor(WEIGHTS, device=device).to(dtype)
        uin = torch.as_tensor(uin, device=device).to(dtype)               # [samples][nz][3]
        self.wall = uin[:, torch.as_tensor(links.slot_z, device=device)]  # [samples][moving links][3]
        dirs = torch.as_tensor(links.slot_dir, device=device)
        self.slot_c, self.slot_w = self.c[dirs], 6 * self.w[dirs]
        self.f = self.w[:, None].expand(19, links.n).repeat(uin.shape[0], 1, 1)
        self.level = 0

    def step(self, n):
        for _ in range(n):
            post = _collide(self.f, self.case, self.tables, self.c, self.w).flatten(1)
            self.level += 1
            turn, scale = _factor(self.case, self.seed, self.level)
            ux = math.cos(turn) * self.wall[..., 0] - math.sin(turn) * self.wall[..., 1]
            uy = math.sin(turn) * self.wall[..., 0] + math.cos(turn) * self.wall[..., 1]
            term = self.slot_w * scale * (self.slot_c[:, 0] * ux + self.slot_c[:, 1] * uy
                                          + self.slot_c[:, 2] * self.wall[..., 2])
            f = post[:, self.L.source]
            f[:, self.L.slot] += term
            self.f = f.view(self.f.shape)

    def velocity(self):
        u = torch.einsum("ia,sin->san", self.c, self.f) / self.f.sum(1, keepdim=True)
        return u * self.L.fluid


def _speeds(case, seed, d, steps, device):
    """|u| [samples][n] of domain d after `steps`, the first sample's velocity, the coordinates and the weights."""
    nx, ny, nz, level = _domains(case)[d]
    s, a = _samples(case, level)
    links = _Links(case, seed, d, device)
    q = torch.empty(len(a), links.n, dtype=torch.float64, device=device)
    group, first = max(1, int(2.5e7 // links.n)), None
    for b in range(0, len(a), group):
        flow = _Flow(case, seed, d, np.stack([_inflow(case, seed, v, nz) for v in s[b:b + group]]), links, device)
        flow.step(steps)
        u = flow.velocity()
        q[b:b + group] = u.square().sum(1).sqrt()
        first = u[0].clone() if first is None else first
    return q, first, s, torch.as_tensor(a, device=device)


def _statistics(case, q, s, a):
    mean = torch.einsum("s,sn->n", a, q) / a.sum()
    std = (torch.einsum("s,sn->n", a, (q - mean) ** 2) / a.sum()).clamp_min(0).sqrt()
    phi = torch.as_tensor(_basis(case["rule"], _exponents(case["inputs"], case["degree"]), s), device=q.device)
    return mean, std, torch.einsum("s,sp,sn->pn", a, phi, q)


def exact(case, seed):
    if not case["exact"]:
        return None
    device = "cuda" if torch.cuda.is_available() else "cpu"
    kind = case["kind"]
    if kind == "quantiles":
        return [_exact_quantiles(case, seed, device)]
    if kind == "adjoint":
        return _exact_adjoint(case, seed, device)
    if kind == "fields":
        return _exact_fields(case, seed, device)
    results = []
    for d, (nx, ny, nz, _) in enumerate(_domains(case)):
        q, first, s, a = _speeds(case, seed, d, case["warm"] + case["steps"], device)
        mean, std, coef = _statistics(case, q, s, a)
        out = [mean, std, coef]
        if kind == "run":
            columns = [(m.view(nz, ny, nx)[:, y, x], v.view(nz, ny, nx)[:, y, x])
                       for m, v, (x, y) in ((mean, std, p) for p in _columns(nx, ny))]
            out += [torch.stack([torch.stack([m, v, m - 1.959963984540054 * v, m + 1.959963984540054 * v], -1)
                                 for m, v in columns]), first]
        results.append(out)
    if kind == "average":
        return results[0] + [q[0]]
    return results if kind == "run" else results[0]


def _exact_quantiles(case, seed, device):
    coef, cells, samples, probabilities = _surrogate(case, seed)
    phi = torch.as_tensor(_basis(case["rule"], _exponents(case["inputs"], case["degree"]), samples), device=device)
    y = (torch.as_tensor(coef[:, cells], device=device).T @ phi.T).sort(dim=1).values
    ranks = [min(max(math.ceil(p * case["samples"]), 1), case["samples"]) for p in probabilities]
    return torch.stack([y[:, k - 1] for k in ranks])


def _exact_fields(case, seed, device):
    nx, ny, nz, level = _domains(case)[0]
    links = _Links(case, seed, 0, device)
    s, _ = _samples(case, level)
    flow = _Flow(case, seed, 0, _inflow(case, seed, s[0], nz)[None], links, device)
    flow.step(case["warm"])
    u = flow.velocity()[0]
    fluid, v = links.fluid.view(nz, ny, nx), u.view(3, nz, ny, nx)
    J = torch.zeros(3, 3, nz, ny, nx, dtype=u.dtype, device=u.device)
    for a, dim in enumerate((2, 1, 0)):  # x, y, z
        def shifted(t, k, dim):
            return torch.roll(t, -k, dim)
        n = fluid.shape[dim]
        index = torch.arange(n, device=u.device).view([-1 if i == dim else 1 for i in range(3)])
        up = shifted(fluid, 1, dim) & (index < n - 1)
        down = shifted(fluid, -1, dim) & (index > 0)
        hi = torch.where(up, shifted(v, 1, dim + 1), v)
        lo = torch.where(down, shifted(v, -1, dim + 1), v)
        J[:, a] = (hi - lo) * torch.where(up & down, 0.5, 1.0)
    sym, skew = (J + J.transpose(0, 1)) / 2, (J - J.transpose(0, 1)) / 2
    q = 0.5 * (skew.square().sum((0, 1)) - sym.square().sum((0, 1))) * fluid
    return [u, q.reshape(-1)]


def _exact_adjoint(case, seed, device):
    """Loss and gradient by complex steps of the inflow's speed and exponent: exact to rounding."""
    nx, ny, nz, _ = _domains(case)[0]
    links = _Links(case, seed, 0, device)
    points, target = _probes(case, seed)
    at = torch.as_tensor([x + nx * (y + ny * z) for x, y, z in points], device=device)
    w = _wind(case, seed)
    u_ref, alpha = (float(np.float32(v)) for v in (w["u_ref"], w["alpha"]))
    turn, h, eps = math.radians(w["angle"]), (np.arange(nz) + 0.5) / nz, 1e-30
    both = []
    for du, da in ((eps, 0.0), (0.0, eps)):
        u = (u_ref + 1j * du) * h ** (alpha + 1j * da)
        both.append(np.stack([u * math.cos(turn), u * math.sin(turn), 0 * u], 1))
    flow = _Flow(case, seed, 0, np.stack(both), links, device, torch.complex128)
    flow.step(case["steps"])
    f = flow.f[:, :, at]
    v = torch.einsum("ia,sin->sna", flow.c, f) / f.sum(1)[..., None]
    J = ((v - torch.as_tensor(target, device=device)) ** 2).sum((1, 2))
    return [J[0].real, J.imag / eps]
