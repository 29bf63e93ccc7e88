"""The solver's work as its users call it, case by case, for timing.

Every case is one call of a public entry point (`Plan.solve`, `Batch.solve`, `Plan.gradient`,
`ccmf_solve_static`) on a seeded periodic cell with a fixed number of ADMM updates (or a
tolerance below the precision's reach and a maximum number of updates), so that a pass is the
same amount of work on every input. The cells are the kinds that the studies, tests and
benchmarks of this repository solve: a single ball, Boolean balls, short fibres, pores of
vanishing resistance, 2-D disks, a lognormal field; they are stamped on the GPU so that making
them is quick.
"""

import ctypes
import math

import numpy as np
import torch

from paper_2103_05968_gb300 import ccmf

DEV = "cuda"
RULES = {"bb": ccmf.CCMF_RHO_BB, "const": ccmf.CCMF_RHO_CONST, "ltd": ccmf.CCMF_RHO_LTD, "rb": ccmf.CCMF_RHO_RB}
H = math.sqrt(0.5)


def _solve(name, cell, n, solves=1, precision="fp32", iters=20, tol=0.0, rule="bb", delta=0.25, fields=True):
    c = {"kind": "solve", "cell": cell, "n1": n[0], "n2": n[1], "n3": n[2], "solves": solves, "precision": precision,
         "iters": iters, "tol": tol, "rule": rule, "delta": delta, "fields": fields}
    return dict(c, name=name) if name else c


def _batch(name, grids, realisations, persistent, iters):
    c = {"kind": "batch", "cell": "polyballs", "grids": grids, "realisations": realisations, "precision": "fp32",
         "persistent": persistent, "iters": iters, "rule": "bb", "delta": 0.25, "tol": 0.0}
    return dict(c, name=name) if name else c


def _gradient(name, n, iters, every):
    c = {"kind": "gradient", "cell": "lognormal", "n1": n[0], "n2": n[1], "n3": n[2], "solves": 1,
         "precision": "fp32", "iters": iters, "every": every, "rule": "bb", "delta": 0.25, "tol": 0.0}
    return dict(c, name=name) if name else c


def _static(name, cell, n, precision, iters):
    c = {"kind": "static", "cell": cell, "n1": n[0], "n2": n[1], "n3": n[2], "solves": 1, "precision": precision,
         "iters": iters, "rule": "bb", "delta": 0.25, "tol": 0.0}
    return dict(c, name=name) if name else c


def listed():
    return [
        # the validation cell: one ball, double precision, stopped by a residual that it is too early to meet,
        # so that the host looks at the counter every 32 updates as a tolerance run does
        _solve("ball 32^3 fp64 tol", "ball", (32, 32, 32), precision="fp64", iters=96, tol=1e-9),
        # the 2-D penalty study: a flat cell, double precision, undamped
        _solve("disks 128^2 fp64", "disks", (128, 128, 1), precision="fp64", iters=64, delta=0.5),
        # a single small cell, the size of a realisation in a statistical study
        _solve("balls 64^3", "balls", (64, 64, 64), iters=24),
        # axis lengths with odd factors, an odd number of voxels along z, two normals
        _solve("balls 90x100x75 x2", "balls", (90, 100, 75), solves=2),
        # the anisotropy study: one fibre cell, several normals as one batch
        _solve("fibres 96^3 x6", "fibres", (96, 96, 96), solves=6),
        # the usual cell: 128^3 overlapping balls, three normals
        _solve("balls 128^3 x3", "balls", (128, 128, 128), solves=3),
        # the same cell in double precision, the reference for stated errors
        _solve("balls 128^3 fp64", "balls", (128, 128, 128), precision="fp64", iters=6),
        # the porosity study: pores of vanishing resistance
        _solve("pores 256^3", "pores", (256, 256, 256), iters=8),
        # the large fibre cell
        _solve("fibres 512^3", "fibres", (512, 512, 512), iters=10),
        # realisations on uneven grids with three normals each, as one graph and as one persistent launch
        _batch("uneven batch graph", "64,96,128,160", 8, False, 12),
        _batch("uneven batch persistent", "64,96,128,160", 8, True, 12),
        # d gamma_eff / d gamma, double-precision forward and single-precision reverse sweep
        _gradient("gradient 80^3", (80, 80, 80), 12, 6),
    ]


# axis lengths with factors 2, 3, 5
_SMOOTH = sorted(2 ** a * 3 ** b * 5 ** c for a in range(10) for b in range(6) for c in range(4)
                 if 12 <= 2 ** a * 3 ** b * 5 ** c <= 640)


def _axis(rng, side):
    x = side * math.exp(rng.uniform(-0.4, 0.4))
    return min(_SMOOTH, key=lambda n: abs(math.log(n / x)))


def draw(rng):
    kind = rng.choice(["solve"] * 6 + ["batch", "persistent", "gradient", "static"])
    if kind in ("batch", "persistent"):
        grids = sorted(rng.sample([48, 60, 64, 80, 90, 96, 100, 120, 128, 144, 160], rng.randint(2, 4)))
        return _batch(None, ",".join(str(x) for x in grids), rng.randint(3, 10), kind == "persistent",
                      rng.randint(6, 14))
    if kind == "gradient":
        side = math.exp(rng.uniform(math.log(32), math.log(90)))
        return _gradient(None, [_axis(rng, side) for _ in range(3)], rng.randint(8, 14), rng.randint(4, 7))
    if kind == "static":
        side = math.exp(rng.uniform(math.log(14), math.log(38)))
        return _static(None, rng.choice(["ball", "balls", "pores"]), [_axis(rng, side) for _ in range(3)],
                       rng.choice(["fp32", "fp32", "fp64"]), rng.randint(12, 32))
    fp64 = rng.random() < 0.25
    side = math.exp(rng.uniform(math.log(16), math.log(110 if fp64 else 400)))
    n = [_axis(rng, side) for _ in range(3)]
    cell = rng.choice(["ball", "balls", "balls", "fibres", "pores"])
    if rng.random() < 0.1:
        n, cell = [max(n), max(n), 1], "disks"
    vox = n[0] * n[1] * n[2]
    solves = rng.choice([s for s in (1, 1, 2, 3, 6, 8) if s * vox <= (2e6 if fp64 else 1.2e8) or s == 1])
    iters = rng.randint(8, 24 if fp64 else 16)
    iters = max(4, min(iters, int((1.2e7 if fp64 else 1.3e9) / (vox * solves))))
    if not fp64 and cell in ("ball", "pores") and max(n) > 120:
        # one large soft region: the potential's jump, and with it the rounding of a single-precision field,
        # grows with the cell and the updates
        cell, iters = ("balls", iters) if max(n) > 270 else (cell, min(iters, 10))
    rule = rng.choice(["bb"] * 5 + ["const", "ltd", "rb"])
    return _solve(None, cell, n, solves=solves, precision="fp64" if fp64 else "fp32", iters=iters,
                  tol=1e-9 if rng.random() < 0.3 else 0.0, rule=rule, delta=rng.choice([0.25, 0.25, 0.5]),
                  fields=rng.random() < 0.7)


# ---- cells -------------------------------------------------------------------------------

def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _ball_offsets(radius):
    r = int(math.ceil(radius))
    ax = torch.arange(-r, r + 1, device=DEV)
    o = torch.stack(torch.meshgrid(ax, ax, ax, indexing="ij"), -1).reshape(-1, 3)
    return o[(o * o).sum(-1) < radius * radius]


def _stamp(mask, centres, radius):
    """Marks the voxels of the periodic balls around the integer centres [M, 3]."""
    n = torch.tensor(mask.shape, device=DEV)
    off = _ball_offsets(radius)
    for c in centres.split(max(1, 20_000_000 // len(off))):
        p = (c[:, None, :] + off[None]) % n
        mask[p[..., 0], p[..., 1], p[..., 2]] = True


def _cell(kind, n, seed):
    """gamma [n1, n2, n3] in double, on the GPU."""
    g = torch.Generator(device=DEV).manual_seed(int(seed))
    nt = torch.tensor(n, device=DEV, dtype=torch.float64)
    vox = n[0] * n[1] * n[2]
    mask = torch.zeros(n, dtype=torch.bool, device=DEV)
    if kind == "ball":
        _stamp(mask, (_rand(g, 1, 3) * nt).long(), max(1.5, min(n) / 4.0))
        return torch.where(mask, 0.1, 1.0).double()
    if kind == "balls":       # radius 6, 20 % of the volume, weak inclusions
        r = min(6.0, max(1.5, min(n) / 8.0))
        count = max(1, round(-math.log(0.8) * vox / (4.0 / 3.0 * math.pi * r ** 3)))
        _stamp(mask, (_rand(g, count, 3) * nt).long(), r)
        return torch.where(mask, 0.3, 1.0).double()
    if kind == "polyballs":   # radii 4 .. 8
        for r in (4.0, 5.0, 6.0, 7.0, 8.0):
            count = max(1, round(0.045 * vox / (4.0 / 3.0 * math.pi * r ** 3)))
            _stamp(mask, (_rand(g, count, 3) * nt).long(), r)
        return torch.where(mask, 0.2, 1.0).double()
    if kind == "pores":       # 25 %, no resistance in the pores
        r = max(1.5, min(n) / 16.0)
        count = max(1, round(-math.log(0.75) * vox / (4.0 / 3.0 * math.pi * r ** 3)))
        _stamp(mask, (_rand(g, count, 3) * nt).long(), r)
        return torch.where(mask, 0.0, 1.0).double()
    if kind == "fibres":      # diameter 6, aspect ratio 20, 12 %, tough
        d = min(6.0, max(2.5, min(n) / 8.0))
        length = min(20.0 * d, 0.9 * max(n))
        count = max(1, round(-math.log(0.88) * vox / (math.pi * d * d / 4.0 * length)))
        mid, a = _rand(g, count, 1, 3) * nt, torch.randn(count, 1, 3, generator=g, device=DEV, dtype=torch.float64)
        t = torch.linspace(-0.5, 0.5, int(length * 1.5), device=DEV, dtype=torch.float64)[None, :, None]
        _stamp(mask, (mid + a / a.norm(dim=-1, keepdim=True) * t * length).round().long().reshape(-1, 3), d / 2)
        return torch.where(mask, 3.0, 1.0).double()
    if kind == "disks":       # flat cell, 40 % of tough disks
        r = n[0] / 12.0
        ii, jj = (torch.arange(n[a], device=DEV, dtype=torch.float64) for a in (0, 1))
        for c in _rand(g, 23, 2) * nt[:2]:
            di, dj = ((ii - c[0] + n[0] / 2) % n[0] - n[0] / 2), ((jj - c[1] + n[1] / 2) % n[1] - n[1] / 2)
            mask[..., 0] |= di[:, None] ** 2 + dj[None, :] ** 2 < r * r
        return torch.where(mask, 10.0, 1.0).double()
    # lognormal: exp(0.5 g), correlation length 8
    k2 = sum((torch.fft.fftfreq(m, device=DEV, dtype=torch.float64) ** 2).reshape([-1 if a == b else 1 for b in range(3)])
             for a, m in enumerate(n))
    white = torch.fft.fftn(torch.randn(n, generator=g, device=DEV, dtype=torch.float64))
    f = torch.fft.ifftn(white * torch.exp(-(math.pi * 8.0) ** 2 * k2)).real
    return torch.exp(0.5 * (f - f.mean()) / f.std())


def _normals(count, seed, flat):
    """e1, e2, e3 first, then the directions of a golden-angle spiral, turned by the seed; on a flat cell,
    directions in its plane."""
    if flat:
        t = [math.pi * (k / count + 0.05 * (seed % 7)) for k in range(count)]
        return [[math.cos(x), math.sin(x), 0.0] for x in t]
    out = [[1.0, 0.0, 0.0], [0.0, 1.0, 0.0], [0.0, 0.0, 1.0]]
    if count == 1:
        return [out[seed % 3]]
    for k in range(3, count):
        z = 1.0 - (k - 2.5) / max(1, count - 3)
        p = math.pi * (3.0 - math.sqrt(5.0)) * k + 0.1 * (seed % 7)
        out.append([math.sqrt(1.0 - z * z) * math.cos(p), math.sqrt(1.0 - z * z) * math.sin(p), z])
    return out[:count]


# ---- inputs and passes -------------------------------------------------------------------

def _types(case):
    return (ccmf.CCMF_FP64, torch.float64) if case["precision"] == "fp64" else (ccmf.CCMF_FP32_MIXED, torch.float32)


def _members(case):
    """(grid, cell number, normal) of every solve of a batch."""
    grids = [int(x) for x in case["grids"].split(",")]
    return [((grids[r % len(grids)],) * 3, r, a) for r in range(case["realisations"]) for a in range(3)]


def _rho0(case, gamma):
    """The study's lower bound for a constant penalty; a start off the tie |z| = min gamma where a rule divides
    by |e| or the branch of the projection is differentiated."""
    if case["rule"] == "const":
        return float(gamma[gamma > 0].min())
    return 0.9 * float(gamma[gamma > 0].min()) if case["rule"] == "ltd" or case["kind"] == "gradient" else 0.0


def _params(case, gamma):
    p = dict(delta=case["delta"], rho_rule=RULES[case["rule"]], rho0=_rho0(case, gamma))
    if case["tol"] > 0:
        return ccmf.Params(tol=case["tol"], max_iter=case["iters"], **p)
    return ccmf.Params(fixed_iters=case["iters"], **p)


def prepare(case, seed):
    prec, dt = _types(case)
    st = {"case": case, "dtype": dt}
    if case["kind"] == "batch":
        cells = {}
        for grid, r, _ in _members(case):
            if r not in cells:
                cells[r] = _cell(case["cell"], grid, seed * 100 + r).to(dt)
        st["gammas"] = [cells[r] for _, r, _ in _members(case)]
        st["normals"] = np.eye(3)[[a for _, _, a in _members(case)]]
        st["params"] = _params(case, st["gammas"][0])
        st["plan"] = ccmf.Batch([grid for grid, _, _ in _members(case)], precision=prec, device=DEV)
        st["plan"].set_persistent(case["persistent"])
        return st
    n = (case["n1"], case["n2"], case["n3"])
    st["gamma"] = _cell(case["cell"], n, seed).to(dt)
    st["normals"] = _normals(case["solves"], seed, case["n3"] == 1)
    st["params"] = _params(case, st["gamma"])
    if case["kind"] != "static":
        st["plan"] = ccmf.Plan(n, batch=case["solves"], precision=prec, device=DEV)
    if case["kind"] == "gradient":
        st["plan"].set_adjoint_forward(ccmf.CCMF_FP64)
    return st


_NUMBERS = ("gamma_eff", "gamma_primal", "residual", "mean_v_norm", "rho")


def _numbers(results, dt):
    out = {k: torch.tensor([r[k] for r in results], dtype=dt) for k in _NUMBERS}
    out.update({k: torch.tensor([r[k] for r in results]) for k in ("iters", "converged", "status")})
    return out


def run(state):
    case, dt = state["case"], state["dtype"]
    if case["kind"] == "batch":
        return _numbers(state["plan"].solve(state["gammas"], state["normals"], state["params"]), dt)
    if case["kind"] == "gradient":
        grad, res, rho = state["plan"].gradient(state["gamma"], state["normals"], case["iters"], case["every"],
                                                state["params"])
        return dict(_numbers(res, dt), grad=grad, schedule=rho)
    if case["kind"] == "static":
        prec, _ = _types(case)
        n, g = (case["n1"], case["n2"], case["n3"]), state["gamma"]
        flow, cut = (torch.empty((c, *n), dtype=dt, device=DEV) for c in (3, 6))
        res = ccmf.ccmf_result()
        code = ccmf.ccmf_solve_static(*n, prec, ctypes.c_void_p(g.data_ptr()), state["normals"][0],
                                      state["params"].to_c(), ctypes.c_void_p(flow.data_ptr()),
                                      ctypes.c_void_p(cut.data_ptr()), ctypes.byref(res),
                                      ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))
        if code != ccmf.CCMF_OK:
            raise ccmf.CCMFError(code, "ccmf_solve_static")
        one = {f[0]: getattr(res, f[0]) for f in ccmf.ccmf_result._fields_}
        return dict(_numbers([one], dt), flow=flow[None], cut=cut[None])
    res, flow, cut = state["plan"].solve(state["gamma"], state["normals"], state["params"], want_flow=case["fields"],
                                         want_cut=case["fields"])
    out = _numbers(res, dt)
    if case["fields"]:
        out.update(flow=flow, cut=cut)
    return out


def work(case):
    """Bytes: the state between two updates has to be read and written once an update, with gamma read once. Both
    fields of the state are functions of the six components of z = v + rho xi, of gamma and of rho, so that is 13
    values a voxel. The reverse sweep reads z and gamma, and reads and writes the six components of its own state
    and the gradient. Operations: the two real transforms and about 150 for the projections of a voxel."""
    if case["kind"] == "batch":
        vox = [g[0] * g[1] * g[2] for g, _, _ in _members(case)]
    else:
        vox = [case["n1"] * case["n2"] * case["n3"]] * case["solves"]
    es, k = (8 if case["precision"] == "fp64" else 4), case["iters"]
    flops = sum(k * v * (150.0 + 5.0 * math.log2(v)) for v in vox)
    if case["kind"] == "gradient":
        return {"bytes": sum(k * v * (13 * 8 + 21 * 4.0) for v in vox), "flops": 2.0 * flops}
    out = 9 * es if case["kind"] == "static" or case.get("fields") else 0
    return {"bytes": float(sum(v * (k * 13 * es + out) for v in vox)), "flops": flops}


# ---- the same in 64 bits -----------------------------------------------------------------

def _next(x, a):
    return torch.roll(x, -1, a)


def _prev(x, a):
    return torch.roll(x, 1, a)


class _Exact:
    """Eq. 28 and Eq. 30 of the paper for one solve, in double, as the reduced updates read."""

    def __init__(self, gamma, normal, case):
        self.g, self.case = gamma, case
        xi = np.asarray(normal, dtype=np.float64)
        self.xi = [float(x) for x in xi / np.linalg.norm(xi)]
        n = gamma.shape
        lam = 0.0
        for a, m in enumerate(n):
            k = torch.arange(n[2] // 2 + 1 if a == 2 else m, device=DEV, dtype=torch.float64)
            s = 4.0 * torch.sin(math.pi * k / m) ** 2
            lam = lam + s.reshape([-1 if b == a else 1 for b in range(3)])
        lam[0, 0, 0] = math.inf
        self.gain = -1.0 / lam

    def start(self):
        e = [torch.full_like(self.g, H * self.xi[c % 3]) for c in range(6)]
        rho0 = _rho0(self.case, self.g)
        if rho0 <= 0.0:
            low = float(self.g.min())
            rho0 = low if low > 0.0 else float(self.g.mean())
        return e, [torch.zeros_like(self.g) for _ in range(6)], rho0

    def project(self, e, v, rho):
        """xi^{k + 1/2} = P_K(e - v / rho)"""
        w = [a - b / rho for a, b in zip(e, v)]
        u = [H * (w[a] + _next(w[3 + a], a)) for a in range(3)]
        d = sum(u[a] - _prev(u[a], a) for a in range(3))
        phi = torch.fft.irfftn(torch.fft.rfftn(d) * self.gain, s=self.g.shape)
        y = [u[a] - (_next(phi, a) - phi) - self.xi[a] for a in range(3)]
        return [w[a] - H * y[a] for a in range(3)] + [w[3 + a] - H * _prev(y[a], a) for a in range(3)]

    def update(self, e, v, rho):
        delta = self.case["delta"]
        x = self.project(e, v, rho)
        z = [b + rho * (2.0 * (1.0 - delta) * c - (1.0 - 2.0 * delta) * a) for a, b, c in zip(e, v, x)]
        n2 = sum(c * c for c in z)
        clip = n2 > self.g * self.g
        scale = torch.where(clip, self.g / torch.sqrt(torch.where(clip, n2, torch.ones_like(n2))), torch.ones_like(n2))
        v2 = [c * scale for c in z]
        return [(c - b) / rho for c, b in zip(z, v2)], v2, x

    def penalty(self, e, v, e2, v2, x, rho):
        """The next rho of the case's rule, from detached sums."""
        def dot(p, q):
            return sum(float((a * b).sum()) for a, b in zip(p, q))
        rule = self.case["rule"]
        lo, hi = rho / 2.0, rho * 2.0
        with torch.no_grad():
            if rule == "const":
                return rho
            if rule == "ltd":
                nv, ne = math.sqrt(dot(v2, v2)), math.sqrt(dot(e2, e2))
                return min(max(nv / ne, lo), hi) if nv > 0.0 and ne > 0.0 else rho
            de, dv = [a - b for a, b in zip(e2, e)], [a - b for a, b in zip(v2, v)]
            if rule == "rb":
                r = math.sqrt(sum(float(((a - b) ** 2).sum()) for a, b in zip(e, x)))
                s = rho * math.sqrt(dot(de, de))
                return hi if r > 10.0 * s else lo if s > 10.0 * r else rho
            ve, ee, vv = dot(dv, de), dot(de, de), dot(dv, dv)
            ok = ve > 0.0 and ee > 0.0 and vv > 0.0 and ve / math.sqrt(vv * ee) > 0.2
            return min(max(ve / ee, lo), hi) if ok else rho

    def dual(self, v):
        return sum(self.xi[a] * H * (v[a].mean() + v[3 + a].mean()) for a in range(3))

    def solve(self):
        e, v, rho = self.start()
        schedule = []
        for _ in range(self.case["iters"]):
            schedule.append(rho)
            e2, v2, x = self.update(e, v, rho)
            rho = self.penalty(e, v, e2, v2, x, rho)
            e, v = e2, v2
            del e2, v2, x
        return e, v, rho, schedule

    def outputs(self):
        e, v, rho, _ = self.solve()
        x = self.project(e, v, rho)
        num = {"gamma_eff": float(self.dual(v)),
               "gamma_primal": float((self.g * torch.sqrt(sum(c * c for c in x))).mean()),
               "residual": math.sqrt(sum(float(((a - b) ** 2).mean()) for a, b in zip(e, x))),
               "mean_v_norm": math.sqrt(sum(float(c.mean()) ** 2 for c in v)), "rho": rho}
        return num, torch.stack([H * (v[a] + _next(v[3 + a], a)) for a in range(3)]), torch.stack(x)


def _exact_numbers(nums):
    out = {k: torch.tensor([m[k] for m in nums], dtype=torch.float64) for k in _NUMBERS}
    return dict(out, iters=None, converged=None, status=None)


def exact(case, seed):
    _, dt = _types(case)
    if case["kind"] == "batch":
        cells, nums = {}, []
        for grid, r, a in _members(case):
            if r not in cells:
                cells = {r: _cell(case["cell"], grid, seed * 100 + r).to(dt).double()}
            nums.append(_Exact(cells[r], np.eye(3)[a], case).outputs()[0])
        return _exact_numbers(nums)
    n = (case["n1"], case["n2"], case["n3"])
    gamma = _cell(case["cell"], n, seed).to(dt).double()
    normals = _normals(case["solves"], seed, case["n3"] == 1)
    if case["kind"] == "gradient":
        g = gamma.requires_grad_(True)
        s = _Exact(g, normals[0], case)
        e, v, _, schedule = s.solve()
        j = s.dual(v)
        (grad,) = torch.autograd.grad(j, g)
        s.g = g.detach()
        e, v = [c.detach() for c in e], [c.detach() for c in v]
        x = s.project(e, v, schedule[-1])
        num = {"gamma_eff": float(j.detach()),
               "gamma_primal": float((s.g * torch.sqrt(sum(c * c for c in x))).mean()),
               "residual": math.sqrt(sum(float(((a - b) ** 2).mean()) for a, b in zip(e, x))),
               "mean_v_norm": math.sqrt(sum(float(c.mean()) ** 2 for c in v)), "rho": schedule[-1]}
        return dict(_exact_numbers([num]), grad=grad[None], schedule=np.asarray(schedule)[None])
    every = [_Exact(gamma, x, case).outputs() for x in normals]
    out = _exact_numbers([m for m, _, _ in every])
    if case["kind"] == "static" or case["fields"]:
        out.update(flow=torch.stack([f for _, f, _ in every]), cut=torch.stack([c for _, _, c in every]))
    return out
