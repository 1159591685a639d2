"""Performance cases: the work a user has the sweeping preconditioner do, through its public entry points.

Five kinds of case:
  matvec  one 7-point operator product (GMRES does one per iteration);
  apply   one preconditioner application (Alg. 1.5) with a handle the program keeps;
  setup   a new handle for a new velocity model (Alg. 1.4) and its first application;
  solve   GMRES(k) to a relative residual of 1e-5 with a handle the program keeps;
  step    a batch of independent problems, or one problem, set up and solved.
Grids, PML thickness, panel depths and options are those of this repository's benchmark and tests (20^3
to 100^3 cubes, the 4-plane panels of the paper, the 8-plane panels of the salt workload, 1 to 8 right-hand
sides) and ragged boxes between them.

A handle with complex64 factors returns its complex128 vectors with single-precision accuracy, and a
program that chose it keeps what it gets (wavefields, corrections of an outer iteration) as complex64: so
do the cases.
"""
import math

import torch

from paper_1204_0111_gb300 import psp
from paper_1204_0111_gb300 import workloads as wl

ALPHA = 2.0 * math.pi


def _case(name, kind, nx, ny, nz, model, prec="c128", nrhs=1, gamma=8, depth=4, pad=8, si="extended", which=0,
          k=20, nprob=1):
    d = dict(kind=kind, nx=nx, ny=ny, nz=nz, model=model, prec=prec, nrhs=nrhs, gamma=gamma, depth=depth, pad=pad,
             si=si, which=which, k=k, nprob=nprob)
    if name:
        d["name"] = name
    return d


def listed():
    return [
        # the matvec of every GMRES iteration on the benchmark's grid, and the damped operator on a ragged box
        _case("matvec_A_100", "matvec", 100, 100, 100, "lens"),
        _case("matvec_J_ragged_x3", "matvec", 61, 83, 47, "layered", nrhs=3, which=1),
        # the smallest application: the CPU-seconds problem, a chain of tiny fronts
        _case("apply_c128_20", "apply", 20, 20, 20, "lens", gamma=5, pad=5),
        # one application of the benchmark's preconditioner, in both precisions
        _case("apply_c128_100", "apply", 100, 100, 100, "lens"),
        _case("apply_c64_100", "apply", 100, 100, 100, "lens", prec="c64"),
        # the paper's factor form on an odd box with a few right-hand sides
        _case("apply_c128_paper_x3", "apply", 57, 45, 51, "layered", nrhs=3, si="paper"),
        # many shots at once: one problem of the batch workload, and a half-size salt body with deep panels
        _case("apply_c64_88_x8", "apply", 88, 88, 88, "smooth", prec="c64", nrhs=8),
        _case("apply_c64_salt_128_x8", "apply", 128, 128, 128, "salt", prec="c64", nrhs=8, gamma=12, depth=8),
        # a new velocity model: factorisation and first application
        _case("setup_c128_80", "setup", 80, 80, 80, "lens"),
        _case("setup_c64_100", "setup", 100, 100, 100, "layered", prec="c64"),
        # whole calls: the paper's waveguide with four right-hand sides, and a small batch from c(x) to u
        _case("solve_c128_waveguide_48_x4", "solve", 48, 48, 48, "waveguide", nrhs=4, gamma=5, pad=5),
        _case("step_c64_batch3_x8", "step", 40, 40, 40, "smooth", prec="c64", nrhs=8, nprob=3),
    ]


def draw(rng):
    kind = rng.choice(["matvec", "apply", "apply", "apply", "setup", "setup", "solve", "step"])

    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    top = {"matvec": 128, "apply": 88, "setup": 72, "solve": 48, "step": 44}[kind]
    # GMRES is for models it converges on quickly at every seed
    models = ["lens", "smooth", "waveguide"] if kind in ("solve", "step") else ["lens", "layered", "smooth", "salt", "waveguide"]
    n = size(16, top)
    nx, ny, nz = (max(13, min(top, int(round(n * rng.uniform(0.8, 1.2))))) for _ in range(3))
    prec = "c128" if kind == "matvec" else rng.choice(["c128", "c64"])
    gamma = rng.choice([5, 6, 8])
    return _case("", kind, nx, ny, nz, rng.choice(models), prec=prec,
                 nrhs=8 if kind == "step" else rng.choice([1, 1, 2, 3, 4, 8]), gamma=gamma, depth=rng.choice([3, 4, 4, 5]),
                 pad=gamma, si=rng.choice(["extended", "extended", "paper"]) if kind in ("apply", "setup") else "extended",
                 which=rng.choice([0, 1]) if kind == "matvec" else 0, nprob=rng.choice([1, 2, 3]) if kind == "step" else 1)


# ---------------------------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------------------------
def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _problem(case, seed, q=0):
    """Problem q of a case: its grid, seeded wave speed (device, (nz, ny, nx)) and the handle's parameters."""
    nx, ny, nz = (case[a] + 8 * q for a in ("nx", "ny", "nz"))
    h = 1.0 / (max(nx, ny, nz) + 1)
    g = torch.Generator().manual_seed(1000 * seed + q)
    r = torch.rand(64, generator=g, dtype=torch.float64)
    dev = _device()
    x, y, z = ((torch.arange(n, dtype=torch.float64, device=dev) + 1) * h for n in (nx, ny, nz))
    x, y, z = x[None, None, :], y[None, :, None], z[:, None, None]
    model, c_ref = case["model"], 1.0
    if model == "lens":
        p = 0.45 + 0.1 * r[:3]
        c = 1.0 - 0.4 * torch.exp(-32.0 * ((x - p[0]) ** 2 + (y - p[1]) ** 2 + (z - p[2]) ** 2))
    elif model == "waveguide":   # invariant along the sweep direction: its interior panels share a factorisation
        p = 0.45 + 0.1 * r[:2]
        c = 1.25 * (1.0 - 0.4 * torch.exp(-32.0 * ((x - p[0]) ** 2 + (y - p[1]) ** 2))) + 0.0 * z
        c_ref = 1.25
    elif model == "layered":     # dipping layers, as in the 200^3 model
        zz = z + 0.3 * (r[0] - 0.5) * (x - 0.5) + 0.3 * (r[1] - 0.5) * (y - 0.5)
        layer = torch.bucketize(zz, torch.sort(r[2:14]).values.to(dev))
        c = (1.5 + 4.5 * r[16:29]).to(dev)[layer]
        c_ref = 6.0
    elif model == "smooth":      # a smooth random field, c in (1.5, 2.5)
        f = sum(torch.sin((20 * r[4 * i] - 10) * x + (20 * r[4 * i + 1] - 10) * y + (20 * r[4 * i + 2] - 10) * z
                          + 6.28 * r[4 * i + 3]) for i in range(12))
        c = 2.0 + 0.5 * torch.tanh(f / math.sqrt(6.0))
        c_ref = 2.5
    else:                        # salt body in a depth gradient
        p = 0.45 + 0.1 * r[:3]
        d = torch.sqrt(((x - p[0]) / 0.3) ** 2 + ((y - p[1]) / 0.3) ** 2 + ((z - p[2]) / 0.2125) ** 2)
        blend = 0.5 * (1.0 + torch.tanh((1.0 - d) * 0.2125 / (2.0 * h)))
        c = (1.5 + 3.0 * z) * (1.0 - blend) + 4.5 * blend
        c_ref = 4.5
    c = c.expand(nz, ny, nx).contiguous()
    ppw = 8.0 if model == "salt" else 10.0
    return dict(nx=nx, ny=ny, nz=nz, h=h, c=c, omega=wl.omega_for_ppw(float(c.min()), ppw, h), gamma=case["gamma"],
                depth=case["depth"], pad=case["pad"], C=wl.pml_amplitude(4.0, c_ref))


def _shots(case, p, seed, q=0):
    """(nrhs, N) Gaussian shots (sigma = 2h) at seeded positions above the model's lower half."""
    g = torch.Generator().manual_seed(1000 * seed + 77 + q)
    r = torch.rand(case["nrhs"], 3, generator=g, dtype=torch.float64)
    dev = p["c"].device
    out = []
    for s in range(case["nrhs"]):
        e = [torch.exp(-((torch.arange(n, dtype=torch.float64, device=dev) + 1) * p["h"] - float(0.25 + 0.5 * r[s, a])
                         * n * p["h"]) ** 2 / (8.0 * p["h"] ** 2)) for a, n in enumerate((p["nx"], p["ny"], p["nz"]))]
        out.append((e[2][:, None, None] * e[1][None, :, None] * e[0][None, None, :]).reshape(-1))
    return torch.stack(out).to(torch.complex128)


def _vectors(case, p, seed):
    """(nrhs, N) vectors of unit length, as Krylov vectors are: noise with energy everywhere."""
    n = p["nx"] * p["ny"] * p["nz"]
    dev = p["c"].device
    g = torch.Generator(device=dev).manual_seed(1000 * seed + 5)
    v = torch.randn(case["nrhs"], n, generator=g, dtype=torch.complex128, device=dev)
    return v / torch.linalg.vector_norm(v, dim=1, keepdim=True)


def _handle(case, p):
    return psp.SweepingPreconditioner(p["c"], p["h"], p["omega"], p["gamma"], p["depth"], pad=p["pad"], pml_C=p["C"],
                                      alpha=ALPHA, precision=case["prec"], selective_inversion=case["si"])


def prepare(case, seed):
    if case["kind"] == "step":
        ps = [_problem(case, seed, q) for q in range(case["nprob"])]
        fs = [_shots(case, p, seed, q) for q, p in enumerate(ps)]
        f = torch.cat([b.reshape(-1) for b in fs]) if len(fs) > 1 else fs[0]
        return {"case": case, "problems": ps, "f": f, "u": torch.zeros_like(f)}
    p = _problem(case, seed)
    f = _shots(case, p, seed) if case["kind"] == "solve" else _vectors(case, p, seed)
    state = {"case": case, "problem": p, "f": f, "u": torch.zeros_like(f)}
    if case["kind"] != "setup":
        state["handle"] = _handle(case, p)
    return state


def run(state):
    case, f, u = state["case"], state["f"], state["u"]
    kind = case["kind"]
    if kind == "matvec":
        return state["handle"].matvec(f, u, which=case["which"])
    if kind == "apply":
        state["handle"].apply(f, u)
    elif kind == "setup":
        P = _handle(case, state["problem"])
        P.apply(f, u)
        P.close()
    elif kind == "solve":
        state["handle"].solve(f, u, tol=1e-5, k=case["k"], maxit=300)
    else:
        ps = state["problems"]
        if len(ps) == 1:
            P = _handle(case, ps[0])
        else:
            P = psp.SweepingPreconditionerBatch(
                [dict(c=p["c"], h=p["h"], omega=p["omega"], gamma=p["gamma"], panel_depth=p["depth"]) for p in ps],
                pad=ps[0]["pad"], pml_C=ps[0]["C"], alpha=ALPHA, precision=case["prec"])
        P.solve(f, u, tol=1e-5, k=case["k"], maxit=300)
        P.close()
    return u.to(torch.complex64) if case["prec"] == "c64" else u


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _fronts(nx, ny, D, leaf=64):
    """(s, u) of every front of a box's nested dissection: separators are cut across the longer side."""
    out = []

    def rec(x0, x1, y0, y1):
        wx, wy = x1 - x0, y1 - y0
        if wx <= 0 or wy <= 0:
            return
        u = D * (wy * ((x0 > 0) + (x1 < nx)) + wx * ((y0 > 0) + (y1 < ny)))
        if wx * wy * D <= leaf:
            out.append((wx * wy * D, u))
        elif wx >= wy:
            m = x0 + wx // 2
            rec(x0, m, y0, y1)
            rec(m + 1, x1, y0, y1)
            out.append((wy * D, u))
        else:
            m = y0 + wy // 2
            rec(x0, x1, y0, m)
            rec(x0, x1, m + 1, y1)
            out.append((wx * D, u))

    rec(0, nx, 0, ny)
    return out


def _plan(nz, gamma, depth, pad):
    """Panels (z0, z1, pad planes)."""
    first = min(gamma + depth, nz)
    cuts = [0, first] + list(range(first + depth, nz, depth)) + ([nz] if first < nz else [])
    return [(a, b, 0 if a == 0 else pad) for a, b in zip(cuts[:-1], cuts[1:])]


def _box_counts(case, q=0):
    """Per panel: factor entries and factorisation multiply-adds (LDL^T, F_BL solve, Schur update)."""
    nx, ny, nz = (case[a] + 8 * q for a in ("nx", "ny", "nz"))
    memo, out = {}, []
    for z0, z1, pad in _plan(nz, case["gamma"], case["depth"], case["pad"]):
        D = pad + z1 - z0
        if D not in memo:
            fr = _fronts(nx, ny, D)
            memo[D] = (sum(s * (s + 1) / 2 + s * u for s, u in fr),
                       sum(s ** 3 / 3 + u * s * s / 2 + u * (u + 1) / 2 * s for s, u in fr))
        out.append(memo[D])
    return nx * ny * nz, out


def work(case):
    """bytes and flops of one pass.  An application solves with every panel twice (the last one once); a panel
    solve reads the panel's factors up and down the tree, for all right-hand sides at once."""
    item = 8 if case["prec"] == "c64" else 16
    nrhs, by, fl = case["nrhs"], 0.0, 0.0
    for q in range(case["nprob"]):
        n, boxes = _box_counts(case, q)
        entries = sum(e for e, _ in boxes)
        reads = 2 * (2 * entries - boxes[-1][0])
        apply_b, apply_f = reads * item + 32.0 * n * nrhs, 8.0 * reads * nrhs
        mat_b, mat_f = 8.0 * n + 32.0 * n * nrhs, 56.0 * n * nrhs
        distinct = 3 if case["model"] == "waveguide" else len(boxes)   # z-invariant: first, interior, last panels
        setup_b = 8.0 * n + entries * item * min(1.0, distinct / len(boxes))
        setup_f = 8.0 * sum(f for _, f in boxes) * min(1.0, distinct / len(boxes))
        its = 12   # GMRES iterations to 1e-5 on these models, about
        gmres_b = its * (apply_b + mat_b) + 16.0 * n * nrhs * its * (its + 1)
        gmres_f = its * (apply_f + mat_f) + 8.0 * n * nrhs * its * (its + 1)
        kind = case["kind"]
        by += {"matvec": mat_b, "apply": apply_b, "setup": setup_b + apply_b, "solve": gmres_b, "step": setup_b + gmres_b}[kind]
        fl += {"matvec": mat_f, "apply": apply_f, "setup": setup_f + apply_f, "solve": gmres_f, "step": setup_f + gmres_f}[kind]
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------------------------
# the same results in plain torch, in 64 bits
# ---------------------------------------------------------------------------------------------
def _sigma(xi, n, g, C, h, lo=True, hi=True):
    s = torch.zeros_like(xi)
    for on, dist in ((lo, (xi + 1.0) * h), (hi, (n - xi) * h)):
        if on:
            s = s + C / (g * h) * torch.clamp(((g + 1) * h - dist) / (g * h), min=0.0) ** 2
    return s


def _axis(p, n, shift=0, count=None):
    """Stretches of a domain axis at nodes and half-points, from node `shift` on."""
    count = n if count is None else count
    dev = p["c"].device
    node = torch.arange(count, dtype=torch.float64, device=dev) + shift
    half = torch.arange(count + 1, dtype=torch.float64, device=dev) - 0.5 + shift
    return tuple(torch.complex(torch.ones_like(t), _sigma(t, n, p["gamma"], p["C"], p["h"]) / p["omega"])
                 for t in (node, half))


def _pad_axis(p, z0, z1, pad):
    """The x3 stretch of a panel's box: a pad profile below the panel on top of the domain's own."""
    dev = p["c"].device
    out = []
    for t in (torch.arange(pad + z1 - z0, dtype=torch.float64, device=dev),
              torch.arange(pad + z1 - z0 + 1, dtype=torch.float64, device=dev) - 0.5):
        sig = _sigma(t, 0, pad, p["C"], p["h"], hi=False) if pad > 0 else torch.zeros_like(t)
        own = _sigma(t + z0 - pad, p["nz"], p["gamma"], p["C"], p["h"])
        sig = sig + torch.where(t >= pad - 0.5, own, torch.zeros_like(own))
        out.append(torch.complex(torch.ones_like(t), sig / p["omega"]))
    return tuple(out)


def _coefficients(p, k2, s1, s2, s3):
    """Diagonal, and the couplings below each node along x, y and z, of the symmetrised operator on a box."""
    n1, n2, n3 = s1[0][None, None, :], s2[0][None, :, None], s3[0][:, None, None]
    ih2 = 1.0 / (p["h"] * p["h"])
    a1 = n2 * n3 / s1[1][None, None, :] * ih2
    a2 = n1 * n3 / s2[1][None, :, None] * ih2
    a3 = n1 * n2 / s3[1][:, None, None] * ih2
    d = a1[:, :, :-1] + a1[:, :, 1:] + a2[:, :-1] + a2[:, 1:] + a3[:-1] + a3[1:] - k2 * n1 * n2 * n3
    return d, a1, a2, a3


def _k2(p, which):
    w = complex(p["omega"], ALPHA if which else 0.0)
    return (w * w) / (p["c"] ** 2).to(torch.complex128)


def _product(co, x):
    d, a1, a2, a3 = co
    y = d * x
    y[..., 1:] -= a1[:, :, 1:-1] * x[..., :-1]
    y[..., :-1] -= a1[:, :, 1:-1] * x[..., 1:]
    y[..., 1:, :] -= a2[:, 1:-1] * x[..., :-1, :]
    y[..., :-1, :] -= a2[:, 1:-1] * x[..., 1:, :]
    y[..., 1:, :, :] -= a3[1:-1] * x[..., :-1, :, :]
    y[..., :-1, :, :] -= a3[1:-1] * x[..., 1:, :, :]
    return y


class _BoxSolver:
    """Block elimination of a box by its x slabs (dense inverses of the Schur complements)."""

    def __init__(self, co):
        d, a1, a2, a3 = co
        self.D, self.ny, self.nx = d.shape
        b = self.D * self.ny
        ix = torch.arange(b, device=d.device).reshape(self.D, self.ny)
        self.off = [a1[:, :, x].expand(self.D, self.ny).reshape(-1) for x in range(1, self.nx)]
        self.inv = []
        for x in range(self.nx):
            m = torch.zeros(b, b, dtype=torch.complex128, device=d.device)
            m[ix.reshape(-1), ix.reshape(-1)] = d[:, :, x].reshape(-1)
            for i, j, v in ((ix[:, 1:], ix[:, :-1], a2[:, 1:-1, x]), (ix[1:], ix[:-1], a3[1:-1, :, x])):
                i, j, v = i.reshape(-1), j.reshape(-1), v.expand(i.shape).reshape(-1)
                m[i, j] = -v
                m[j, i] = -v
            if x:
                o = self.off[x - 1]
                m -= o[:, None] * self.inv[-1] * o[None, :]
            self.inv.append(torch.linalg.inv(m))

    def solve(self, v):
        """v: (nrhs, D, ny, nx)."""
        f = v.permute(3, 1, 2, 0).reshape(self.nx, self.D * self.ny, -1)
        y = []
        for x in range(self.nx):
            t = f[x] if x == 0 else f[x] + self.off[x - 1][:, None] * y[-1]
            y.append(self.inv[x] @ t)
        for x in range(self.nx - 2, -1, -1):
            y[x] = y[x] + self.inv[x] @ (self.off[x][:, None] * y[x + 1])
        return torch.stack(y).reshape(self.nx, self.D, self.ny, -1).permute(3, 1, 2, 0)


def _exact_apply(p, f):
    s1, s2, s3 = _axis(p, p["nx"]), _axis(p, p["ny"]), _axis(p, p["nz"])
    k2 = _k2(p, 1)
    plan = _plan(p["nz"], p["gamma"], p["depth"], p["pad"])
    plane = s1[0][None, :] * s2[0][:, None] / (p["h"] * p["h"])     # J's coupling across a plane, times s3 there
    boxes = []
    for z0, z1, pad in plan:
        kk = torch.cat([k2[z0:z0 + 1].expand(pad, -1, -1), k2[z0:z1]])
        s = _axis(p, p["nz"], 0, z1) if z0 == 0 else _pad_axis(p, z0, z1, pad)
        boxes.append(_BoxSolver(_coefficients(p, kk, s1, s2, s)))

    def T(i, v):
        pad = plan[i][2]
        w = torch.zeros(v.shape[0], pad, v.shape[2], v.shape[3], dtype=v.dtype, device=v.device)
        return boxes[i].solve(torch.cat([w, v], dim=1))[:, pad:]

    u = f.reshape(f.shape[0], p["nz"], p["ny"], p["nx"]).clone()
    for i, (z0, z1, _) in enumerate(plan):
        v = u[:, z0:z1].clone()
        if i:
            v[:, 0] += plane / s3[1][z0] * u[:, z0 - 1]
        u[:, z0:z1] = T(i, v)
    for i in range(len(plan) - 2, -1, -1):
        z0, z1, _ = plan[i]
        v = torch.zeros_like(u[:, z0:z1])
        v[:, -1] = -plane / s3[1][z1] * u[:, z1]
        u[:, z0:z1] -= T(i, v)
    return u.reshape(f.shape)


def _exact_solution(p, f):
    s1, s2, s3 = _axis(p, p["nx"]), _axis(p, p["ny"]), _axis(p, p["nz"])
    b = f.reshape(f.shape[0], p["nz"], p["ny"], p["nx"]) * (s3[0][:, None, None] * s2[0][None, :, None] * s1[0])
    return _BoxSolver(_coefficients(p, _k2(p, 0), s1, s2, s3)).solve(b).reshape(f.shape)


def exact(case, seed):
    kind = case["kind"]
    if kind == "matvec":
        p = _problem(case, seed)
        co = _coefficients(p, _k2(p, case["which"]), _axis(p, p["nx"]), _axis(p, p["ny"]), _axis(p, p["nz"]))
        f = _vectors(case, p, seed)
        return _product(co, f.reshape(-1, p["nz"], p["ny"], p["nx"])).reshape(f.shape)
    # seconds of the dense block eliminations at about 0.5 TFLOP/s
    cost = 0.0
    for q in range(case["nprob"]):
        nx, ny, nz = (case[a] + 8 * q for a in ("nx", "ny", "nz"))
        depths = [pad + b - a for a, b, pad in _plan(nz, case["gamma"], case["depth"], case["pad"])]
        cost += sum(nx * (ny * d) ** 3 for d in (depths if kind in ("apply", "setup") else [nz])) * 16 / 5e11
    if cost > 10.0:
        return None
    if kind in ("apply", "setup"):
        p = _problem(case, seed)
        return _exact_apply(p, _vectors(case, p, seed))
    if kind == "solve":
        p = _problem(case, seed)
        return _exact_solution(p, _shots(case, p, seed))
    out = []
    for q in range(case["nprob"]):
        p = _problem(case, seed, q)
        out.append(_exact_solution(p, _shots(case, p, seed, q)))
    return torch.cat([o.reshape(-1) for o in out]) if len(out) > 1 else out[0]
