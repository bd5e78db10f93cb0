"""What is timed: relaxation runs, their diagnostics and their gradients,
each as a program of this library does it through the package's entry
points, over the range of grids the library is used on.

A case is a dict of plain values:

  kind       "relax"  set_x, `steps` accepted steps, the state back
             "study"  the same, then every diagnostic of the state
             "adjoint" the loss gradient over `steps` replayed steps
  field      the initial field and grid: "tube", "braid", "isohelix" or
             "periodic" (the shapes of the workloads the tests and the
             benchmark use, with seeded amplitudes, twists and phases)
  nx, ny, nz nodes per axis
  precision  "fp64" or "mixed"
  curl       "mimetic", "direct" or "nnn"
  steps      accepted steps of one pass

The runs are at a chosen largest step (grow_max = 1): a quarter of the
squared grid spacing in FP64 -- the step control rejects it and shrinks where
it is too long -- and a tenth in mixed precision.  (A run that lets the step
grow ends at the stability limit, where modes grown from rounding errors set
the step sizes and no two evaluations agree.)  The mixed-precision runs hand
back the displacement checkpoint, which is FP32 as that mode stores it.

`exact` evaluates the same runs with plain torch operations in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_1405_0942_gb300 as G

# ------------------------------------------------------------------ cases


def _case(name, kind, field, nx, ny, nz, precision, curl, steps):
    c = dict(kind=kind, field=field, nx=nx, ny=ny, nz=nz, precision=precision, curl=curl,
             steps=steps)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest run: a single flux tube on 16^3, where launches and
        # latency count
        _case("tube16", "relax", "tube", 16, 16, 16, "fp64", "mimetic", 20),
        # a validation run of the IsoHelix experiment on its 33^3 grid: a few
        # steps, then every diagnostic (sigma, alpha*, epsilon*, kappa, E, xi, u)
        _case("study33", "study", "isohelix", 33, 33, 33, "fp64", "mimetic", 4),
        # the FP64 run the benchmark quotes
        _case("braid64", "relax", "braid", 64, 64, 64, "fp64", "mimetic", 10),
        # a larger FP64 run on a box of three different, odd extents
        _case("braid129x97x75", "relax", "braid", 129, 97, 75, "fp64", "mimetic", 6),
        # a small mixed-precision run (a first look at a field)
        _case("mixed48", "relax", "braid", 48, 48, 48, "mixed", "mimetic", 20),
        # the mixed-precision run at 128^3
        _case("mixed128", "relax", "braid", 128, 128, 128, "mixed", "mimetic", 10),
        # mixed precision on a grid whose rows are not a multiple of 16 bytes
        _case("mixed101x90x75", "relax", "braid", 101, 90, 75, "mixed", "mimetic", 10),
        # the production size
        _case("mixed384", "relax", "braid", 384, 384, 384, "mixed", "mimetic", 3),
        # the classic method the mimetic one is compared with
        _case("direct65", "relax", "isohelix", 65, 65, 65, "fp64", "direct", 5),
        # the next-nearest-neighbour current of the same comparison
        _case("nnn65", "relax", "isohelix", 65, 65, 65, "fp64", "nnn", 5),
        # periodic boundaries in z
        _case("periodic64", "relax", "periodic", 64, 64, 64, "fp64", "mimetic", 10),
        # forward and backward: the gradient of the final energy with respect
        # to the initial field and positions
        _case("adjoint64", "adjoint", "braid", 64, 64, 64, "fp64", "mimetic", 4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _extents(rng, lo, hi, most):
    """Three extents spread over the logarithm of [lo, hi], odd ones among
    them, their product at most `most`."""
    n = [_log_int(rng, lo, hi) for _ in range(3)]
    while n[0] * n[1] * n[2] > most:
        a = n.index(max(n))
        n[a] = max(lo, int(n[a] * 0.9))
    return n


def draw(rng):
    kind = rng.choice(["fp64", "fp64", "fp64", "mixed", "mixed", "mixed", "direct", "direct32",
                       "nnn", "periodic", "study", "adjoint"])
    if kind == "fp64":
        n = _extents(rng, 12, 150, 1_500_000)
        return _case(None, "relax", rng.choice(["braid", "tube", "isohelix"]), *n, "fp64",
                     "mimetic", rng.randint(3, 9))
    if kind == "mixed":
        n = _extents(rng, 32, 400, 24_000_000)
        return _case(None, "relax", "braid", *n, "mixed", "mimetic", rng.randint(2, 8))
    if kind in ("direct", "direct32"):
        n = _extents(rng, 16, 110, 600_000)
        return _case(None, "relax", rng.choice(["braid", "isohelix"]) if kind == "direct"
                     else "braid", *n, "fp64" if kind == "direct" else "mixed", "direct",
                     rng.randint(2, 6))
    if kind == "nnn":
        n = _extents(rng, 16, 90, 400_000)
        return _case(None, "relax", "isohelix", *n, "fp64", "nnn", rng.randint(2, 6))
    if kind == "periodic":
        n = _extents(rng, 16, 110, 700_000)
        return _case(None, "relax", "periodic", *n, "fp64", "mimetic", rng.randint(3, 8))
    if kind == "study":
        n = _extents(rng, 16, 80, 300_000)
        return _case(None, "study", "isohelix", *n, "fp64", "mimetic", rng.randint(1, 6))
    n = _extents(rng, 16, 90, 400_000)
    return _case(None, "adjoint", rng.choice(["braid", "tube"]), *n, "fp64", "mimetic",
                 rng.randint(2, 5))


# ------------------------------------------------------------------ inputs


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _box(case):
    """(lo, hi, h): the paper's box for the IsoHelix field, else [-1, 1]^3."""
    if case["field"] == "isohelix":
        lo, hi = (-4.0, -4.0, -10.0), (4.0, 4.0, 10.0)
    else:
        lo, hi = (-1.0,) * 3, (1.0,) * 3
    n = (case["nx"], case["ny"], case["nz"])
    return lo, hi, tuple((hi[a] - lo[a]) / (n[a] - 1) for a in range(3))


def _labels(case, dev):
    lo, _, h = _box(case)
    f = dict(dtype=torch.float64, device=dev)
    x = lo[0] + h[0] * torch.arange(case["nx"], **f)
    y = lo[1] + h[1] * torch.arange(case["ny"], **f)
    z = lo[2] + h[2] * torch.arange(case["nz"], **f)
    return x[None, None, :], y[None, :, None], z[:, None, None]


def _fields(case, seed, dev):
    """Positions x0 and field B0 at the labels, float64 (3, nz, ny, nx)."""
    gen = torch.Generator().manual_seed(seed)
    u = torch.rand(64, generator=gen, dtype=torch.float64).tolist()
    X = _labels(case, dev)
    x, y, z = X
    shape = (3, case["nz"], case["ny"], case["nx"])
    x0 = torch.empty(shape, dtype=torch.float64, device=dev)
    B0 = torch.zeros(shape, dtype=torch.float64, device=dev)
    B0[2] = 1.0
    for a in range(3):
        x0[a] = X[a]
    ph = [2.0 * math.pi * v for v in u[:5]]
    if case["field"] == "tube":
        k, l = 0.8 + 0.4 * u[5], 0.45 + 0.1 * u[6]
        g = k * torch.exp(-x * x / l ** 2) * torch.exp(-y * y / l ** 2) * torch.exp(-z * z)
        B0[0] += -y * g
        B0[1] += x * g
    elif case["field"] == "braid":
        m = 6
        for i in range(m):
            xc, zc = (0.4 if i % 2 == 0 else -0.4), -0.75 + 1.5 * i / (m - 1)
            k = (1.0 if i % 2 == 0 else -1.0) * (0.5 + u[8 + i])
            g = (k * torch.exp(-(x - xc) ** 2 / 0.09) * torch.exp(-y * y / 0.09) *
                 torch.exp(-(z - zc) ** 2 / 0.0625))
            B0[0] += -y * g
            B0[1] += (x - xc) * g
        for a in range(3):
            x0[a] += 0.05 * torch.sin(math.pi * X[a] + ph[a])
    elif case["field"] == "isohelix":
        phi = math.pi / 4 * (0.8 + 0.4 * u[5])
        g = (2.0 * phi / 4.0 * z * torch.exp(-z * z / 4.0) * torch.exp(-x * x / 2.0) *
             torch.exp(-y * y / 2.0))
        B0[0] += g * y
        B0[1] += -g * x
    else:
        w = 2.0 * math.pi / ((case["nz"] - 2) * _box(case)[2][2])
        g1 = torch.exp(-x * x / 0.25) * torch.exp(-y * y / 0.25) * torch.sin(w * z + ph[3])
        dx, dy = x - 0.3, y + 0.2
        g2 = (-0.8 * torch.exp(-dx * dx / 0.16) * torch.exp(-dy * dy / 0.16) *
              torch.cos(2.0 * w * z + ph[4]))
        B0[0] += -y * g1 - dy * g2
        B0[1] += x * g1 + dx * g2
        for a in range(2):
            x0[a] += 0.05 * torch.sin(math.pi * X[a] + ph[a])
        x0[2] += 0.05 * torch.sin(w * z + ph[2])
    return x0, B0


def _relaxed(case, seed, dev):
    """The IsoHelix field's closed-form relaxed state (x_ref, B_ref) the
    deviations are measured against."""
    gen = torch.Generator().manual_seed(seed)
    u = torch.rand(64, generator=gen, dtype=torch.float64).tolist()
    phi = math.pi / 4 * (0.8 + 0.4 * u[5])
    x, y, z = _labels(case, dev)
    th = phi * torch.exp(-(x * x + y * y) / 2.0 - z * z / 4.0)
    c, s = torch.cos(th), torch.sin(th)
    xr = torch.stack([c * x + s * y, c * y - s * x, z.expand_as(th).clone()])
    Br = torch.zeros_like(xr)
    Br[2] = 1.0
    return xr, Br


def _dt0(case):
    return (0.25 if case["precision"] == "fp64" else 0.1) * min(_box(case)[2]) ** 2


def prepare(case, seed):
    dev = _device()
    x0, B0 = _fields(case, seed, dev)
    lo, hi, _ = _box(case)
    mixed = case["precision"] == "mixed"
    r = G.Relaxation(case["nx"], case["ny"], case["nz"], lo=lo, hi=hi,
                     precision=G.MIXED if mixed else G.FP64,
                     curl={"mimetic": G.MIMETIC, "direct": G.DIRECT, "nnn": G.NNN}[case["curl"]],
                     dt0=_dt0(case), grow_max=1.0,
                     periodic_z=1 if case["field"] == "periodic" else None)
    r.set_B0(B0)
    s = dict(case=case, relax=r, x0=x0)
    if case["kind"] == "study":
        s["x_ref"], s["B_ref"] = _relaxed(case, seed, dev)
    if case["kind"] == "adjoint":
        s["dts"] = [_dt0(case) * (1.0 + 0.25 * i) for i in range(case["steps"])]
    return s


# ------------------------------------------------------------------ one pass


def run(s):
    case, r = s["case"], s["relax"]
    if case["kind"] == "adjoint":
        value, dB0, dx0 = r.adjoint_segment(s["x0"], s["dts"], G.LOSS_ENERGY, 2)
        return dict(value=value, dB0=dB0, dx0=dx0)
    r.set_x(s["x0"])
    st = r.step(case["steps"])
    if case["precision"] == "mixed":
        return dict(d=r.get_state().view(torch.float32), t=st["t"])
    out = dict(x=r.get_x(), t=st["t"], dt=st["dt"], accepted=st["accepted"],
               rejected=st["rejected"])
    if case["kind"] == "study":
        out["energy"] = r.energy()
        out["xi"], out["xi_sin"] = r.forcefree_err()
        out["u"] = r.velocity()
        out["sigma_x"], out["sigma_B"] = r.deviation(s["x_ref"], s["B_ref"])
        out["alpha"], out["eps"] = r.alpha_line(case["nx"] // 2, case["ny"] // 2, math.sqrt(2.0))
        out["concave"], out["kappa"] = r.convexity(with_field=True)
    return out


def work(case):
    """Inputs read once and outputs written once in each step (the state in
    and out, B0 in; the steps depend on one another through the whole grid),
    and the operations of the method (an FMA is two): per interior node and
    stage 151 mimetic, 330 direct, 729 next-nearest-neighbour; the reverse of
    a step adds 527 a stage."""
    N = case["nx"] * case["ny"] * case["nz"]
    inner = (case["nx"] - 2) * (case["ny"] - 2) * (case["nz"] - 2)
    el = 4 if case["precision"] == "mixed" else 8
    flops = {"mimetic": 151, "direct": 330, "nnn": 729}[case["curl"]]
    bytes_ = 9 * el * N * case["steps"]
    if case["kind"] == "adjoint":  # forwards, recomputed, and back
        flops += 527
        bytes_ += 15 * el * N * case["steps"]
    if case["kind"] == "study":
        bytes_ += (9 + 3) * el * N + N
    return {"bytes": bytes_, "flops": 6 * flops * inner * case["steps"]}


# ------------------------------------------------------------------ 64 bits

_A = ((), (1 / 5,), (3 / 40, 9 / 40), (3 / 10, -9 / 10, 6 / 5),
      (-11 / 54, 5 / 2, -70 / 27, 35 / 27),
      (1631 / 55296, 175 / 512, 575 / 13824, 44275 / 110592, 253 / 4096))
_B5 = (37 / 378, 0.0, 250 / 621, 125 / 594, 0.0, 512 / 1771)
_B4 = (2825 / 27648, 0.0, 18575 / 48384, 13525 / 55296, 277 / 14336, 1 / 4)


def _cut(f, a, off, margin=(1, 1, 1)):
    """f (.., nz, ny, nx) at the nodes at least `margin` from the faces,
    shifted by `off[b]` nodes along axis b (0 = x); a is unused when None."""
    s = []
    for b in (2, 1, 0):
        n, m, o = f.shape[-1 - b], margin[b], off[b]
        s.append(slice(m + o, n - m + o))
    return f[(Ellipsis, *s)]


def _unit(a, s=1):
    o = [0, 0, 0]
    o[a] = s
    return o


def _central(f, a, margin=(1, 1, 1)):
    return _cut(f, a, _unit(a), margin) - _cut(f, a, _unit(a, -1), margin)


def _column(d, a, h):
    """Index-space derivative 2 h_a dx/dX_a at every node: central, and
    second-order one-sided on the faces."""
    ax = 3 - a
    n = d.shape[ax]
    p = lambda i: d.narrow(ax, i, 1)  # noqa: E731
    g = torch.cat([4 * p(1) - 3 * p(0) - p(2), d.narrow(ax, 2, n - 2) - d.narrow(ax, 0, n - 2),
                   3 * p(n - 1) - 4 * p(n - 2) + p(n - 3)], dim=ax)
    e = torch.zeros(3, 1, 1, 1, dtype=d.dtype, device=d.device)
    e[a] = 2.0 * h[a]
    return g + e


def _cross(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2],
                        a[0] * b[1] - a[1] * b[0]])


def _dot(a, b):
    return a[0] * b[0] + a[1] * b[1] + a[2] * b[2]


def _pull(d, B0, h, periodic):
    """Columns of the scaled Jacobian, its determinant and B."""
    g = [_column(d, a, h) for a in range(3)]
    if periodic:
        g[2] = torch.cat([g[2][:, :1], _central_z(d, h), g[2][:, -1:]], dim=1)
    det = _dot(g[0], _cross(g[1], g[2]))
    s = [4 * h[1] * h[2], 4 * h[2] * h[0], 4 * h[0] * h[1]]
    B = (g[0] * (B0[0] * s[0]) + g[1] * (B0[1] * s[1]) + g[2] * (B0[2] * s[2])) / det
    if periodic:
        B = torch.cat([B[:, -2:-1], B[:, 1:-1], B[:, 1:2]], dim=1)
    return g, det, B


def _central_z(d, h):
    g = d[:, 2:] - d[:, :-2]
    e = torch.zeros(3, 1, 1, 1, dtype=d.dtype, device=d.device)
    e[2] = 2.0 * h[2]
    return g + e


def _loops(P, g, det):
    c = [_dot(P[(a + 1) % 3], g[(a + 2) % 3]) - _dot(P[(a + 2) % 3], g[(a + 1) % 3])
         for a in range(3)]
    return (c[0] * g[0] + c[1] * g[1] + c[2] * g[2]) / det


def _current(d, B0, h, curl, periodic):
    """(J, B, det G) : the current at the interior nodes, B everywhere."""
    g, det, B = _pull(d, B0, h, periodic)
    z = (0, 0, 0)
    gi = [_cut(v, None, z) for v in g]
    di = _cut(det, None, z)
    if curl == "mimetic":
        return _loops([_central(B, a) for a in range(3)], gi, di), B, det
    if curl == "direct":
        s = [4 * h[1] * h[2], 4 * h[2] * h[0], 4 * h[0] * h[1]]
        bs = torch.stack([B0[a] * s[a] for a in range(3)])
        b, Db = _cut(bs, None, z), [_central(bs, a) for a in range(3)]
        S = [[None] * 3 for _ in range(3)]
        for a in range(3):
            S[a][a] = 4 * (_cut(d, a, _unit(a)) + _cut(d, a, _unit(a, -1)) - 2 * _cut(d, a, z))
            for e in range(a + 1, 3):
                v = 0
                for p in (1, -1):
                    for q in (1, -1):
                        o = _unit(a, p)
                        o[e] = q
                        v = v + p * q * _cut(d, a, o)
                S[a][e] = S[e][a] = v
        V = gi[0] * b[0] + gi[1] * b[1] + gi[2] * b[2]
        cof = [_cross(gi[1], gi[2]), _cross(gi[2], gi[0]), _cross(gi[0], gi[1])]
        DB = []
        for c in range(3):
            Dd = sum(_dot(cof[a], S[a][c]) for a in range(3))
            DV = sum(S[a][c] * b[a] + gi[a] * Db[c][a] for a in range(3))
            DB.append((DV - V * (Dd / di)) / di)
        # dB/dx = dB/dX (dx/dX)^-1; its antisymmetric part is the loop form
        return _loops(DB, gi, di), B, det
    # octilateral loops: edge-mean circulation and the loop's vector area
    op, oq = (1, 1, 1, 0, -1, -1, -1, 0), (-1, 0, 1, 1, 1, 0, -1, -1)
    M, cr = [], []
    for r in range(3):
        p, q = (r + 1) % 3, (r + 2) % 3
        xv, Bv = [], []
        for m in range(8):
            o = [0, 0, 0]
            o[p], o[q] = op[m], oq[m]
            e = torch.zeros(3, 1, 1, 1, dtype=d.dtype, device=d.device)
            e[p], e[q] = op[m] * h[p], oq[m] * h[q]
            xv.append(_cut(d, None, o) - _cut(d, None, z) + e)
            Bv.append(_cut(B, None, o))
        cr.append(sum(_dot(0.5 * (Bv[m] + Bv[(m + 1) % 8]), xv[(m + 1) % 8] - xv[m])
                      for m in range(8)))
        M.append(sum(0.5 * _cross(xv[m], xv[(m + 1) % 8]) for m in range(8)))
    adj = [_cross(M[1], M[2]), _cross(M[2], M[0]), _cross(M[0], M[1])]
    return (cr[0] * adj[0] + cr[1] * adj[1] + cr[2] * adj[2]) / _dot(M[0], adj[0]), B, det


def _velocity(d, B0, h, curl, periodic):
    J, B, det = _current(d, B0, h, curl, periodic)
    u = _cross(J, _cut(B, None, (0, 0, 0)))
    return torch.nn.functional.pad(u, (1, 1, 1, 1, 1, 1)), det


def _ghosts(d, periodic):
    return torch.cat([d[:, -2:-1], d[:, 1:-1], d[:, 1:2]], dim=1) if periodic else d


def _attempt(d, B0, h, curl, periodic, dt):
    """(new displacement, error, a trial stage folded the grid)."""
    k, folded = [], False
    for s in range(6):
        y = d
        for j in range(s):
            y = y + (dt * _A[s][j]) * k[j]
        u, det = _velocity(_ghosts(y, periodic), B0, h, curl, periodic)
        if s and not torch.is_grad_enabled():
            folded = folded or bool((det <= 0).any())
        k.append(u)
    new, err = d, 0
    for j in range(6):
        new = new + (dt * _B5[j]) * k[j]
        err = err + (dt * (_B5[j] - _B4[j])) * k[j]
    return _ghosts(new, periodic), err, folded


def _energy(d, B0, h):
    g, det, B = _pull(d, B0, h, False)
    w = 1.0 / 16.0
    for ax in range(3):
        v = torch.ones(d.shape[1 + ax], dtype=d.dtype, device=d.device)
        v[0] = v[-1] = 0.5
        w = w * v.view([-1 if i == ax else 1 for i in range(3)])
    return (w * _dot(B, B) * det).sum()


def exact(case, seed):
    dev = _device()
    x0, B0 = _fields(case, seed, dev)
    lo, _, h = _box(case)
    X = torch.empty_like(x0)
    for a, v in enumerate(_labels(case, dev)):
        X[a] = v
    curl, periodic = case["curl"], case["field"] == "periodic"
    mixed = case["precision"] == "mixed"
    if case["kind"] == "adjoint":
        d0 = (x0 - X).requires_grad_(True)
        b = B0.clone().requires_grad_(True)
        d = d0
        for i in range(case["steps"]):
            d, _, _ = _attempt(d, b, h, curl, False, _dt0(case) * (1.0 + 0.25 * i))
        E = _energy(d, b, h)
        dx0, dB0 = torch.autograd.grad(E, (d0, b))
        inner = torch.nn.functional.pad(_cut(dx0, None, (0, 0, 0)), (1, 1, 1, 1, 1, 1))
        return dict(value=float(E.detach()), dB0=dB0, dx0=inner)
    with torch.no_grad():
        d = _ghosts(x0 - X, periodic)
        lambda0, shrink = 1e-7, 0.1  # the library's defaults
        dt, t, accepted = _dt0(case), 0.0, 0
        for _ in range(400):
            if accepted == case["steps"]:
                break
            new, err, folded = _attempt(d, B0, h, curl, periodic, dt)
            lam = float(err.abs().max())
            if folded:
                dt *= shrink
            elif lam > lambda0:
                dt *= max((lambda0 / lam) ** 0.2, shrink)
            else:
                d, t, accepted = new, t + dt, accepted + 1
                if 0.0 < lam < 0.5 * lambda0:  # never beyond grow_max = 1
                    dt *= min((lambda0 / lam) ** 0.2, 1.0)
        if accepted < case["steps"]:
            return None
        if mixed:
            return dict(d=d.reshape(-1), t=t)
        out = dict(x=X + d, t=t, dt=dt, accepted=None, rejected=None)
        if case["kind"] != "study":
            return out
        J, B, _ = _current(d, B0, h, curl, periodic)
        Bi = _cut(B, None, (0, 0, 0))
        u = _cross(J, Bi)
        u2, b2, j2 = _dot(u, u), _dot(Bi, Bi), _dot(J, J)
        out["energy"] = float(_energy(d, B0, h))
        out["xi"] = float((u2.sqrt() / b2).max())
        jb = j2 * b2
        out["xi_sin"] = float(torch.where(jb > 0, u2 / jb, torch.zeros_like(jb)).max().sqrt())
        out["u"] = torch.nn.functional.pad(u, (1, 1, 1, 1, 1, 1))
        xr, Br = _relaxed(case, seed, dev)
        N = case["nx"] * case["ny"] * case["nz"]
        out["sigma_x"] = math.sqrt(float(((X + d - xr) ** 2).sum()) / N)
        out["sigma_B"] = math.sqrt(float(((B - Br) ** 2).sum()) / N)
        i, j = case["nx"] // 2 - 1, case["ny"] // 2 - 1
        al = (_dot(J, Bi)[:, j, i] / b2[:, j, i]).cpu().numpy()
        alpha = np.full(case["nz"], np.nan)
        alpha[1:-1] = al
        k = np.arange(al.size)
        dz = np.abs(k[:, None] - k[None, :]) * h[2]
        np.fill_diagonal(dz, 1.0)
        out["alpha"] = alpha
        out["eps"] = float((math.sqrt(2.0) * (al[:, None] - al[None, :]) / dz).max())
        out["concave"] = out["kappa"] = None
        return out
