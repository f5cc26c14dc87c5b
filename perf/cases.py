"""The workloads this library is timed on, through its public entry points.

A case is a problem (or batch), the arithmetic and options it is run with, and
the call a program makes: an evaluation of the spatial operator inside a
caller's own time loop (``operator_noalloc``), a run to a final time
(``advance``), or a number of steps (``enqueue_steps``).  A pass of the last
two hands the initial averages over, marches, and takes the state back.

The FP64 form returns its FP64 state.  The mixed form computes its fluxes in
FP32 and is chosen by programs that go on in FP32, so its state is handed on
as FP32.

``exact`` evaluates the same scheme in 64 bits with plain torch operations:
rows first, one Thomas (or block Thomas) walk over all lines at once.
"""
from __future__ import annotations

import math
import random

import torch

from paper_1402_5618_gb300 import binding as B

PER, TRANS, REFL = 0, 1, 2
GAMMA, WGL, EPS_WENO, EPS_POS = 1.4, 1.0 / 12.0, 1e-13, 1e-13
FORMS = {"fp64": B.PREC_FP64, "mixed": B.PREC_MIXED}


def listed():
    return [
        # the smallest call: the operator of the 200-cell density wave, asked
        # for by a program that integrates in time by itself
        dict(name="operator_wave_200", kind="wave", call="operator", n=200, form="fp64"),
        # the same service on a 2-D grid of odd sizes with jumps, mixed
        # boundaries and the Lax-Friedrichs flux
        dict(name="operator_jumps_517x253_llf", kind="jumps", call="operator", nx=517, ny=253,
             form="fp64", flux="llf"),
        # a 1-D accuracy study: N = 200 periodic density wave, many tiny steps
        dict(name="wave_200", kind="wave", call="advance", n=200, form="fp64", steps=128),
        # a 1-D shock problem as the paper runs it: interacting blast waves
        # between walls, characteristic-wise reconstruction
        dict(name="walls_800_char", kind="walls", call="advance", n=800, form="fp64", recon="char",
             steps=32),
        # thousands of uneven 1-D Riemann problems with checked steps, in
        # both arithmetics
        dict(name="riemann_4096_mixed", kind="riemann", call="steps", problems=4096, lo=256,
             hi=8192, form="mixed", checked=True, steps=6),
        dict(name="riemann_4096_fp64", kind="riemann", call="steps", problems=4096, lo=256,
             hi=8192, form="fp64", checked=True, steps=2),
        # smooth periodic flow on a large grid, in both arithmetics
        dict(name="vortex_2048_mixed", kind="vortex", call="steps", nx=2048, ny=2048,
             form="mixed", steps=12),
        dict(name="vortex_1024_fp64", kind="vortex", call="steps", nx=1024, ny=1024,
             form="fp64", steps=2),
        # the large production grid: a blast between two walls, checked steps
        dict(name="blast_4096_mixed", kind="blast", call="steps", nx=4096, ny=4096, form="mixed",
             checked=True, steps=6),
        # uneven 2-D four-quadrant problems, in both arithmetics
        dict(name="quadrants_64_mixed", kind="quadrants", call="steps", problems=64, lo=128,
             hi=1024, form="mixed", checked=True, steps=8),
        dict(name="quadrants_32_fp64", kind="quadrants", call="steps", problems=32, lo=128,
             hi=1024, form="fp64", checked=True, steps=1),
        # the characteristic-wise reconstruction on a large grid
        dict(name="blast_2048_char_mixed", kind="blast", call="steps", nx=2048, ny=2048,
             form="mixed", recon="char", checked=True, steps=3),
    ]


# about how long a cell-stage takes (ns) by form, dimension and reconstruction
_COST = {("fp64", 1, "comp"): 2.1, ("fp64", 2, "comp"): 5.9, ("mixed", 1, "comp"): 0.3,
         ("mixed", 2, "comp"): 0.4, ("fp64", 1, "char"): 25.0, ("fp64", 2, "char"): 14.0,
         ("mixed", 1, "char"): 4.0, ("mixed", 2, "char"): 0.8}


def draw(rng: random.Random):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["wave", "walls", "riemann", "vortex", "jumps", "blast", "quadrants"])
    form = rng.choice(["fp64", "mixed"])
    c = dict(kind=kind, form=form, flux=rng.choice(["hllc", "hllc", "llf"]))
    if kind in ("wave", "walls"):
        c.update(n=log(64, 8192), call=rng.choice(["advance", "operator"]), steps=log(8, 128))
    elif kind == "riemann":
        c.update(problems=log(64, 4096), lo=256, hi=log(512, 8192), call="steps",
                 checked=True, steps=log(1, 16))
    elif kind == "quadrants":
        c.update(problems=log(4, 64), lo=128, hi=log(256, 1024), call="steps",
                 checked=True, steps=log(1, 8))
    else:
        c.update(nx=log(96, 4096), ny=log(96, 4096), steps=log(1, 16), call="steps")
        if kind == "jumps":
            c.update(nx=min(c["nx"], 1000), ny=min(c["ny"], 1000),
                     call=rng.choice(["steps", "operator"]))
        if kind == "blast":
            c.update(ny=c["nx"], checked=True)
    if c["call"] == "operator":      # the allocation-free operator: FP64, component-wise
        c.update(form="fp64")
        c.pop("steps")
    elif kind in ("walls", "blast", "riemann", "jumps") and rng.random() < 0.3:
        c.update(recon="char")
    # no dearer than the largest listed case: steps, then problems, then cells
    def cost():
        dims = 1 if kind in ("wave", "walls", "riemann") else 2
        return sum(x["nx"] * x["ny"] for x in _grids(c)) * 3 * c.get("steps", 1) * _COST[
            c["form"], dims, c.get("recon", "comp")] * 1e-9
    while cost() > 0.1 and c.get("steps", 1) > 1:
        c["steps"] -= 1
    while cost() > 0.1 and c.get("problems", 1) > 8:
        c["problems"] = c["problems"] * 3 // 4
    while cost() > 0.1 and "nx" in c:
        c["nx"] = c["nx"] * 7 // 8
        c["ny"] = c["nx"] if kind == "blast" else c["ny"] * 7 // 8
    return c


# ------------------------------------------------------------------ problems
def _grids(case):
    """Size, domain, boundaries and CFL number of each problem of a case."""
    k = case["kind"]
    if k == "wave":       # dt = 0.6 dx^(5/3) / max(|u| + a)
        n = case["n"]
        return [dict(nx=n, ny=1, dx=2.0 / n, dy=1.0, bc=(PER, PER, 0, 0),
                     cfl=0.6 * (2.0 / n) ** (2.0 / 3.0))]
    if k == "walls":
        n = case["n"]
        return [dict(nx=n, ny=1, dx=1.0 / n, dy=1.0, bc=(REFL, REFL, 0, 0), cfl=1.0 / 12.0)]
    if k in ("riemann", "quadrants"):   # log-uniform sizes, the same for every seed
        r = random.Random(case["problems"] * 100003 + case["hi"])
        out = []
        for _ in range(case["problems"]):
            n = int(round(math.exp(r.uniform(math.log(case["lo"]), math.log(case["hi"])))))
            two = k == "quadrants"
            out.append(dict(nx=n, ny=n if two else 1, dx=1.0 / n, dy=1.0 / n if two else 1.0,
                            bc=(TRANS,) * 4, cfl=0.5))
        return out
    nx, ny = case["nx"], case["ny"]
    if k == "vortex":
        return [dict(nx=nx, ny=ny, dx=10.0 / nx, dy=10.0 / ny, bc=(PER,) * 4, cfl=0.5)]
    if k == "jumps":
        return [dict(nx=nx, ny=ny, dx=1.0 / max(nx, ny), dy=1.0 / max(nx, ny),
                     bc=(REFL, TRANS, TRANS, REFL), cfl=1.0 / 12.0)]
    return [dict(nx=nx, ny=ny, dx=1.1 / nx, dy=1.1 / ny, bc=(REFL, TRANS, REFL, TRANS), cfl=0.5)]


def _dims(case):
    return 1 if case["kind"] in ("wave", "walls", "riemann") else 2


def _configs(case):
    nd = _dims(case)
    return [B.make_config(
        nd, g["nx"], g["ny"], 0.0, g["dx"] * g["nx"], 0.0, g["dy"] * g["ny"], GAMMA, g["cfl"],
        g["bc"], FORMS[case["form"]], cfl_positivity_cap=bool(case.get("checked")),
        flux=B.FLUX_LLF if case.get("flux") == "llf" else B.FLUX_HLLC,
        recon=B.RECON_CHARACTERISTIC if case.get("recon") == "char" else B.RECON_COMPONENT)
        for g in _grids(case)]


def _cons(rho, u, v, p):
    m = [rho * u] + ([] if v is None else [rho * v])
    kin = u * u if v is None else u * u + v * v
    return torch.stack([rho, *m, p / (GAMMA - 1.0) + 0.5 * rho * kin])


def _initial(case, seed, dev):
    """Initial cell averages, one [nv, cells] tensor per problem."""
    g = torch.Generator().manual_seed(int(seed) * 7919 + 17)

    def uni(lo, hi, *shape):
        return lo + (hi - lo) * torch.rand(*shape, generator=g, dtype=torch.float64)

    def logu(lo, hi, *shape):
        return torch.exp(uni(math.log(lo), math.log(hi), *shape))

    grids, k = _grids(case), case["kind"]
    G = grids[0]
    nx, ny = G["nx"], G["ny"]
    x = (torch.arange(nx, dtype=torch.float64, device=dev) + 0.5) * G["dx"]
    y = (torch.arange(ny, dtype=torch.float64, device=dev) + 0.5) * G["dy"]
    if k == "wave":
        amp, ph = uni(0.1, 0.3, 2).tolist()
        rho = 1.0 + amp * torch.sin(math.pi * x + 20.0 * ph)
        return [_cons(rho, torch.ones_like(x), None, torch.ones_like(x))]
    if k == "walls":
        f = uni(0.8, 1.25, 3).tolist()
        p = torch.where(x < 0.1, 1000.0 * f[0], torch.where(x < 0.9, 0.01 * f[1], 100.0 * f[2]))
        return [_cons(torch.ones_like(x), torch.zeros_like(x), None, p)]
    if k == "riemann":
        # rho log-U[0.1, 10], u U[-3, 3], p log-U[0.01, 10]; one in ten a
        # near-vacuum double rarefaction rho = 1, p = 0.4, u = -/+ 2 to 4
        P = len(grids)
        rho, u, p = logu(0.1, 10.0, 2, P), uni(-3.0, 3.0, 2, P), logu(0.01, 10.0, 2, P)
        vac, s = uni(0.0, 1.0, P) < 0.1, uni(2.0, 4.0, P)
        rho[:, vac], p[:, vac] = 1.0, 0.4
        u[0, vac], u[1, vac] = -s[vac], s[vac]
        n = torch.tensor([q["nx"] for q in grids], device=dev)
        ends = _cons(rho, u, None, p).to(dev)                       # [3, 2, P]
        pid = torch.repeat_interleave(torch.arange(P, device=dev), n)
        i = torch.arange(pid.numel(), device=dev) - (torch.cumsum(n, 0) - n)[pid]
        left = (0.5 * n[pid] - i).clamp(0.0, 1.0)                   # part of a cell left of 1/2
        U = left * ends[:, 0, pid] + (1.0 - left) * ends[:, 1, pid]
        return list(torch.split(U, n.tolist(), dim=1))
    if k == "quadrants":
        out = []
        for q in grids:
            m = q["nx"]
            s = _cons(logu(0.1, 2.0, 4), uni(-1.0, 1.0, 4), uni(-1.0, 1.0, 4), logu(0.02, 2.0, 4))
            s = s.to(dev)                                           # [4 variables, 4 quadrants]
            lo = torch.arange(m, dtype=torch.float64, device=dev)
            f = (0.5 * m - lo).clamp(0.0, 1.0)
            w = torch.stack([torch.outer(1 - f, 1 - f), torch.outer(1 - f, f), torch.outer(f, f),
                             torch.outer(f, 1 - f)])
            out.append((s @ w.reshape(4, -1)))
        return out
    if k == "vortex":
        cx, cy = uni(3.0, 7.0, 2).tolist()
        strength = float(uni(4.0, 5.0, 1))
        U = 0.0
        q = math.sqrt(0.15)                        # 3 x 3 Gauss-Legendre cell averages
        for a, wa in ((-q, 5 / 18), (0.0, 8 / 18), (q, 5 / 18)):
            for b, wb in ((-q, 5 / 18), (0.0, 8 / 18), (q, 5 / 18)):
                dy = (y + a * G["dy"] - cy + 5.0)[:, None] % 10.0 - 5.0
                dx = (x + b * G["dx"] - cx + 5.0)[None, :] % 10.0 - 5.0
                r2 = dx * dx + dy * dy
                e = strength / (2 * math.pi) * torch.exp(0.5 * (1.0 - r2))
                T = 1.0 - (GAMMA - 1.0) * strength ** 2 / (8 * GAMMA * math.pi ** 2) * torch.exp(1.0 - r2)
                rho = T ** (1.0 / (GAMMA - 1.0))
                U = U + wa * wb * _cons(rho, 1.0 - e * dy, 1.0 + e * dx, rho ** GAMMA)
        return [U.reshape(4, -1)]
    if k == "jumps":
        nb = 4
        r, p = logu(0.2, 5.0, nb, nb), logu(0.05, 5.0, nb, nb)
        u, v = uni(-1.0, 1.0, nb, nb), uni(-1.0, 1.0, nb, nb)
        cuts = [torch.sort(uni(0.05, 0.95, nb - 1))[0].to(dev) * m for m in (ny, nx)]
        j = torch.bucketize(torch.arange(ny, device=dev, dtype=torch.float64), cuts[0])
        i = torch.bucketize(torch.arange(nx, device=dev, dtype=torch.float64), cuts[1])
        U = _cons(r, u, v, p).to(dev)[:, j][:, :, i]
        return [U.reshape(4, -1).contiguous()]
    # a blast from the corner some way into its run: a strong cylindrical
    # shock at radius R moving into cold gas at rest, the interior emptied
    R, s = float(uni(0.4, 0.8, 1)), float(uni(0.5, 2.0, 1))
    rr = torch.sqrt(x[None, :] ** 2 + y[:, None] ** 2)
    xi = (rr / R).clamp(max=1.0)
    inside = rr < R
    rho = torch.where(inside, (6.0 * xi ** 7).clamp(min=0.05), torch.ones_like(rr))
    vel = torch.where(inside, s / 1.2 * xi, torch.zeros_like(rr))
    p = torch.where(inside, s * s / 1.2 * (0.4 + 0.6 * xi ** 8), torch.full_like(rr, 4e-11))
    U = _cons(rho, vel * x[None, :] / rr, vel * y[:, None] / rr, p)
    return [U.reshape(4, -1)]


def _t_final(case):
    """Final time of an ``advance``: about case["steps"] steps of the case's data."""
    G = _grids(case)[0]
    top = 1.0 + math.sqrt(GAMMA / 0.7) if case["kind"] == "wave" else math.sqrt(GAMMA * 1250.0)
    return case["steps"] * G["cfl"] * G["dx"] / top


# ------------------------------------------------------------------ the interface
def prepare(case, seed):
    """The initial averages on the GPU, the solver handle (or the config of a
    handle-free operator call) and the array the result goes to."""
    U = torch.cat([u.reshape(-1) for u in _initial(case, seed, "cuda")]).contiguous()
    cfgs = _configs(case)
    st = dict(case=case, U=U, out=torch.empty_like(U))
    if case["call"] == "operator":
        st["cfg"] = cfgs[0]
    elif case["kind"] in ("riemann", "quadrants"):
        st["solver"] = B.Solver(None, batch=cfgs)
    else:
        st["solver"] = B.Solver(cfgs[0])
    return st


def run(state):
    case, U, out = state["case"], state["U"], state["out"]
    if case["call"] == "operator":
        B.operator_noalloc(state["cfg"], U, out)
        return out
    s = state["solver"]
    s.set_state(U)
    if case["call"] == "advance":
        s.advance(_t_final(case))
    else:
        s.enqueue_steps(case["steps"])
    s.get_state(out)
    return out.float() if case["form"] == "mixed" else out


def work(case):
    nd = _dims(case)
    nv = nd + 2
    cells = sum(g["nx"] * g["ny"] for g in _grids(case))
    limit, flux = (97, 95) if nv == 3 else (121, 118)
    if case.get("recon") == "char":
        # per side and face: Roe average and eigenvectors, characteristic
        # variables of five cells, weights and rows, one step of block Thomas
        recon = 2 * (60 + 5 * nv * (2 * nv - 1) + nv * 76
                     + 2 * nv * nv * (nv + 1) + 2 * nv ** 3 // 3 + 2 * nv * nv * (nv + 1) + 2 * nv * nv)
    else:
        recon = nv * 135     # indicators 33, weights 44, rows 42, both solves 16
    sweep = recon + limit + flux + 2 * nv
    stages = 1 if case["call"] == "operator" else 3 * case["steps"]
    combine = 0 if case["call"] == "operator" else 5 * nv + 15
    out = 4 if case["form"] == "mixed" else 8
    return {"bytes": (8 + out) * nv * cells, "flops": stages * cells * (nd * sweep + combine)}


# ------------------------------------------------------------------ 64-bit evaluation
class _Lines:
    """All grid lines of one direction: position-first gather indices of both
    walks (left to right, and mirrored), lengths and boundaries per line."""

    def __init__(self, grids, xdir, nd, dev):
        base, start, step, n, lo, hi, h, pid = 0, [], [], [], [], [], [], []
        for k, g in enumerate(grids):
            nx, ny = g["nx"], g["ny"]
            m, ln = (ny, nx) if xdir else (nx, ny)
            i = torch.arange(m, device=dev)
            start.append(base + i * (nx if xdir else 1))
            one = torch.ones(m, dtype=torch.long, device=dev)
            step.append(one * (1 if xdir else nx))
            n.append(one * ln)
            lo.append(one * g["bc"][0 if xdir else 2])
            hi.append(one * g["bc"][1 if xdir else 3])
            h.append(one.double() * (g["dx"] if xdir else g["dy"]))
            pid.append(one * k)
            base += nx * ny
        cat = torch.cat
        start, step, self.n, self.lo, self.hi = cat(start), cat(step), cat(n), cat(lo), cat(hi)
        self.h, self.pid = cat(h), cat(pid)
        self.N, self.L = int(self.n.max()), self.n.numel()
        self.order = [0, 1, 2][:nd + 2] if nd == 1 else ([0, 1, 2, 3] if xdir else [0, 2, 1, 3])
        self.per = self.lo == PER
        pos = torch.arange(-2, self.N + 2, device=dev)[:, None]
        n1 = self.n[None]

        def address(i):
            i = torch.where(i > n1 + 1, n1 - 1, torch.where(i < -2, torch.zeros_like(i), i))
            low, high = i < 0, i >= n1
            j = torch.where(low, torch.where(self.lo == PER, i + n1, torch.where(self.lo == TRANS, 0 * i, -i - 1)), i)
            j = torch.where(high, torch.where(self.hi == PER, i - n1, torch.where(self.hi == TRANS, n1 - 1 + 0 * i, 2 * n1 - 1 - i)), j)
            neg = (low & (self.lo == REFL)) | (high & (self.hi == REFL))
            return start + step * j.clamp(min=0), neg

        a, na = address(pos)
        b, nb = address(n1 - 1 - pos)
        self.ids, self.neg = cat([a, b], 1), cat([na, nb], 1)
        self.valid = pos[2:-2] < n1                        # [N, L]
        self.cells = a[2:-2]
        self.mirror = (n1 - 1 - pos[2:-2]).clamp(min=0)    # walk position of a cell in the other walk


def _z(w, eps, c):
    """WENO-Z weights over five cells."""
    b = [13 / 12 * (w[0] - 2 * w[1] + w[2]) ** 2 + 0.25 * (w[0] - 4 * w[1] + 3 * w[2]) ** 2,
         13 / 12 * (w[1] - 2 * w[2] + w[3]) ** 2 + 0.25 * (w[1] - w[3]) ** 2,
         13 / 12 * (w[2] - 2 * w[3] + w[4]) ** 2 + 0.25 * (3 * w[2] - 4 * w[3] + w[4]) ** 2]
    tau = (b[2] - b[0]).abs()
    al = [ck * (1 + (tau / (bk + eps)) ** 2) for ck, bk in zip(c, b)]
    s = al[0] + al[1] + al[2]
    return [a / s for a in al]


def _rows(w, ends, live):
    """Compact rows (a, b, c, r) at every position; explicit rows at `ends`
    of bounded lines, unit rows where a shorter line has ended."""
    w0, w1, w2 = _z(w, EPS_WENO, (0.2, 0.5, 0.3))
    a, b, c = (2 * w0 + w1) / 3, (w0 + 2 * (w1 + w2)) / 3, w2 / 3
    r = (w0 * w[1] + (5 * (w0 + w1) + w2) * w[2] + (w1 + 5 * w2) * w[3]) / 6
    w0, w1, w2 = _z(w, EPS_WENO, (0.1, 0.6, 0.3))
    f = (w0 * (2 * w[0] - 7 * w[1] + 11 * w[2]) + w1 * (5 * w[2] - w[1] + 2 * w[3])
         + w2 * (2 * w[2] + 5 * w[3] - w[4])) / 6
    r = torch.where(ends, f, r)
    off = ends | ~live
    a, c, b = a.masked_fill(off, 0.0), c.masked_fill(off, 0.0), b.masked_fill(off, 1.0)
    return a, b, c, r.masked_fill(~live, 0.0)


def _walk(a, b, c, rhs):
    """Thomas over the leading dimension for the right-hand sides rhs[n, k, ...]."""
    S = torch.cat([b[:, None], rhs], 1)
    t = S[0].clone()
    for p in range(a.shape[0]):
        if p:
            torch.addcmul(S[p], a[p], S[p - 1], value=-1, out=t)
        torch.div(t[1:], t[0], out=S[p, 1:])
        torch.div(c[p], t[0], out=S[p, 0])
    for p in range(a.shape[0] - 2, -1, -1):
        torch.addcmul(S[p, 1:], S[p, 0], S[p + 1, 1:], value=-1, out=S[p, 1:])
    return S[:, 1:]


def _faces_component(W, ln, ends, live):
    N = W.shape[0] - 4
    a, b, c, r = _rows([W[k:k + N] for k in range(5)], ends, live)
    if not bool(ln.per.any()):
        return _walk(a, b, c, r[:, None])[:, 0]
    # Sherman-Morrison: v = e_first - (a0 / b0) e_last, u = -b0 e_first + c_last e_last
    n = ln.N
    a0, b0, cl = a[0].clone(), b[0].clone(), c[n - 1].clone()
    u = torch.zeros_like(r)
    u[0], u[n - 1] = -b0, cl
    b[0] = 2 * b0
    b[n - 1] += cl * a0 / b0
    a[0], c[n - 1] = 0.0, 0.0
    X = _walk(a, b, c, torch.stack([r, u], 1))
    y, z = X[:, 0], X[:, 1]
    f = (y[0] - a0 / b0 * y[n - 1]) / (1 + z[0] - a0 / b0 * z[n - 1])
    return y - f * z


def _faces_characteristic(W, ln, ends, live):
    N, nv, M = W.shape[0] - 4, W.shape[1], W.shape[2]

    def half(Q):
        s = Q[:, 0].sqrt()
        p = _pressure(Q)
        return s, [Q[:, k] / s for k in range(1, nv - 1)], (Q[:, -1] + p) / s

    (sa, va, Ha), (sb, vb, Hb) = half(W[2:N + 2]), half(W[3:N + 3])
    vel = [(p + q) / (sa + sb) for p, q in zip(va, vb)]
    H = (Ha + Hb) / (sa + sb)
    k2 = sum(q * q for q in vel)
    a2 = (GAMMA - 1) * (H - 0.5 * k2)
    ia, c1 = a2.rsqrt(), (GAMMA - 1) / a2
    c2, u = 0.5 * k2 * c1, vel[0]
    L = torch.zeros(N, M, nv, nv, dtype=W.dtype, device=W.device)
    for row, sgn in ((0, 1.0), (nv - 1, -1.0)):
        L[..., row, 0] = 0.5 * (c2 + sgn * u * ia)
        L[..., row, 1] = -0.5 * (c1 * u + sgn * ia)
        L[..., row, -1] = 0.5 * c1
    L[..., 1, 0], L[..., 1, 1], L[..., 1, -1] = 1 - c2, c1 * u, -c1
    if nv == 4:
        v = vel[1]
        L[..., 0, 2] = L[..., 3, 2] = -0.5 * c1 * v
        L[..., 1, 2] = c1 * v
        L[..., 2, 0], L[..., 2, 2] = -v, 1.0
    Q = W.permute(0, 2, 1)[..., None]
    w = [(L @ Q[k:k + N])[..., 0] for k in range(5)]                # [N, M, nv]
    a, b, c, r = _rows(w, ends.permute(0, 2, 1), live.permute(0, 2, 1))
    L = torch.where(live.permute(0, 2, 1)[..., None], L, torch.eye(nv, dtype=W.dtype, device=W.device))
    S = torch.zeros(N, M, nv, nv + 1, dtype=W.dtype, device=W.device)   # Y | g
    T = torch.zeros(M, nv, nv + 1, dtype=W.dtype, device=W.device)
    for p in range(N):
        if p:
            T = a[p][..., None] * (L[p] @ S[p - 1])
        Bp = b[p][..., None] * L[p] - T[..., :nv]
        rhs = torch.cat([c[p][..., None] * L[p], (r[p] - T[..., nv])[..., None]], -1)
        S[p] = torch.linalg.solve_ex(Bp, rhs)[0]
    X = S[..., nv].clone()
    for p in range(N - 2, -1, -1):
        X[p] -= (S[p, :, :, :nv] @ X[p + 1][..., None])[..., 0]
    return X.permute(0, 2, 1)


def _pressure(Q):
    return (GAMMA - 1) * (Q[:, -1] - 0.5 * (Q[:, 1:-1] ** 2).sum(1) / Q[:, 0])


def _limit(ub, um, up, eps):
    """Zhang-Shu limiter with the round-off allowance of its thresholds."""
    uu = 2.0 ** -53
    inner = lambda: (ub - WGL * up - WGL * um) / (1 - 2 * WGL)  # noqa: E731
    rmin = torch.minimum(torch.minimum(um[:, 0], up[:, 0]), inner()[:, 0])
    er = eps + 8 * uu * (ub[:, 0].abs() + rmin.abs())
    th = torch.where(rmin < er, ((ub[:, 0] - er) / (ub[:, 0] - rmin)).clamp(0.0, 1.0), torch.ones_like(rmin))
    um, up = um.clone(), up.clone()
    for q in (um, up):
        q[:, 0] = torch.where(rmin < er, th * (q[:, 0] - ub[:, 0]) + ub[:, 0], q[:, 0])
    th = torch.ones_like(rmin)
    for w in (um, up, inner()):
        eta = 16 * uu * ((ub[:, -1].abs() + w[:, -1].abs()) * (ub[:, 0].abs() + w[:, 0].abs())
                         + ((ub[:, 1:-1].abs() + w[:, 1:-1].abs()) ** 2).sum(1))
        g = w[:, 0] * w[:, -1] - 0.5 * (w[:, 1:-1] ** 2).sum(1) - eps * w[:, 0] ** 2
        d = w - ub
        A = d[:, -1] * d[:, 0] - 0.5 * (d[:, 1:-1] ** 2).sum(1) - eps * d[:, 0] ** 2
        Bq = ub[:, -1] * d[:, 0] + d[:, -1] * ub[:, 0] - (ub[:, 1:-1] * d[:, 1:-1]).sum(1) - 2 * eps * ub[:, 0] * d[:, 0]
        C = ub[:, -1] * ub[:, 0] - 0.5 * (ub[:, 1:-1] ** 2).sum(1) - eps * ub[:, 0] ** 2 - eta
        den = (Bq * Bq - 4 * A * C).clamp(min=0.0).sqrt() - Bq
        root = torch.where((C > 0) & (den > 0), 2 * C / den, torch.zeros_like(C)).nan_to_num(0.0).clamp(0.0, 1.0)
        th = torch.where(g < eta, torch.minimum(th, root), th)
    hit = (th < 1)[:, None]
    th = th[:, None]
    return torch.where(hit, th * (um - ub) + ub, um), torch.where(hit, th * (up - ub) + ub, up)


def _phys(Q, p):
    u = Q[:, 1:2] / Q[:, 0:1]
    F = Q * u
    F[:, 1] += p
    F[:, -1] += u[:, 0] * p
    return F


def _flux(Ql, Qr, llf):
    """(flux, largest |u| + a of the two states) at every face."""
    pl, pr = _pressure(Ql), _pressure(Qr)
    rl, rr, ul, ur = Ql[:, 0], Qr[:, 0], Ql[:, 1] / Ql[:, 0], Qr[:, 1] / Qr[:, 0]
    al, ar = (GAMMA * pl / rl).sqrt(), (GAMMA * pr / rr).sqrt()
    top = torch.maximum(ul.abs() + al, ur.abs() + ar)
    Fl, Fr = _phys(Ql, pl), _phys(Qr, pr)
    if llf:
        return 0.5 * (Fl + Fr) - 0.5 * top[:, None] * (Qr - Ql), top
    R = (rr / rl).sqrt()
    roe = lambda a, b: (a + b * R) / (1 + R)  # noqa: E731
    ut, Ht = roe(ul, ur), roe((Ql[:, -1] + pl) / rl, (Qr[:, -1] + pr) / rr)
    k2 = ut * ut
    if Ql.shape[1] == 4:
        k2 = k2 + roe(Ql[:, 2] / rl, Qr[:, 2] / rr) ** 2
    at = ((GAMMA - 1) * (Ht - 0.5 * k2)).sqrt()
    SL, SR = torch.minimum(ul - al, ut - at), torch.maximum(ur + ar, ut + at)
    SM = (rr * ur * (SR - ur) - rl * ul * (SL - ul) + pl - pr) / (rr * (SR - ur) - rl * (SL - ul))

    def star(Q, F, u, p, S):
        q = Q[:, 0] * (S - u) / (S - SM)
        ps = Q[:, 0] * (u - S) * (u - SM) + p
        V = Q * (q / Q[:, 0])[:, None]
        V[:, 1] = q * SM
        V[:, -1] = ((S - u) * Q[:, -1] - p * u + ps * SM) / (S - SM)
        return F + S[:, None] * (V - Q)

    F = torch.where((SM > 0)[:, None], star(Ql, Fl, ul, pl, SL),
                    torch.where((SR >= 0)[:, None], star(Qr, Fr, ur, pr, SR), Fr))
    return torch.where((SL > 0)[:, None], Fl, F), top


def _sweep(U, ln, case, eps):
    """(flux difference [nv, cells], largest face speed / h per problem) of one direction."""
    nv = U.shape[0]
    W = U[ln.order][:, ln.ids].permute(1, 0, 2).contiguous()       # [N + 4, nv, 2 L]
    W[:, 1] = torch.where(ln.neg, -W[:, 1], W[:, 1])
    N, L = ln.N, ln.L
    n2, per2 = torch.cat([ln.n, ln.n]), torch.cat([ln.per, ln.per])
    pos = torch.arange(N, device=U.device)[:, None, None]
    live = (pos < n2).expand(N, 1, 2 * L)
    ends = ((pos == 0) | (pos == n2 - 1)) & ~per2
    faces = _faces_characteristic if case.get("recon") == "char" else _faces_component
    X = faces(W, ln, ends, live)
    um = X[:, :, :L]
    up = X[:, :, L:].gather(0, ln.mirror[:, None].expand(N, nv, L))
    ub = W[2:N + 2, :, :L]
    ok = ln.valid[:, None]
    um, up = torch.where(ok, um, ub), torch.where(ok, up, ub)
    um, up = _limit(ub, um, up, eps[ln.pid])
    last = (ln.n - 1)[None, None].expand(1, nv, L)
    ml, p0 = um.gather(0, last)[0], up[0]
    sign = torch.ones(nv, 1, dtype=U.dtype, device=U.device)
    sign[1] = -1.0
    low = torch.where(ln.per, ml, torch.where(ln.lo == REFL, sign * p0, p0))
    high = torch.where(ln.per, p0, torch.where(ln.hi == REFL, sign * ml, ml))
    Ql = torch.cat([low[None], um])
    Qr = torch.cat([up, high[None]]).scatter(0, last + 1, high[None])
    F, top = _flux(Ql, Qr, case.get("flux") == "llf")
    D = torch.empty_like(U)
    Lf = (F[:-1] - F[1:]) / ln.h
    sel = ln.cells[ln.valid]
    for k, v in enumerate(ln.order):
        D[v, sel] = Lf[:, k][ln.valid]
    faces_live = torch.arange(N + 1, device=U.device)[:, None] <= ln.n
    line_top = top.masked_fill(~faces_live, 0.0).amax(0) / ln.h
    rate = torch.zeros_like(eps).scatter_reduce(0, ln.pid, line_top, "amax")
    return D, rate


def exact(case, seed):
    grids, nd = _grids(case), _dims(case)
    nv = nd + 2
    cells = [g["nx"] * g["ny"] for g in grids]
    stages = 1 if case["call"] == "operator" else 3 * case["steps"]
    dev = "cuda" if sum(cells) > 20000 else "cpu"
    # about how long: rows of the walks one after another, cells in bulk
    row = 5e-5 if case.get("recon") != "char" else 5e-4 if dev == "cuda" else 1.2e-4
    rows = sum(max(g[k] for g in grids) for k in ("nx", "ny")[:nd])
    bulk = nd * sum(g["ny"] for g in grids) * max(g["nx"] for g in grids)
    if stages * (rows * row + bulk * 1.2e-8) > 20.0 or (
            case.get("recon") == "char" and grids[0]["bc"][0] == PER):
        return None
    U = torch.cat([u.reshape(nv, -1) for u in _initial(case, seed, "cuda")], 1).to(dev)
    lines = [_Lines(grids, True, nd, dev)] + ([_Lines(grids, False, nd, dev)] if nd == 2 else [])
    t64 = lambda v: torch.tensor(v, dtype=torch.float64, device=dev)  # noqa: E731
    pid = torch.repeat_interleave(torch.arange(len(grids), device=dev), torch.tensor(cells, device=dev))
    h = [t64([g["dx"] for g in grids]), t64([g["dy"] for g in grids])][:nd]

    def reduced(Q):
        rho = Q[0]
        e = Q[-1] / rho - 0.5 * (Q[1:-1] ** 2).sum(0) / rho ** 2
        a = (GAMMA * (GAMMA - 1) * e).sqrt()
        rate = sum(((Q[1 + k] / rho).abs() + a) / h[k][pid] for k in range(nd))
        new = torch.zeros(len(grids), dtype=torch.float64, device=dev)
        return (new.scatter_reduce(0, pid, rate, "amax"),
                (new + math.inf).scatter_reduce(0, pid, rho, "amin"))

    def L(Q, mn):
        eps = mn.clamp(max=EPS_POS)
        parts = [_sweep(Q, ln, case, eps) for ln in lines]
        return sum(p[0] for p in parts), sum(p[1] for p in parts)

    def whole(Q):   # back to one [nv, cells] block per problem
        q = torch.cat([b.reshape(-1) for b in torch.split(Q, cells, dim=1)])
        return q.float() if case["form"] == "mixed" else q

    rate, mn = reduced(U)
    if case["call"] == "operator":
        return whole(L(U, mn)[0])
    checked = bool(case.get("checked"))
    cfl = t64([min(g["cfl"], 0.5 * WGL) if checked else g["cfl"] for g in grids])
    t, frate = torch.zeros_like(rate), torch.zeros_like(rate)
    t_final = _t_final(case) if case["call"] == "advance" else math.inf
    left = case["steps"] if case["call"] == "steps" else 1 << 30
    while left > 0 and float(t.min()) < t_final:
        left -= 1
        dt = torch.minimum(cfl / torch.maximum(rate, frate), t_final - t)
        d = dt[pid]
        Q, m, worst = U, mn, torch.zeros_like(rate)
        for c0, c1 in ((0.0, 1.0), (0.75, 0.25), (1.0 / 3.0, 2.0 / 3.0)):
            D, fr = L(Q, m)
            worst = torch.maximum(worst, fr)
            Q = c0 * U + c1 * (Q + d * D)
            r2, m = reduced(Q)
        ok = dt * worst <= WGL if checked else torch.ones_like(rate, dtype=torch.bool)
        U = torch.where(ok[pid], Q, U)
        rate, mn, t = torch.where(ok, r2, rate), torch.where(ok, m, mn), torch.where(ok, t + dt, t)
        frate = torch.where(torch.isfinite(worst), worst, 2 * cfl / dt) if checked else frate
        t = torch.where(t >= t_final * (1 - 1e-14), torch.full_like(t, t_final), t) if t_final < math.inf else t
    return whole(U)
