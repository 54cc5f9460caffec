"""Performance cases: what a user of the solver has it do, over the sizes it is used at.

A case is a dict of plain values.  `kind` says which call it stands for:

  iteration  Solver.design_iteration on cached factors: the inner loop of adjoint inverse design
             (design refactor, forward solves, objective, adjoint solves, pixel gradient)
  solve      Solver.solve forward and transposed with many sources on one cached factorisation
             (scattering parameters, several ports or modes per wavelength)
  structure  Solver.factor of a new permittivity on the whole grid, then one forward solve
             (evaluating a structure, or the first call of a loop)
  density    filter + projection of the density, the differentiable objective and its backward pass
             through autograd (a user's own optimiser in torch)

Grids are nx x ny cells with npml absorbing cells on each side, silicon guides on oxide, a centred
design box of a blurred random density, n_omega wavelengths and nrhs sources per wavelength.  Every
case refines to ir_tol = 1e-11: two digits below the 1e-9 default, so that objective values of weakly
transmitting random devices keep nine digits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2307_05388_gb300 import autograd as AG
from paper_2307_05388_gb300 import fdfd as FD

EPS_LO, EPS_HI = 2.085, 12.11      # oxide, silicon
LARGEST = 2 * (1760 * 1760) ** 1.5  # n_omega * cells^1.5 of the largest listed case
MOST_SYSTEMS = 4 * 1760 * 1760     # unknowns over all systems of the largest listed case
IR_TOL = 1e-11


def _case(name, kind, nx, ny, npml, bw, bh, n_omega, nrhs, dx=0.04, lam0=1.50, lam1=1.60, mode="mixed",
          target=False):
    c = dict(kind=kind, nx=nx, ny=ny, npml=npml, bw=bw, bh=bh, n_omega=n_omega, nrhs=nrhs, dx=dx, lam0=lam0,
             lam1=lam1, mode=mode, target=target)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # a 4 um coupler at 50 nm cells: the smallest device; launches and latency count
        _case("iteration 100x100", "iteration", 100, 100, 10, 40, 40, 1, 1, dx=0.05, lam0=1.55, lam1=1.55),
        # a single-wavelength waveguide device, the most common single design problem
        _case("iteration 340x340", "iteration", 340, 340, 20, 250, 250, 1, 1, lam0=1.55, lam1=1.55),
        # a mode multiplexer: eight wavelengths, two sources each, transmission targets
        _case("iteration 540x540 8x2", "iteration", 540, 540, 20, 400, 400, 8, 2, target=True),
        # a large broadband device
        _case("iteration 1040x1040 4x1", "iteration", 1040, 1040, 20, 900, 900, 4, 1, lam0=1.53, lam1=1.57),
        # the largest footprint: a duplexer at two bands with two modes each
        _case("iteration 1760x1760 2x2", "iteration", 1760, 1760, 20, 1680, 1680, 2, 2, dx=0.05, lam0=1.31, lam1=1.55),
        # a long ragged device (a taper or a grating) at three wavelengths
        _case("iteration 713x259 3x1", "iteration", 713, 259, 15, 602, 181, 3, 1),
        # many sources on one factorisation: an eight-port scattering matrix, forward and transposed
        _case("solve 540x540 1x8", "solve", 540, 540, 20, 400, 400, 1, 8, lam0=1.55, lam1=1.55),
        # the same for a large grid with few ports
        _case("solve 1201x903 2x3", "solve", 1201, 903, 20, 1001, 701, 2, 3),
        # evaluating a new structure: full factorisation and one solve, ragged grid
        _case("structure 457x331 2x1", "structure", 457, 331, 17, 0, 0, 2, 1),
        # double-precision factors (no refinement), for users who want direct complex128 solves
        _case("iteration f64 200x200", "iteration", 200, 200, 15, 150, 150, 1, 1, dx=0.05, mode="f64"),
        # a differentiable loop: filter, projection, objective and backward at a small grid
        _case("density 200x200 4x1", "density", 200, 200, 20, 150, 150, 4, 1, lam0=1.53, lam1=1.57),
        # the same at a mid-size grid
        _case("density 640x480 2x1", "density", 640, 480, 20, 560, 400, 2, 1),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["iteration", "iteration", "iteration", "solve", "structure", "density"])
    mode = "f64" if kind == "iteration" and rng.random() < 0.15 else "mixed"
    top = 260 if mode == "f64" else 900 if kind == "density" else 1760
    while True:
        side = _log_uniform(rng, 90, top)
        nx = int(min(1760, max(80, side * rng.uniform(0.7, 1.4))))
        ny = int(min(1760, max(80, side * side / nx)))
        n_omega = rng.randint(1, 8)
        nrhs = rng.randint(2, 8) if kind == "solve" else rng.randint(1, 2) if kind == "iteration" else 1
        if n_omega * (nx * ny) ** 1.5 <= LARGEST and n_omega * nrhs * nx * ny <= MOST_SYSTEMS:
            break
    npml = rng.randint(10, 20)
    room_x, room_y = nx - 2 * npml - 8, ny - 2 * npml - 8
    bw = bh = 0
    if kind != "structure":
        bw, bh = int(room_x * rng.uniform(0.5, 1.0)), int(room_y * rng.uniform(0.5, 1.0))
    return _case("", kind, nx, ny, npml, bw, bh, n_omega, nrhs, dx=rng.choice([0.04, 0.05]), lam0=1.50, lam1=1.60,
                 mode=mode, target=rng.random() < 0.5)


# ---------------------------------------------------------------------------
# inputs (plain torch, from the seed alone)
# ---------------------------------------------------------------------------
def _wavelengths(case):
    n = case["n_omega"]
    return np.linspace(case["lam0"], case["lam1"], n) if n > 1 else np.array([case["lam0"]])


def _box(case):
    bw, bh = case["bw"], case["bh"]
    return ((case["nx"] - bw) // 2, (case["ny"] - bh) // 2, bw, bh) if bw and bh else (0, 0, 0, 0)


def _blurred(gen, w, h, dev):
    """A random density in [0, 1] smoothed over 8 x 8 cells."""
    r = torch.rand((1, 1, w + 7, h + 7), generator=gen, device=dev, dtype=torch.float64)
    return torch.nn.functional.avg_pool2d(r, 8, stride=1)[0, 0].contiguous()


def _profile(order, u):
    """Hermite-Gauss profiles of a guide, order 0, 1, 2, ..."""
    h0, h1 = torch.ones_like(u), 2.0 * u
    for n in range(1, order + 1):
        h0, h1 = h1, 2.0 * u * h1 - 2.0 * n * h0
    p = h0 * torch.exp(-u * u / 2)
    return p / p.norm()


def _inputs(case, seed):
    dev = torch.device("cuda")
    gen = torch.Generator(device=dev)
    gen.manual_seed(int(seed))
    nx, ny, npml, dx = case["nx"], case["ny"], case["npml"], case["dx"]
    nw, nr = case["n_omega"], case["nrhs"]
    x0, y0, bw, bh = _box(case)
    f8 = dict(dtype=torch.float64, device=dev)
    # oxide with a 0.5 um silicon guide through the middle; the design box (or, for a new structure,
    # everything between the absorbers) holds the density
    eps = torch.full((nx, ny), EPS_LO, **f8)
    half = max(1, int(round(0.25 / dx)))
    eps[:, ny // 2 - half:ny // 2 + half] = EPS_HI
    if bw:
        rho = _blurred(gen, bw, bh, dev)
    else:
        inner = _blurred(gen, nx - 2 * npml - 8, ny - 2 * npml - 8, dev)
        eps[npml + 4:nx - npml - 4, npml + 4:ny - npml - 4] = EPS_LO + inner * (EPS_HI - EPS_LO)
        rho = None
    j = torch.arange(ny, **f8)
    b = torch.zeros((nw, nr, nx, ny), dtype=torch.complex128, device=dev)
    g = torch.zeros((nw, nr, ny), dtype=torch.complex128, device=dev)
    for w in range(nw):
        for r in range(nr):
            if case["kind"] == "solve":      # ports spread over the sides, alternating left and right
                centre = npml + (ny - 2 * npml) * (r + 0.5) / nr
                col = npml if r % 2 == 0 else nx - npml - 1
                b[w, r, col] = -1j * _profile(0, (j - centre) * dx / 0.4)
            else:
                b[w, r, npml] = -1j * _profile(r, (j - ny / 2 + 0.5) * dx / 0.4)
            g[w, r] = _profile(r % 2, (j - ny / 2 + 0.5) * dx / 0.6)
    inside = (j >= npml) & (j < ny - npml)
    b *= inside
    g *= inside
    phase = torch.rand((nw, nr), generator=gen, **f8) * (2 * math.pi)   # the sources' relative phases
    b *= torch.polar(torch.ones_like(phase), phase)[:, :, None, None]
    cols = torch.full((nw * nr,), nx - npml - 1, dtype=torch.int32, device=dev)
    # desired transmissions, of the order that such a random device reaches
    target = torch.rand((nw * nr,), generator=gen, **f8) if case["target"] and case["kind"] == "iteration" else None
    return dict(eps=eps, rho=rho, b=b.reshape(nw, nr, nx * ny), g=g.reshape(nw * nr, ny), cols=cols, target=target,
                box=(x0, y0, bw, bh))


RADIUS, BETA, ETA = 5.0, 8.0, 0.5   # 200 nm filter at 40 nm cells and the usual projection


def prepare(case, seed):
    d = _inputs(case, seed)
    mode = FD.MODE_F64 if case["mode"] == "f64" else FD.MODE_MIXED
    solver = FD.Solver(case["nx"], case["ny"], case["dx"], 2 * np.pi / _wavelengths(case), case["npml"],
                       box=d["box"], options=FD.default_options(mode=mode, ir_tol=IR_TOL))
    st = dict(case=case, solver=solver, **d)
    x0, y0, bw, bh = d["box"]
    kind = case["kind"]
    if kind == "iteration":
        # the loop's first factorisation: a plain oxide box; the design arrives with each call
        solver.factor(d["eps"])
        st["eps_d"] = (EPS_LO + d["rho"] * (EPS_HI - EPS_LO)).reshape(-1).contiguous()
        st["x"], st["xa"] = torch.empty_like(d["b"]), torch.empty_like(d["b"])
    elif kind == "solve":
        d["eps"][x0:x0 + bw, y0:y0 + bh] = EPS_LO + d["rho"] * (EPS_HI - EPS_LO)
        solver.factor(d["eps"])
        st["x"], st["xt"] = torch.empty_like(d["b"]), torch.empty_like(d["b"])
    elif kind == "structure":
        solver.analyze()
    else:
        st["problem"] = AG.DesignProblem(solver, d["eps"], d["b"], d["cols"], d["g"])
        solver.factor(d["eps"])
        st["problem"].factored = True
    return st


def run(st):
    s, kind = st["solver"], st["case"]["kind"]
    if kind == "iteration":
        F, grad = s.design_iteration(st["eps_d"], st["b"], st["cols"], st["g"], target=st["target"],
                                     x_out=st["x"], xadj_out=st["xa"])
        return {"F": F, "grad": grad, "x": st["x"], "xadj": st["xa"]}
    if kind == "solve":
        return {"x": s.solve(st["b"], out=st["x"]), "xt": s.solve(st["b"], transpose=True, out=st["xt"])}
    if kind == "structure":
        s.factor(st["eps"])
        return {"x": s.solve(st["b"])}
    rho = st["rho"].clone().requires_grad_(True)
    eps = AG.FilterProject.apply(rho, s, RADIUS, BETA, ETA, EPS_LO, EPS_HI)
    F = st["problem"](eps)
    F.backward()
    return {"F": F.detach(), "grad": rho.grad, "eps": eps.detach()}


def work(case):
    """Operations: the sparse LU of an n x n grid in nested-dissection order takes 2 * 9.87 n^3 complex
    multiply-adds (8 flops each); the fronts outside the design box are not redone (their share is at
    most the box's share of the grid).  Each solve takes two multiply-adds (8 flops each) per factor
    entry, 7.75 n^2 log2 n entries in L and as many in U.  Bytes: the inputs and outputs once, the
    factor written once and read once by each of the solves, which share one pass over it."""
    n = case["nx"] * case["ny"]
    nw, nr, kind = case["n_omega"], case["nrhs"], case["kind"]
    es = 16 if case["mode"] == "f64" else 8
    share = 1.0 if kind == "structure" else case["bw"] * case["bh"] / n
    factor = 0.0 if kind == "solve" else 8 * 2 * 9.87 * n ** 1.5 * nw * share
    entries = 2 * 7.75 * n * math.log2(math.sqrt(n)) * nw
    solves = 1 if kind == "structure" else 2
    flops = factor + 8 * entries * nr * solves
    by = 16 * n * nw * nr * 2 * solves + es * entries * solves
    if kind != "solve":
        by += es * entries * share + 16 * case["bw"] * case["bh"] + (8 * n if kind == "structure" else 0)
    if kind == "density":
        taps = math.pi * RADIUS ** 2
        by += 8 * case["bw"] * case["bh"] * 6
        flops += 2 * 2 * taps * case["bw"] * case["bh"]
    return {"bytes": by, "flops": flops}


# ---------------------------------------------------------------------------
# the same results in 64 bits, plain torch: block elimination along x
# ---------------------------------------------------------------------------
def _tables(n, npml, k0dx, dev):
    """Lower, upper and centre couplings of one axis with its absorbing layers."""
    def s(u):
        d = torch.clamp(torch.maximum(npml - u, u - (n - npml)), min=0) / npml
        smax = -4 * math.log(1e-8) / (2 * k0dx * npml)
        return torch.complex(torch.ones_like(u), -smax * d ** 3)
    c = torch.arange(n, dtype=torch.float64, device=dev)
    mid = s(c + 0.5)
    return -1 / (mid * s(c)), -1 / (mid * s(c + 1))


def _solve_exact(case, k0dx, eps, rhs, rhs_t):
    """x = A^-1 rhs and y = A^-T rhs_t ([nx, ny, columns] each, or a function of x) for one wavelength."""
    nx, ny, npml = case["nx"], case["ny"], case["npml"]
    dev = eps.device
    xm, xp = _tables(nx, npml, k0dx, dev)
    ym, yp = _tables(ny, npml, k0dx, dev)
    inv = torch.empty((nx, ny, ny), dtype=torch.complex128, device=dev)
    off = torch.diag(ym[1:], -1) + torch.diag(yp[:-1], 1)
    xml, xpl = xm.cpu().tolist(), xp.cpu().tolist()
    for i in range(nx):
        t = off + torch.diag(-(xm[i] + xp[i] + ym + yp) - k0dx ** 2 * eps[i])
        if i:
            t = t - (xml[i] * xpl[i - 1]) * inv[i - 1]
        inv[i] = torch.linalg.inv(t)
    def sweep(b, transposed):
        low = [0j] + (xpl[:-1] if transposed else xml[1:])     # coupling of row i to row i - 1
        up = (xml[1:] if transposed else xpl[:-1]) + [0j]      # ... to row i + 1
        z = b.clone()
        m = (lambda i, v: inv[i].T @ v) if transposed else (lambda i, v: inv[i] @ v)
        for i in range(1, nx):
            z[i] -= low[i] * m(i - 1, z[i - 1])
        x = torch.empty_like(z)
        x[nx - 1] = m(nx - 1, z[nx - 1])
        for i in range(nx - 2, -1, -1):
            x[i] = m(i, z[i] - up[i] * x[i + 1])
        return x
    def apply(x, transposed):
        low = torch.cat([torch.zeros_like(xm[:1]), xp[:-1] if transposed else xm[1:]])
        up = torch.cat([xm[1:] if transposed else xp[:-1], torch.zeros_like(xm[:1])])
        lo_y = torch.cat([torch.zeros_like(ym[:1]), yp[:-1] if transposed else ym[1:]])
        up_y = torch.cat([ym[1:] if transposed else yp[:-1], torch.zeros_like(ym[:1])])
        y = (-(xm + xp)[:, None] - (ym + yp)[None] - k0dx ** 2 * eps)[..., None] * x
        y[1:] += low[1:, None, None] * x[:-1]
        y[:-1] += up[:-1, None, None] * x[1:]
        y[:, 1:] += lo_y[None, 1:, None] * x[:, :-1]
        y[:, :-1] += up_y[None, :-1, None] * x[:, 1:]
        return y
    def solve(b, transposed):
        x = sweep(b, transposed)
        for _ in range(2):
            x = x + sweep(b - apply(x, transposed), transposed)
        return x
    x = solve(rhs, False)
    b2 = rhs_t(x) if callable(rhs_t) else rhs_t
    return x, (solve(b2, True) if b2 is not None else None)


def _filter_exact(rho):
    """(permittivity, function from dF/deps to dF/drho) of the conic filter and tanh projection."""
    r = int(math.ceil(RADIUS))
    k = torch.arange(-r, r + 1, dtype=torch.float64, device=rho.device)
    wt = torch.clamp(RADIUS - torch.sqrt(k[:, None] ** 2 + k[None] ** 2), min=0)
    w, h = rho.shape
    def conv(a):
        p = torch.nn.functional.pad(a, (r, r, r, r))
        out = torch.zeros_like(a)
        for di in range(2 * r + 1):
            for dj in range(2 * r + 1):
                out += wt[di, dj] * p[di:di + w, dj:dj + h]
        return out
    norm = conv(torch.ones_like(rho))
    den = math.tanh(BETA * ETA) + math.tanh(BETA * (1 - ETA))
    th = torch.tanh(BETA * (conv(rho) / norm - ETA))
    eps = EPS_LO + (math.tanh(BETA * ETA) + th) / den * (EPS_HI - EPS_LO)
    slope = BETA * (1 - th * th) / den * (EPS_HI - EPS_LO)
    return eps, lambda g: conv(g * slope / norm)


def exact(case, seed):
    n, nx, ny = case["nx"] * case["ny"], case["nx"], case["ny"]
    if case["n_omega"] * nx * (0.004 + ny ** 3 * 4e-11) > 12:   # the inversions would take too long
        return None
    d = _inputs(case, seed)
    nw, nr, kind = case["n_omega"], case["nrhs"], case["kind"]
    x0, y0, bw, bh = d["box"]
    eps, chain = d["eps"], None
    if bw:
        eps_d = EPS_LO + d["rho"] * (EPS_HI - EPS_LO)
        if kind == "density":
            eps_d, chain = _filter_exact(d["rho"])
        eps[x0:x0 + bw, y0:y0 + bh] = eps_d
    k0dx = 2 * np.pi / _wavelengths(case) * case["dx"]
    b = d["b"].reshape(nw, nr, nx, ny)
    g = d["g"].reshape(nw, nr, ny)
    col = nx - case["npml"] - 1
    F = torch.zeros((), dtype=torch.float64, device=eps.device)
    grad = torch.zeros((bw, bh), dtype=torch.float64, device=eps.device)
    xs, ys = [], []
    for w in range(nw):
        rhs = b[w].permute(1, 2, 0).contiguous()
        over = {}
        def adjoint(x):
            o = (g[w].T * x[col]).sum(0)                      # [nr]
            p = o.abs() ** 2
            t = d["target"][w * nr:(w + 1) * nr] if d["target"] is not None else None
            over["F"] = ((p - t) ** 2).sum() if t is not None else p.sum()
            s = (2 * (p - t) if t is not None else torch.ones_like(p)) * o.conj()
            b2 = torch.zeros_like(x)
            b2[col] = s[None] * g[w].T
            return b2
        x, y = _solve_exact(case, float(k0dx[w]), eps, rhs,
                            rhs if kind == "solve" else None if kind == "structure" else adjoint)
        xs.append(x.permute(2, 0, 1).reshape(nr, n))
        if y is not None:
            ys.append(y.permute(2, 0, 1).reshape(nr, n))
        if kind in ("iteration", "density"):
            F += over["F"]
            grad += 2 * float(k0dx[w]) ** 2 * (x * y).real.sum(-1)[x0:x0 + bw, y0:y0 + bh]
    x = torch.stack(xs)
    if kind == "iteration":
        return {"F": F, "grad": grad.reshape(-1), "x": x, "xadj": torch.stack(ys)}
    if kind == "solve":
        return {"x": x, "xt": torch.stack(ys)}
    if kind == "structure":
        return {"x": x}
    return {"F": F, "grad": chain(grad), "eps": eps_d}
