"""Cases that stand for the work users have this solver do, each through the
public API (`paper_2008_01966_gb300.Cavity`).

Kinds of case (key "kind"):
  solve   the user holds a prepared cavity and solves a batch of incident
          plane waves: aperture coefficients, on request the interior field
          and the backscatter cross-section
  sweep   a wavenumber sweep: every pass visits two wavenumbers, so each solve
          pays for its own preparation (kernel table, elimination,
          preconditioner, and the dense factors where the direct solver is used)
  apply   one application of the aperture operator (the step of a user's own
          iterative solver)
  field   the interior field of given aperture coefficients

All inputs come from the seed: directions, the order of the fill, vectors.
Mixed-precision solves run to 1e-10, where the aperture field no longer
depends on how the iteration got there.
"""

import math

import numpy as np
import torch

from paper_2008_01966_gb300 import Cavity

# relative permittivities of the layered fills (top to bottom, in an order
# drawn from the seed)
EPS = (4 + 1j, 2 + 0.5j, 6 + 0.1j, 1 + 0j)
DEPTH = 0.5


def _case(kind, nx, ny, nz, ndir, **more):
    c = dict(kind=kind, nx=nx, ny=ny, nz=nz, ndir=ndir, b=1.0, layers=1, precision="mixed",
             field=False, rcs=False, solver="krylov", modes=0, points=10.0)
    c.update(more)
    return c


def listed():
    cases = [
        # one plane wave on a small cavity, the default (FP64) precision with
        # the field: the call of a user who tries the method or runs a unit test
        _case("solve", 32, 32, 32, 1, precision="fp64", field=True, name="small_fp64"),
        # backscatter of one small layered cavity for 64 angles, one step of a
        # sweep over many cavities
        _case("solve", 64, 64, 32, 64, layers=3, rcs=True, name="rcs_64"),
        # the same on a medium cavity
        _case("solve", 256, 256, 128, 64, layers=2, rcs=True, name="rcs_256"),
        # interior field of an empty medium cavity for 16 waves
        _case("solve", 256, 256, 128, 16, field=True, name="field_256"),
        # the largest usual case: four layers, 8 waves, the whole field
        _case("solve", 512, 512, 256, 8, layers=4, field=True, name="layered_512"),
        # the largest grid side, aperture only (a shallow cavity)
        _case("solve", 1024, 1024, 64, 3, layers=4, name="aperture_1024"),
        # FP64 throughout on a layered cavity, field included
        _case("solve", 128, 128, 64, 4, layers=4, precision="fp64", field=True,
              name="fp64_128"),
        # two wavenumbers of a frequency sweep, preparation included
        _case("sweep", 128, 128, 64, 16, layers=3, rcs=True, name="sweep_128"),
        # the direct solver on a truncated expansion, assembly and factors of
        # each wavenumber included
        _case("sweep", 128, 128, 64, 16, layers=2, solver="dense", modes=26, rcs=True,
              points=5.0, name="dense_128"),
        # the operator in the three arithmetics, on a rectangle, a square and
        # an odd number of vectors
        _case("apply", 512, 256, 16, 5, precision="mixed", name="apply_fp32"),
        _case("apply", 256, 256, 16, 6, precision="pair32", name="apply_pair32"),
        # the field of three aperture vectors on a rectangular cavity with an
        # odd number of levels
        _case("field", 256, 128, 91, 3, layers=3, name="field_rect"),
    ]
    return cases


def _cost(c):
    """Rough relative cost of a pass (aperture points times vectors, levels
    for the field), to keep drawn cases below the largest listed one."""
    pts = c["nx"] * c["ny"] * c["ndir"]
    w = {"solve": 25, "sweep": 60, "apply": 1, "field": 0}[c["kind"]] * pts
    if c["precision"] == "fp64":
        w *= 20
    if c["precision"] == "pair32":
        w *= 9
    if c["field"] or c["kind"] == "field":
        w += pts * c["nz"] * (4 if c["precision"] == "fp64" else 0.15)
    return w


def draw(rng):
    """One more case: grids of 16 to 1024 intervals per side (squares and
    rectangles), 1 to 64 waves, 1 to 4 layers, odd level counts."""
    limit = 25 * 512 * 512 * 8
    while True:
        kind = rng.choice(["solve", "solve", "solve", "apply", "apply", "field", "field", "sweep"])
        lx = rng.randint(4, 10)
        ly = lx if rng.random() < 0.5 else min(10, max(4, lx + rng.choice([-2, -1, 1, 2])))
        nx, ny = 1 << lx, 1 << ly
        layers = rng.randint(1, 4)
        nz = max(4 * layers, int(round(math.exp(rng.uniform(math.log(8), math.log(180))))))
        ndir = int(round(math.exp(rng.uniform(0, math.log(64)))))
        b = 1.0 if nx == ny else rng.choice([1.0, 0.75, 0.5 if ny < nx else 1.5])
        c = _case(kind, nx, ny, nz, ndir, b=b, layers=layers,
                  points=round(rng.uniform(8.0, 14.0), 2))
        if kind == "apply":
            c["precision"] = rng.choice(["mixed", "fp64", "pair32"])
        elif rng.random() < 0.3:
            c["precision"] = "fp64"
        if kind == "solve":
            c["field"] = rng.random() < 0.5
            c["rcs"] = rng.random() < 0.5
        if kind == "sweep":
            c["rcs"] = True
            if rng.random() < 0.4:
                c["solver"] = "dense"
                c["modes"] = rng.randint(8, min(40, min(nx, ny) - 1))
        if _cost(c) > limit or c["nx"] * c["ny"] * c["nz"] > 2 ** 25 or \
                (max(nx, ny) == 1024 and kind == "sweep"):
            continue
        return c


# ------------------------------------------------------------------ inputs
def _problem(case, seed):
    """Everything of the problem that is drawn from the seed (host values)."""
    rng = np.random.Generator(np.random.PCG64(int(seed)))
    nl, nz = case["layers"], case["nz"]
    base = nz // nl
    lev = [base] * nl
    lev[0] += nz - base * nl
    eps = [1.0 + 0j] if nl == 1 else [EPS[i] for i in rng.permutation(4)[:nl]]
    # `points` grid steps per wavelength in the densest layer, in every
    # direction of the grid
    emax = max(e.real for e in eps)
    step = max(DEPTH / nz, 1.0 / case["nx"], case["b"] / case["ny"])
    kappa = 2 * math.pi / (case["points"] * step * math.sqrt(emax))
    th = rng.uniform(0.0, math.pi / 3, case["ndir"])
    ph = rng.uniform(0.0, 2 * math.pi, case["ndir"])
    al = rng.uniform(0.0, math.pi / 2, case["ndir"])
    return dict(layers=list(zip(lev, eps)), kappa=kappa, theta=th, phi=ph, alpha=al)


def _vectors(case, seed, n, dtype):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) + 77)
    v = torch.randn((case["ndir"], n, 2), generator=gen, device="cuda", dtype=torch.float64)
    return torch.view_as_complex(v).to(dtype)


def _n_ap(case):
    M, N = case["nx"] - 1, case["ny"] - 1
    return 3 * M * N + M + N


class _State:
    pass


def _kappas(case, p):
    return [p["kappa"]] if case["kind"] != "sweep" else [p["kappa"], 0.75 * p["kappa"]]


def prepare(case, seed):
    p = _problem(case, seed)
    s = _State()
    s.case, s.p = dict(case), p
    prec = case["precision"]
    tol = 0.0 if prec == "fp64" else 1e-10
    s.cav = Cavity(a=1.0, b=case["b"], c=DEPTH, nx=case["nx"], ny=case["ny"], nz=case["nz"],
                   precision="fp64" if prec == "fp64" else "mixed", gmres_tol=tol,
                   modes_m=case["modes"], modes_n=case["modes"], aperture_solver=case["solver"])
    if case["kind"] != "sweep":
        s.cav.prepare(p["kappa"], p["layers"])
    if case["kind"] == "apply":
        s.x = _vectors(case, seed, _n_ap(case),
                       torch.complex64 if prec == "mixed" else torch.complex128)
    if case["kind"] == "field":
        s.x = _vectors(case, seed, _n_ap(case), torch.complex128)
    return s


def run(s):
    c, p, cav = s.case, s.p, s.cav
    if c["kind"] == "apply":
        return {"y": cav.apply(s.x, c["precision"])}
    if c["kind"] == "field":
        return {"field": cav.field(s.x)}
    out = []
    for k in _kappas(c, p):
        ap, fl, _, _ = cav.solve(k, p["layers"], p["theta"], p["phi"], p["alpha"],
                                 field=c["field"])
        r = {"aperture": ap}
        if c["field"]:
            r["field"] = fl
        if c["rcs"]:
            r["sigma"] = cav.rcs(ap, p["theta"], p["phi"], "theta")
        out.append(r)
    return out


def work(case):
    """One operator application per vector and wavenumber (four line
    transforms of the padded box along each axis), one field synthesis; the
    resident profiles and the kernel table read once, the outputs written."""
    nx, ny, nz, nd = case["nx"], case["ny"], case["nz"], case["ndir"]
    n, prec = _n_ap(case), case["precision"]
    cb = 16 if prec == "fp64" else 8
    samples = (nx + 1) * (ny - 1) + (nx - 1) * (ny + 1) + (nx - 1) * (ny - 1)
    op = 3 * 5.0 * (nx * 4 * ny * math.log2(4 * ny) * 2 + 4 * ny * 4 * nx * math.log2(4 * nx) * 2)
    syn = 5.0 * 1.5 * 2 * nx * ny * (math.log2(2 * nx) + math.log2(2 * ny))
    prof = n * nz * cb * (1 if case["layers"] == 1 else 5 / 3.0)
    table = 4.0 * nx * ny * cb
    if case["kind"] == "apply":
        vb = 8 if prec == "mixed" else 16
        return {"bytes": 2.0 * n * nd * vb + table, "flops": op * nd}
    if case["kind"] == "field":
        return {"bytes": prof + 16.0 * n * nd + samples * nz * nd * cb, "flops": syn * nz * nd}
    nk = 2 if case["kind"] == "sweep" else 1
    by, fl = 16.0 * n * nd + table, op * nd
    if case["field"]:
        by += prof + samples * nz * nd * cb
        fl += syn * nz * nd
    if case["kind"] == "sweep":
        by += prof                                  # written by the preparation
    if case["solver"] == "dense":
        nk_un = 3.0 * case["modes"] ** 2 + 2 * case["modes"]
        fl += 8.0 / 3 * nk_un ** 3 + 8 * nk_un ** 2 * nd
        by += 8 * nk_un ** 2
    return {"bytes": by * nk, "flops": fl * nk}


# ------------------------------------------------------------------ 64-bit values
# A plain complex128 restatement of the discretised problem with dense factor
# matrices per axis (torch matmul), one GMRES per wave.
def _dev():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _t(x):
    return torch.as_tensor(x, device=_dev())


def _elimination(case, p, kappa):
    """Profiles on the full (m, n) grid: P1, Q1, P2, Q2, P3 [nz + 1, nx, ny]."""
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    h = DEPTH / nz
    mx = _t(np.arange(nx) * np.pi)
    my = _t(np.arange(ny) * np.pi / case["b"])
    lam = mx[:, None] ** 2 + my[None, :] ** 2
    lay, face, top = {}, {}, nz
    for l, (k, _) in enumerate(p["layers"]):
        for j in range(top - k + 1, top):
            lay[j] = l
        top -= k
        if top > 0:
            face[top] = (l, l + 1)
    eps = [e for _, e in p["layers"]]
    sig = [h * h * (kappa ** 2 * e - lam) for e in eps]
    one = torch.ones_like(lam) + 0j
    r3, r = [one], [0 * one]
    for j in range(1, nz):
        if j in face:
            up, lo = face[j]
            r3.append(1 / (1 + eps[up] / eps[lo] * (1 - r3[-1])))
            r.append(-1 / (-2 + r[-1]))
        else:
            r3.append(-1 / (sig[lay[j]] - 2 + r3[-1]))
            r.append(-1 / (sig[lay[j]] - 2 + r[-1]))
    P3 = [None] * (nz + 1)
    P3[nz], low = one, one
    for j in range(nz - 1, 0, -1):
        P3[j] = r3[j] * low              # the value the layer above sees
        low = P3[j]
        if j in face:
            up, lo = face[j]
            low = eps[up] / eps[lo] * P3[j]
    P3[0] = P3[1]
    P = [None] * (nz + 1)
    P[nz] = one
    for j in range(nz - 1, -1, -1):
        P[j] = r[j] * P[j + 1] if j else 0 * one
    # the part driven by E3: T_j = r_j T_{j+1} + s_j, sources on the interfaces
    Q = [None] * (nz + 1)
    Q[nz] = 0 * one
    s = [0 * one]
    for j in range(1, nz):
        f = 0 * one
        if j in face:
            up, lo = face[j]
            f = h * (1 - eps[up] / eps[lo]) * P3[j]
        s.append(-(f - s[-1]) * r[j])
    for j in range(nz - 1, -1, -1):
        Q[j] = r[j] * Q[j + 1] + s[j] if j else 0 * one
    P, Q, P3 = torch.stack(P), torch.stack(Q), torch.stack(P3)
    return P, Q * mx[:, None], P, Q * my[None, :], P3, h


def _j0(x):
    """J0 in 64 bits: torch's function above 30 (its asymptotic branch), the
    trapezoid rule of (1/pi) int_0^pi cos(x sin t) dt below (96 points of the
    full period converge to rounding there)."""
    v = torch.special.bessel_j0(x)
    low = x < 30.0
    xs = x[low]
    t = 0.5 + 0.5 * torch.cos(xs)                   # sin t = 0 and 1, half weights
    for k in range(1, 24):
        t += torch.cos(xs * math.sin(math.pi * k / 48))
    v[low] = t / 24
    return v


def _table(case, kappa):
    """Transform of the truncated Green's function on the quarter box."""
    nx, ny, b = case["nx"], case["ny"], case["b"]
    R = math.sqrt(2.0) * max(1.0, b)
    jx, jy = np.arange(2 * nx), np.arange(2 * ny)
    if 4 * b == 4.0:
        key = jx[:, None] ** 2 + jy[None, :] ** 2
        u, inv = np.unique(key, return_inverse=True)
        rho = np.sqrt(u) / 4.0
    else:
        rho = np.hypot(jx[:, None] / 4.0, jy[None, :] / (4.0 * b)).ravel()
        inv = np.arange(rho.size)
    order = np.argsort(rho)
    val = torch.empty(rho.size, dtype=torch.complex128, device=_dev())
    x, w = np.polynomial.legendre.leggauss(16)
    for part in np.array_split(order, max(1, rho.size // 2000)):
        c = 2 * np.pi * rho[part]
        npan = max(1, int(np.ceil((c.max() + kappa) * R / np.pi)))
        wid = R / npan
        r = (np.arange(npan)[:, None] * wid + 0.5 * wid * (x + 1)).ravel()
        e = _t(np.exp(1j * kappa * r) * np.tile(0.5 * wid * w, npan))
        v = _j0(_t(c)[:, None] * _t(r)[None, :])
        val[_t(part)] = 0.5 * torch.complex(v @ e.real, v @ e.imag)
    q = val[_t(inv.ravel())].reshape(2 * nx, 2 * ny)
    return torch.cat([q[1:].flip(0), q]), q


def _axis(kind, n, side):
    """X[m, j] (inverse DFT at the nodes, trapezoid projection) and Phi[j, k]
    (exact transform of the truncated basis), |j| < 2 n, k < n."""
    j = np.arange(-(2 * n - 1), 2 * n)
    k = np.arange(n)

    def E(d):
        nu = d / (8.0 * side)
        s = np.where(d == 0, 1.0, nu)
        return np.where(d == 0, side + 0j,
                        (1 - np.exp(-2j * np.pi * s * side)) / (2j * np.pi * s))

    em, ep = E(2 * j[:, None] - 4 * k), E(2 * j[:, None] + 4 * k)
    phi = 0.5 * (em + ep) if kind == "c" else (em - ep) / 2j
    q = np.arange(n + 1)
    w = np.full(n + 1, side / n)
    w[[0, -1]] *= 0.5
    base = (np.cos if kind == "c" else np.sin)(np.pi * np.outer(k, q) / n) * w
    inv = np.exp(2j * np.pi * np.outer(q, j) / (4 * n)) / (4 * side)
    return _t(base @ inv), _t(phi)


class _Exact:
    def __init__(self, case, p, kappa):
        self.c, self.k = case, kappa
        self.nx, self.ny, self.b = case["nx"], case["ny"], case["b"]
        self.P1, self.Q1, self.P2, self.Q2, self.P3, self.h = _elimination(case, p, kappa)
        nz = case["nz"]
        self.t1, self.v1 = self.P1[nz - 1], self.Q1[nz - 1]
        self.t2, self.v2, self.t3 = self.P2[nz - 1], self.Q2[nz - 1], self.P3[nz - 1]
        full, _ = _table(case, kappa)
        self.K = torch.cat([full[:, 1:].flip(1), full], 1)
        self.ax = {k: _axis(k, self.nx, 1.0) for k in "cs"}
        self.ay = {k: _axis(k, self.ny, self.b) for k in "cs"}
        self.m = _t(np.arange(self.nx) * np.pi)[:, None]
        self.n = _t(np.arange(self.ny) * np.pi / self.b)[None, :]
        ab = self.b
        self.s1 = _t(np.where(np.arange(self.nx) == 0, 2.0, 4.0) * self.h / ab)[:, None]
        self.s2 = _t(np.where(np.arange(self.ny) == 0, 2.0, 4.0) * self.h / ab)[None, :]
        on = torch.ones((3, self.nx, self.ny), dtype=torch.bool, device=_dev())
        on[0, :, 0] = on[1, 0, :] = on[2, 0, :] = on[2, :, 0] = False
        if case["modes"]:
            on[:, case["modes"] + 1:, :] = False
            on[:, :, case["modes"] + 1:] = False
        self.on = on

    def split(self, x):
        M, N = self.nx - 1, self.ny - 1
        e = torch.zeros((x.shape[0], 3, self.nx, self.ny), dtype=torch.complex128, device=_dev())
        n1, n2 = self.nx * N, M * self.ny
        x = x.to(torch.complex128)
        e[:, 0, :, 1:] = x[:, :n1].reshape(-1, self.nx, N)
        e[:, 1, 1:, :] = x[:, n1:n1 + n2].reshape(-1, M, self.ny)
        e[:, 2, 1:, 1:] = x[:, n1 + n2:].reshape(-1, M, N)
        return e

    def join(self, e):
        nd = e.shape[0]
        return torch.cat([e[:, 0, :, 1:].reshape(nd, -1), e[:, 1, 1:, :].reshape(nd, -1),
                          e[:, 2, 1:, 1:].reshape(nd, -1)], 1)

    def conv(self, kx, ky, c):
        (Xx, Fx), (Xy, Fy) = self.ax[kx], self.ay[ky]
        return Xx @ ((Fx @ c @ Fy.T) * self.K) @ Xy.T

    def diag(self, kx, ky):
        (Xx, Fx), (Xy, Fy) = self.ax[kx], self.ay[ky]
        return (Xx * Fx.T) @ self.K @ (Xy * Fy.T).T

    def apply(self, e):
        y = torch.empty_like(e)
        for d in range(e.shape[0]):
            e1, e2, e3 = e[d]
            U1, U2 = self.conv("c", "s", e1), self.conv("s", "c", e2)
            W = self.conv("c", "c", self.n * e1 - self.m * e2)
            k2 = 2 * self.k ** 2
            y[d, 0] = (self.t1 - 1) * e1 + (self.m * self.h + self.v1) * e3 \
                + self.s1 * (k2 * U1 - 2 * self.n * W)
            y[d, 1] = (self.t2 - 1) * e2 + (self.n * self.h + self.v2) * e3 \
                + self.s2 * (k2 * U2 + 2 * self.m * W)
            y[d, 2] = self.m * self.h * e1 + self.n * self.h * e2 + (self.t3 - 1) * e3
        return y * self.on

    def precond(self):
        d1, d2, d3 = self.diag("c", "s"), self.diag("s", "c"), self.diag("c", "c")
        k2, h, m, n = 2 * self.k ** 2, self.h, self.m, self.n
        B = torch.zeros((self.nx, self.ny, 3, 3), dtype=torch.complex128, device=_dev())
        B[..., 0, 0] = self.t1 - 1 + self.s1 * (k2 * d1 - 2 * n * n * d3)
        B[..., 0, 1] = self.s1 * 2 * n * m * d3
        B[..., 0, 2] = m * h + self.v1
        B[..., 1, 0] = self.s2 * 2 * m * n * d3
        B[..., 1, 1] = self.t2 - 1 + self.s2 * (k2 * d2 - 2 * m * m * d3)
        B[..., 1, 2] = n * h + self.v2
        B[..., 2, 0], B[..., 2, 1] = m * h + 0 * n, n * h + 0 * m
        B[..., 2, 2] = self.t3 - 1
        on = self.on.permute(1, 2, 0)
        keep = on[..., :, None] & on[..., None, :]
        B = torch.where(keep, B, torch.zeros_like(B))
        B = B + torch.diag_embed((~on).to(torch.complex128))
        return torch.linalg.inv(B)

    def rhs(self, p):
        out = []
        for t, f, al in zip(p["theta"], p["phi"], p["alpha"]):
            a1 = -self.k * math.sin(t) * math.cos(f)
            a2 = -self.k * math.sin(t) * math.sin(f)
            be = self.k * math.cos(t)
            th = np.array([math.cos(t) * math.cos(f), math.cos(t) * math.sin(f), -math.sin(t)])
            pv = math.cos(al) * th + math.sin(al) * np.array([-math.sin(f), math.cos(f), 0.0])

            def proj(kind, n, side, g):
                q = np.arange(n + 1)
                w = np.full(n + 1, side / n)
                w[[0, -1]] *= 0.5
                base = (np.cos if kind == "c" else np.sin)(np.pi * np.outer(np.arange(n), q) / n)
                return _t((base * w) @ np.exp(1j * g * q * side / n))

            e = torch.zeros((3, self.nx, self.ny), dtype=torch.complex128, device=_dev())
            e[0] = self.s1 * 2j * (a1 * pv[2] + be * pv[0]) * torch.outer(
                proj("c", self.nx, 1.0, a1), proj("s", self.ny, self.b, a2))
            e[1] = self.s2 * 2j * (a2 * pv[2] + be * pv[1]) * torch.outer(
                proj("s", self.nx, 1.0, a1), proj("c", self.ny, self.b, a2))
            out.append(e)
        return torch.stack(out) * self.on

    def solve(self, p, steps=90):
        b = self.rhs(p)
        nd = b.shape[0]
        Minv = self.precond()
        pre = lambda v: torch.einsum("mnrc,dcmn->drmn", Minv, v) * self.on  # noqa: E731
        x = torch.zeros_like(b)
        for _ in range(2):                       # one restart from the true residual
            r = b - self.apply(x) if bool(x.abs().max() > 0) else b
            beta = r.reshape(nd, -1).norm(dim=1)
            V = [r / beta[:, None, None, None]]
            H = torch.zeros((nd, steps + 1, steps), dtype=torch.complex128, device=_dev())
            k = 0
            for k in range(steps):
                w = self.apply(pre(V[k]))
                for _again in range(2):
                    for i in range(k + 1):
                        g = (V[i].conj() * w).sum(dim=(1, 2, 3))
                        H[:, i, k] += g
                        w = w - g[:, None, None, None] * V[i]
                hn = w.reshape(nd, -1).norm(dim=1)
                H[:, k + 1, k] = hn
                V.append(w / hn[:, None, None, None])
                if k % 4 == 3 or k == steps - 1:
                    e1 = torch.zeros((nd, k + 2, 1), dtype=torch.complex128, device=_dev())
                    e1[:, 0, 0] = beta
                    Hk = H[:, :k + 2, :k + 1]
                    Qr, Rr = torch.linalg.qr(Hk)
                    y = torch.linalg.solve_triangular(Rr, Qr.mH @ e1, upper=True)
                    res = (Hk @ y - e1).reshape(nd, -1).norm(dim=1)
                    if bool((res <= 2e-13 * beta).all()) or bool((res <= 1e-14 * b.reshape(
                            nd, -1).norm(dim=1)).all()):
                        break
            z = sum(y[:, i, 0][:, None, None, None] * V[i] for i in range(k + 1))
            x = x + pre(z)
        return x

    def field(self, e):
        nx, ny, nz = self.nx, self.ny, self.c["nz"]
        px, py = np.arange(nx + 1), np.arange(ny + 1)
        cx = _t(np.cos(np.pi * np.outer(px, np.arange(nx)) / nx)) + 0j
        sx = _t(np.sin(np.pi * np.outer(px[1:-1], np.arange(nx)) / nx)) + 0j
        cy = _t(np.cos(np.pi * np.outer(py, np.arange(ny)) / ny)) + 0j
        sy = _t(np.sin(np.pi * np.outer(py[1:-1], np.arange(ny)) / ny)) + 0j
        out = []
        for d in range(e.shape[0]):
            rows = []
            for j in range(1, nz + 1):
                c1 = self.P1[j] * e[d, 0] + self.Q1[j] * e[d, 2]
                c2 = self.P2[j] * e[d, 1] + self.Q2[j] * e[d, 2]
                c3 = self.P3[j] * e[d, 2]
                rows.append(torch.cat([(cx @ c1 @ sy.T).reshape(-1), (sx @ c2 @ cy.T).reshape(-1),
                                       (sx @ c3 @ sy.T).reshape(-1)]))
            out.append(torch.cat(rows))
        return torch.stack(out)

    def sigma(self, e, p):
        out = []

        def ints(kind, n, side, g):
            k = np.arange(n) * np.pi / side

            def ef(s):
                z = np.where(s == 0, 1.0, s)
                return np.where(s == 0, side + 0j, (1 - np.exp(-1j * z * side)) / (1j * z))

            v = 0.5 * (ef(g - k) + ef(g + k)) if kind == "c" else (ef(g - k) - ef(g + k)) / 2j
            return _t(v)

        for d, (t, f) in enumerate(zip(p["theta"], p["phi"])):
            xh = np.array([math.sin(t) * math.cos(f), math.sin(t) * math.sin(f), math.cos(t)])
            g1, g2 = self.k * xh[0], self.k * xh[1]
            I1 = ints("c", self.nx, 1.0, g1) @ e[d, 0] @ ints("s", self.ny, self.b, g2)
            I2 = ints("s", self.nx, 1.0, g1) @ e[d, 1] @ ints("c", self.ny, self.b, g2)
            L = np.array([-complex(I2), complex(I1), 0.0])
            th = np.array([math.cos(t) * math.cos(f), math.cos(t) * math.sin(f), -math.sin(t)])
            out.append(self.k ** 2 / math.pi * abs(np.dot(th, np.cross(xh, L))) ** 2)
        return np.array(out)


def exact(case, seed):
    """complex128 values of run(); None where they take too long."""
    nx, ny, nz, nd = case["nx"], case["ny"], case["nz"], case["ndir"]
    app = 3 * nd * 8.0 * (4 * nx * nx * ny + 16 * nx * ny * ny + 16 * nx * nx * ny)
    app *= 30 * len(_kappas(case, {"kappa": 1})) if case["kind"] in ("solve", "sweep") else 1
    syn = nz * nd * 48.0 * nx * ny * (nx + ny) if case["field"] or case["kind"] == "field" else 0
    if (0 if case["kind"] == "field" else app) + syn > 8e12 or nx * ny * nz > 2 ** 23 + 2 ** 18:
        return None
    if nx * ny > 2 ** 18:
        return None                              # the kernel table alone takes too long
    p = _problem(case, seed)
    if case["kind"] == "apply":
        x = _vectors(case, seed, _n_ap(case),
                     torch.complex64 if case["precision"] == "mixed" else torch.complex128)
        s = _Exact(case, p, p["kappa"])
        return {"y": s.join(s.apply(s.split(x)))}
    if case["kind"] == "field":
        s = _Exact(case, p, p["kappa"])
        return {"field": s.field(s.split(_vectors(case, seed, _n_ap(case), torch.complex128)))}
    out = []
    for k in _kappas(case, p):
        s = _Exact(case, p, k)
        e = s.solve(p)
        r = {"aperture": s.join(e)}
        if case["field"]:
            r["field"] = s.field(e)
        if case["rcs"]:
            r["sigma"] = s.sigma(e, p)
        out.append(r)
    return out
