"""Performance cases: the calls a user of the solver makes, over the sizes and options they are made with.

Every case goes through the public binding of the C ABI (``paper_2005_05398_gb300.Context``).  A case names
the three-body problem (system, total momentum J, spline grid), the call and its options:

* ``apply``    y = (H - E S) x, the matrix-free operator (any outer iteration of the user's own);
* ``precond``  y = P^{-1} x, the tensor preconditioner, in float64 (the library's default precision);
* ``solve``    (H - E S) x = b to the default relative residual 1e-12, in the three precision modes;
* ``eigs``     the level nearest a shift with its eigenvector.

Problems: He, H- and Ps- with identical electrons, on the library's cubic and quintic Hermite grids.
``exact`` restates the operator, the preconditioner and the solves in plain float64 numpy / torch.
"""
import math
from concurrent.futures import ThreadPoolExecutor

import numpy as np
import torch

import paper_2005_05398_gb300 as fm

MASS = {"He": (1.0, 1.0, 1e15), "Hminus": (1.0, 1.0, 1e15), "Psminus": (1.0, 1.0, 1.0)}
CHARGE = {"He": (-1.0, -1.0, 2.0), "Hminus": (-1.0, -1.0, 1.0), "Psminus": (-1.0, -1.0, 1.0)}
NU, X0, VS_CUT = 2.01, 1.0, 1e-20  # Merkuriev splitting
FP64, FP32, MIXED = 0, 1, 2


def _case(call, system, J, n, R, E, precision=FP64, n3=None, R3=None, basis=0, name=None):
    n3, R3 = n3 or n, R3 or R
    c = {"call": call, "system": system, "J": J, "basis": basis, "precision": precision, "E": E,
         "nx": n[0], "ny": n[1], "nz": n[2], "Rx": R[0], "Ry": R[1],
         "nx3": n3[0], "ny3": n3[1], "nz3": n3[2], "Rx3": R3[0], "Ry3": R3[1]}
    return dict({"name": name}, **c) if name else c


def listed():
    he, ps, b40, b80 = "He", "Psminus", (40.0, 40.0), (80.0, 80.0)
    return [
        # one operator application on a quick-look grid (83 k unknowns): launches and latency
        _case("apply", he, 0, (24, 24, 8), b40, -2.95, name="apply_he_small"),
        # the same on the production grid of the ground state (3.7 M unknowns)
        _case("apply", he, 0, (96, 96, 24), b40, -2.95, name="apply_he_large"),
        # four coupled M' components (4.5 M unknowns)
        _case("apply", ps, 3, (64, 64, 16), b80, -0.35, name="apply_psm_l3"),
        # the paper's 3^1D convergence study: quintic splines, a box per component, odd sizes (166, 52, 40)
        _case("apply", he, 2, (55, 55, 7), (45.0, 45.0), -2.2, n3=(17, 13, 8), R3=(11.0, 6.0), basis=1,
              name="apply_he_3d_quintic"),
        # the preconditioner in the default precision, one M' component (dense mode products, diagonal z modes)
        _case("precond", he, 0, (96, 96, 24), b40, -2.95, name="precond_he_large"),
        # the preconditioner with M' chains (banded y systems of three coupled components)
        _case("precond", ps, 2, (64, 64, 16), b80, -0.35, name="precond_psm_l2"),
        # a whole solve with the default options on the quick-look grid
        _case("solve", he, 0, (24, 24, 8), b40, -2.95, name="solve_he_small"),
        # the paper's comparison table (J = 1, quintic, largest of its bases: 114 k unknowns), default options
        _case("solve", he, 1, (19, 19, 3), (36.0, 36.0), -2.2, n3=(9, 9, 6), R3=(9.0, 6.0), basis=1,
              name="solve_he_j1_quintic"),
        # production solve with the float32 tensor-core preconditioner
        _case("solve", he, 0, (96, 96, 24), b40, -2.95, FP32, name="solve_he_large_fp32"),
        # mixed precision: float32 inner solves inside the float64 iteration, three M' components
        _case("solve", ps, 2, (64, 64, 16), b80, -0.35, MIXED, name="solve_psm_l2_mixed"),
        # a served request of odd sizes (radial counts 74 and 102: the float32 CUDA-core mode products)
        _case("solve", "Hminus", 3, (37, 51, 9), b40, -0.8, FP32, name="solve_hm_l3_ragged"),
        # the headline: the He ground state, shift-invert Arnoldi around the float32-preconditioned solves
        _case("eigs", he, 0, (96, 96, 24), b40, -2.95, FP32, name="eigs_he_large"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A problem of the served mixes: system, momentum, interval counts (equal or ragged), energy, call, precision.

    Energies of solves lie below the system's continuum thresholds, where bound states are computed."""
    while True:
        call = rng.choice(["apply", "apply", "precond", "solve", "solve", "solve"])
        system = rng.choice(["He", "Hminus", "Psminus"])
        J = rng.randint(0, 2) if call == "precond" else rng.randint(0, 4)
        quintic = rng.random() < 0.25
        lo, hi, zlo, zhi = (6, 64, 2, 8) if quintic else (8, 128, 3, 24)
        nx = _log_int(rng, lo, hi)
        ny = nx if rng.random() < 0.4 else _log_int(rng, lo, hi)
        n = (nx, ny, rng.randint(zlo, 6 if quintic and call == "precond" else zhi))
        R = 80.0 if system == "Psminus" else 40.0
        E = rng.uniform(*{"He": (-2.87, -2.2), "Hminus": (-3.0, -0.6), "Psminus": (-3.0, -0.3)}[system])
        precision = rng.choice([FP64, FP32, MIXED]) if call == "solve" else FP64
        c = _case(call, system, J, n, (R, R), round(E, 6), precision, basis=int(quintic))
        cap = {"apply": 4.0e6, "precond": 3.0e6, "solve": 4.0e5 if quintic else 1.0e6}[call]
        if _unknowns(c) <= cap:
            return c


# ---------------------------------------------------------------------------------------------------
# what a user's program holds, and the call
# ---------------------------------------------------------------------------------------------------
def _workload(c):
    w = {"mass": MASS[c["system"]], "charge": CHARGE[c["system"]], "J": c["J"], "tau": 1, "p": 1,
         "identical_pair": 12, "nint": (c["nx"], c["ny"], c["nz"]), "R": (c["Rx"], c["Ry"]), "maps": (0, 0, 2),
         "mode": 0, "nu": NU, "x0": X0, "y0": float("inf"), "vs_cut": VS_CUT, "basis": c["basis"]}
    n3, R3 = (c["nx3"], c["ny3"], c["nz3"]), (c["Rx3"], c["Ry3"])
    if n3 != w["nint"] or R3 != w["R"]:
        w["grids"] = {1: {"nint": w["nint"], "R": w["R"]}, 3: {"nint": n3, "R": R3}}
    return w


def _input(n, seed):
    g = torch.Generator(device="cpu").manual_seed(int(seed))
    return torch.randn(n, dtype=torch.float64, generator=g)


def prepare(case, seed):
    ctx = fm.Context(_workload(case), precision=case["precision"])
    if case["call"] != "apply":
        ctx.fm_set_shift(case["E"])
    v = _input(ctx.n, seed).cuda()
    return {"case": case, "ctx": ctx, "in": v, "out": torch.zeros_like(v)}


def run(state):
    case, ctx, v, out = state["case"], state["ctx"], state["in"], state["out"]
    if case["call"] == "apply":
        ctx.fm_apply(case["E"], v, out)
        return out
    if case["call"] == "precond":
        ctx.fm_precond_apply(v, out)
        return out
    if case["call"] == "solve":
        out.zero_()
        ctx.fm_solve(case["E"], v, out)
        return out
    levels, _ = ctx.fm_eigs(case["E"], 1, v, out)
    return {"levels": np.array(levels), "vector": out}


# ---------------------------------------------------------------------------------------------------
# the least work of one pass
# ---------------------------------------------------------------------------------------------------
def _dims(c):
    q = 3 if c["basis"] else 2
    out = []
    for s in ("", "3"):
        nx, ny, nz = c["nx" + s], c["ny" + s], c["nz" + s]
        out.append((3 * nx + 1, 3 * ny + 1, 3 * nz + 3) if q == 3 else (2 * nx, 2 * ny, 2 * nz + 2))
    return out


def _unknowns(c):
    return (c["J"] + 1) * sum(x * y * z for x, y, z in _dims(c))


def work(case):
    """Float64 operations and bytes of one pass.  Per unknown: r taps per contracted index of each of the
    operator's distinct products; per active point and source of the rotated components, an r^3-tap evaluation
    for every M'; vectors and per-point tables read or written once.  Solves and eigen-solves: as many
    applications, preconditionings and orthogonalisations as the method takes at the given tolerances
    (about 30 iterations; 140 for the eigen-solve)."""
    r, nM, N = (6 if case["basis"] else 4), case["J"] + 1, _unknowns(case)
    act = 0
    for s, (nx, ny, nz) in zip(("", "3"), _dims(case)):
        u = np.linspace(0.0, 1.0, nx)
        x = 4.0 * ((1.0 + case["Rx" + s] / 4.0) ** u - 1.0)
        act += ny * nz * int((x ** NU < 46.5).sum())
    ap_f = N * (2.0 * r * (8 if nM == 1 else 10) + 6) + act * 2 * nM * (2.0 * (r ** 3 + r ** 2 + r) + 2 * nM)
    ap_b = 24.0 * N + act * 2 * (12.0 + 8.0 * (3 * r + nM * nM))
    pc_f = sum(2.0 * nM * x * y * z * (2 * z + 2 * x + 3 * (r // 2) * nM) for x, y, z in _dims(case))
    pc_b = 16.0 * N + sum(16.0 * (z + case["J"]) * x * x for x, y, z in _dims(case))
    if case["call"] == "apply":
        return {"bytes": ap_b, "flops": ap_f}
    if case["call"] == "precond":
        return {"bytes": pc_b, "flops": pc_f}
    its, mean_basis = (30, 15) if case["call"] == "solve" else (140, 6)
    return {"bytes": its * (ap_b + pc_b + 16.0 * N * mean_basis), "flops": its * (ap_f + pc_f + 8.0 * N * mean_basis)}


# ---------------------------------------------------------------------------------------------------
# 64-bit restatement in numpy and torch
# ---------------------------------------------------------------------------------------------------
def _poly_basis(basis):
    """Hermite shape polynomials on [0, 1], ascending coefficients, and the power of h each is scaled with."""
    if basis == 0:
        return [(1, 0, -3, 2), (0, 1, -2, 1), (0, 0, 3, -2), (0, 0, -1, 1)], (0, 1, 0, 1)
    return [(1, 0, 0, -10, 15, -6), (0, 1, 0, -6, 8, -3), (0, 0, .5, -1.5, 1.5, -.5),
            (0, 0, 0, 10, -15, 6), (0, 0, 0, -4, 7, -3), (0, 0, 0, .5, -1, .5)], (0, 1, 2, 0, 1, 2)


class _Axis:
    def __init__(self, basis, nint, R, radial):
        u = np.arange(nint + 1) / nint
        self.t = 4.0 * ((1.0 + R / 4.0) ** u - 1.0) if radial else np.sin(np.pi * (2.0 * u - 1.0) / 2.0)
        self.t[0], self.t[-1] = (0.0, R) if radial else (-1.0, 1.0)
        self.basis, self.q, self.nint, self.radial = basis, 3 if basis else 2, nint, radial
        self.r = 2 * self.q
        self.n = self.q * nint + (1 if basis else 0) if radial else self.q * (nint + 1)
        m = np.full(nint, self.q)
        if nint == 1:
            m[0] = self.n
        elif radial:
            m[0] += 1 if basis else 0
        else:
            m[0] += 1
            m[-1] += 1
            if basis:
                m[nint // 2] += 1
        pts = []
        for k in range(nint):
            g = np.polynomial.legendre.leggauss(int(m[k]))[0]
            pts.append(0.5 * (self.t[k] + self.t[k + 1]) + 0.5 * (self.t[k + 1] - self.t[k]) * g)
        self.pts = np.concatenate(pts)

    def column(self, full):
        """Function number of a (node, derivative) pair; -1 for the dropped value functions at the ends."""
        if not self.radial:
            return full
        last = self.q * self.nint
        return np.where((full == 0) | (full == last), -1, full - 1 - (full > last))

    def taps(self, p, deriv=0):
        """Columns and values of the r functions that are not zero at the points p (zero outside the box)."""
        p = np.asarray(p)
        m = np.clip(np.searchsorted(self.t, p, side="right") - 1, 0, self.nint - 1)
        h = self.t[m + 1] - self.t[m]
        s = (p - self.t[m]) / h
        shapes, powers = _poly_basis(self.basis)
        cols = self.column(self.q * m[:, None] + np.arange(self.r)[None, :])
        vals = np.stack([np.polynomial.polynomial.polyval(s, np.polynomial.polynomial.polyder(np.array(c, float), deriv))
                         * h ** (e - deriv) for c, e in zip(shapes, powers)], axis=1)
        out = (p < self.t[0]) | (p > self.t[-1])
        return cols, np.where((cols < 0) | out[:, None], 0.0, vals)

    def matrix(self, deriv):
        cols, vals = self.taps(self.pts, deriv)
        M = np.zeros((self.n, self.n))
        for k in range(self.r):
            ok = cols[:, k] >= 0
            M[np.nonzero(ok)[0], cols[ok, k]] += vals[ok, k]
        return M


def _wigner(J, M, Mp, w, k=0):
    """d^J_{M Mp}(w) / sin(w)^k by Wigner's sum."""
    f = math.factorial
    c, s = np.cos(w / 2), np.sin(w / 2)
    tot = np.zeros_like(w)
    if abs(M) > J or abs(Mp) > J:
        return tot
    pref = math.sqrt(f(J + M) * f(J - M) * f(J + Mp) * f(J - Mp))
    for i in range(2 * J + 1):
        a = (J + Mp - i, i, M - Mp + i, J - M - i)
        if min(a) >= 0:
            tot += ((-1.0) ** (M - Mp + i) * pref / (f(a[0]) * f(a[1]) * f(a[2]) * f(a[3]))
                    * c ** (2 * J + Mp - M - 2 * i - k) * s ** (M - Mp + 2 * i - k))
    return tot / 2.0 ** k


def _lam(J, M):
    return math.sqrt(max(J * (J + 1) - M * (M + 1), 0))


class _Problem:
    """(H - E S) of two solved components (1 and 3; the second electron's component by exchange symmetry)."""

    def __init__(self, case, dev):
        self.c, self.dev, self.J, self.nM = case, dev, case["J"], case["J"] + 1
        self.m, self.Z = np.array(MASS[case["system"]]), np.array(CHARGE[case["system"]])
        self.ax = {a: (_Axis(case["basis"], case["nz" + s], 1.0, False),
                       _Axis(case["basis"], case["nx" + s], case["Rx" + s], True),
                       _Axis(case["basis"], case["ny" + s], case["Ry" + s], True)) for a, s in ((1, ""), (3, "3"))}
        self.shape = {a: (self.nM, z.n, x.n, y.n) for a, (z, x, y) in self.ax.items()}
        self.mats = {a: [[self.dv(ax.matrix(d)) for d in range(3)] for ax in self.ax[a]] for a in self.ax}
        self.local, self.gather = {}, {}
        for a in (1, 3):
            self._local_tables(a)
            self._coupling_tables(a)

    def dv(self, v):
        return torch.as_tensor(np.ascontiguousarray(v)).to(self.dev)

    def coulomb(self, a, x):
        b, c = [i for i in range(3) if i != a - 1]
        mu = self.m[b] * self.m[c] / (self.m[b] + self.m[c])
        return math.sqrt(2 * mu) * self.Z[b] * self.Z[c] / x

    def chi(self, x):
        with np.errstate(over="ignore"):
            return 2.0 / (1.0 + np.exp((x / X0) ** NU))

    def rotate(self, b, a, x, y, z):
        M, mb, ma = self.m.sum(), self.m[b - 1], self.m[a - 1]
        c = -math.sqrt(mb * ma / ((M - mb) * (M - ma)))
        s = (-1.0) ** (b - a) * np.sign(a - b) * math.sqrt(1.0 - c * c)
        xb = np.sqrt(np.maximum(c * c * x * x + 2 * s * c * x * y * z + s * s * y * y, 0.0))
        yb = np.sqrt(np.maximum(s * s * x * x - 2 * s * c * x * y * z + c * c * y * y, 0.0))
        zb = (s * c * (y * y - x * x) + (c * c - s * s) * x * y * z) / (xb * yb)
        return c, s, xb, yb, np.clip(zb, -1.0, 1.0)

    def _local_tables(self, a):
        z, x, y = (ax.pts for ax in self.ax[a])
        Z, X, Y = z[:, None, None], x[None, :, None], y[None, None, :]
        V = self.coulomb(a, X) + np.zeros((len(z), len(x), len(y)))
        for b in (1, 2, 3):
            if b != a:
                _, _, xb, _, _ = self.rotate(b, a, X, Y, Z)
                V += (1.0 - self.chi(xb)) * self.coulomb(b, xb)
        self.local[a] = [self.dv(v) for v in (V, z, x, y)]

    def _coupling_tables(self, a):
        zp, xp, yp = (ax.pts for ax in self.ax[a])
        near = np.nonzero(self.chi(xp) > VS_CUT)[0]
        k, i, j = (v.reshape(-1) for v in np.meshgrid(np.arange(len(zp)), near, np.arange(len(yp)), indexing="ij"))
        z, x, y = zp[k], xp[i], yp[j]
        pt = (k * len(xp) + i) * len(yp) + j
        vs = self.chi(x) * self.coulomb(a, x)
        found = []
        for b in (1, 2, 3):
            if b == a:
                continue
            src, sign = (b, 1.0) if b != 2 else (1, -1.0)
            c, s, xb, yb, zb = self.rotate(b, a, x, y, z)
            w = np.arccos(np.clip((-s * x * z + c * y) / yb, -1.0, 1.0))
            cyc = (b, a) in ((1, 2), (2, 3), (3, 1))
            w = w if cyc else 2 * np.pi - w
            rho, sin_t = x * y / (xb * yb), np.sqrt(np.clip(1 - z * z, 0, None))
            wt = np.empty((self.nM, self.nM, len(pt)))
            for Mp in range(self.nM):
                for Mq in range(self.nM):
                    kk = max(0, Mp - Mq)
                    F = (_wigner(self.J, Mq, Mp, w, kk) + (-1.0) ** Mp * _wigner(self.J, Mq, -Mp, w, kk)) / math.sqrt(2.0 + 2.0 * (Mp == 0))
                    ang = (-1.0) ** (Mq - Mp) * 2.0 / math.sqrt(2.0 + 2.0 * (Mq == 0)) * F
                    if kk:
                        ang = ang * ((1.0 if cyc else -1.0) * abs(s) * x / yb) ** kk
                    else:
                        ang = ang * sin_t ** (Mq - Mp)
                    wt[Mp, Mq] = vs * rho ** (Mq + 1) * ang * ((-1.0) ** Mq if sign < 0 else 1.0)
            taps = [self.ax[src][d].taps(v) for d, v in enumerate((sign * zb, xb, yb))]
            found.append((src, self.dv(wt), [(self.dv(np.maximum(t, 0)), self.dv(v)) for t, v in taps]))
        self.gather[a] = (self.dv(pt), found)

    def split(self, v):
        n1 = math.prod(self.shape[1])
        return {1: v[:n1].reshape(self.shape[1]), 3: v[n1:].reshape(self.shape[3])}

    def S(self, v):
        parts = self.split(v)
        return torch.cat([(torch.einsum("lk,mkij->mlij", self.mats[a][0][0], self.mats[a][1][0] @ (p @ self.mats[a][2][0].T))).reshape(-1)
                          for a, p in parts.items()])

    def apply(self, E, v):
        parts, out, J = self.split(v), [], self.J
        for a, p in parts.items():
            (Sz, D1, D2), (Sx, _, Dx), (Sy, _, Dy) = self.mats[a]
            V, z, x, y = self.local[a]
            iy2 = 1.0 / (y * y)
            q = (1.0 / (x * x))[:, None] + iy2[None, :]
            py, pd = p @ Sy.T, p @ Dy.T
            P, Q = Sx @ py, Dx @ py + Sx @ pd
            del py, pd
            over = lambda A, T: torch.einsum("lk,kij->lij", A, T)  # noqa: E731
            Z = z[:, None, None]
            o = torch.empty_like(p)
            for M in range(self.nM):
                U, Uz = over(Sz, P[M]), over(D1, P[M])
                o[M] = (V + M * (M + 1) * q + (J * (J + 1) - 2 * M * M) * iy2 - E) * U - over(Sz, Q[M])
                o[M] += q * (2 * (M + 1) * Z * Uz - (1 - Z * Z) * over(D2, P[M]))
                if M + 1 < self.nM:
                    f = _lam(J, M) * math.sqrt(1.0 + (M == 0))
                    o[M] += f * iy2 * (2 * (M + 1) * Z * over(Sz, P[M + 1]) - (1 - Z * Z) * over(D1, P[M + 1]))
                if M >= 1:
                    o[M] += _lam(J, -M) * math.sqrt(1.0 + (M == 1)) * iy2 * over(D1, P[M - 1])
            pt, found = self.gather[a]
            flat = o.reshape(self.nM, -1)
            for src, wt, ((tz, vz), (tx, vx), (ty, vy)) in found:
                _, _, snx, sny = self.shape[src]
                f = parts[src].reshape(self.nM, -1)
                val = torch.zeros((self.nM, len(pt)), dtype=torch.float64, device=self.dev)
                for kz in range(tz.shape[1]):
                    for kx in range(tx.shape[1]):
                        at, wgt = (tz[:, kz] * snx + tx[:, kx]) * sny, vz[:, kz] * vx[:, kx]
                        for ky in range(ty.shape[1]):
                            val += (wgt * vy[:, ky]) * f[:, at + ty[:, ky]]
                flat[:, pt] += torch.einsum("mnp,np->mp", wt, val)
            out.append(o.reshape(-1))
        return torch.cat(out)


def _eig(A):
    lam, W = np.linalg.eig(A)
    order = np.argsort(lam.real, kind="stable")
    return lam[order], W[:, order]


def _real_basis(lam, W):
    """Real and imaginary parts of complex-conjugate pairs as columns."""
    for i in range(len(lam)):
        if lam[i].imag > 0:
            W[:, i + 1] = W[:, i].imag
            W[:, i] = W[:, i].real
    return W.real


class _Precond:
    """P^{-1}: z modes with eigenvalues -l(l+1), x pencils per l, then the y systems of every (l, x mode),
    the M' components of one l coupled."""

    def __init__(self, prob, E, strict):
        self.p, J, nM = prob, prob.J, prob.nM
        self.comp = {}
        for a, (az, ax, ay) in prob.ax.items():
            z, x, y = az.pts, ax.pts, ay.pts
            Sz, D1, D2 = (az.matrix(d) for d in range(3))
            Sx, Dx, Sy, Dy = ax.matrix(0), ax.matrix(2), ay.matrix(0), ay.matrix(2)
            Wz = []
            for M in range(nM):
                Dz = (1 - z * z)[:, None] * D2 - (2 * (M + 1) * z)[:, None] * D1 - M * (M + 1) * Sz
                lam, W = _eig(np.linalg.solve(Sz, -Dz))
                if strict and np.min(np.diff(lam.real) / np.abs(lam.real[1:])) < 1e-7:
                    raise ValueError("z modes degenerate to rounding")
                if np.iscomplexobj(lam) and np.abs(lam.imag).max() > 1e-10 * np.abs(lam).max():
                    if strict:
                        raise ValueError("complex z modes")
                    W = _real_basis(lam, W)
                W = W.real
                f1 = W[az.q * az.nint]  # value at z = 1
                l = M + np.arange(az.n)
                lf = np.array([math.lgamma(v + M + 1) - math.lgamma(v - M + 1) for v in l])
                g1 = np.sqrt((2 * l + 1) / 2.0) * np.exp(0.5 * lf) * (-1.0) ** M / (2.0 ** M * math.factorial(M))
                Wz.append(W * np.where(np.abs(f1) > 1e-12 * np.abs(W).max(0), g1 / np.where(f1 == 0, 1, f1), 1.0))
            Wzb = [np.linalg.inv(Sz @ W) for W in Wz]
            Va = prob.coulomb(a, x)
            iS = np.linalg.inv(Sx)

            def xmode(l):
                lam, W = _eig(iS @ (-Dx + (l * (l + 1.0) / x ** 2 + Va)[:, None] * Sx))
                cx = np.iscomplexobj(lam) and np.abs(lam.imag).max() > 1e-10 * np.abs(lam).max()
                W = _real_basis(lam, W) if cx else W.real
                return lam.real, W, np.linalg.inv(Sx @ W), cx
            with ThreadPoolExecutor(16) as ex:
                xm = list(ex.map(xmode, range(J + az.n)))
            if strict and any(v[3] for v in xm):
                raise ValueError("complex x modes")
            b, c = [i for i in range(3) if i != a - 1]
            m, M3 = prob.m, prob.m.sum()
            mu = m[a - 1] * (m[b] + m[c]) / M3
            Ry = prob.c["Ry" if a == 1 else "Ry3"]
            Vh = prob.Z[a - 1] * (prob.Z[b] + prob.Z[c]) * math.sqrt(2 * mu) / y * (1.0 - np.exp(-(y / (0.05 * Ry)) ** 2))
            B, A2 = -Dy + (Vh - E)[:, None] * Sy, (1.0 / y ** 2)[:, None] * Sy
            inv = []
            for l in range(J + az.n):
                ch = [M for M in range(nM) if M <= l < M + az.n]
                n = len(ch) * len(y)
                K = np.zeros((len(ch), len(y), len(ch), len(y)))
                G = np.zeros_like(K)
                for r, M in enumerate(ch):
                    K[r, :, r] = B + (J * (J + 1) - 2 * M * M + l * (l + 1)) * A2
                    G[r, :, r] = Sy
                    if r + 1 < len(ch):
                        K[r, :, r + 1] = -_lam(J, M) * math.sqrt(1.0 + (M == 0)) * _lam(l, M) * A2
                    if r:
                        K[r, :, r - 1] = -_lam(J, -M) * math.sqrt(1.0 + (M == 1)) * _lam(l, -M) * A2
                mat = prob.dv(K.reshape(n, n))[None] + prob.dv(xm[l][0])[:, None, None] * prob.dv(G.reshape(n, n))[None]
                inv.append((ch, torch.linalg.lu_factor(mat)))
            self.comp[a] = ([prob.dv(w) for w in Wz], [prob.dv(w) for w in Wzb], [prob.dv(v[1]) for v in xm],
                            [prob.dv(v[2]) for v in xm], inv)

    @staticmethod
    def bytes_of(case):
        tot = 0
        for x, y, z in _dims(case):
            tot += 8.0 * (z + case["J"]) * x * ((case["J"] + 1) * y) ** 2
        return tot

    def __call__(self, v):
        out = []
        for a, t in self.p.split(v).items():
            Wz, Wzb, Wx, Wxb, inv = self.comp[a]
            t = torch.stack([torch.einsum("lk,kij->lij", Wzb[M], t[M]) for M in range(self.p.nM)])
            u = torch.empty_like(t)
            for l, (ch, lu) in enumerate(inv):
                rhs = torch.stack([Wxb[l] @ t[M, l - M] for M in ch], 1)  # [x mode][M'][y]
                sol = torch.linalg.lu_solve(*lu, rhs.reshape(len(rhs), -1, 1)).reshape(rhs.shape)
                for r, M in enumerate(ch):
                    u[M, l - M] = Wx[l] @ sol[:, r]
            out.append(torch.stack([torch.einsum("kl,lij->kij", Wz[M], u[M]) for M in range(self.p.nM)]).reshape(-1))
        return torch.cat(out)


def _gmres(A, P, b, tol, cycles=4, m=90):
    x, bn = torch.zeros_like(b), torch.linalg.norm(b)
    r = b.clone()
    for _ in range(cycles):
        beta = torch.linalg.norm(r)
        if beta <= tol * bn:
            break
        V, Zs, H = [r / beta], [], np.zeros((m + 1, m))
        for j in range(m):
            Zs.append(P(V[j]))
            w = A(Zs[j])
            Vm = torch.stack(V)
            for _twice in range(2):
                h = Vm @ w
                w = w - h @ Vm
                H[:j + 1, j] += h.cpu().numpy()
            H[j + 1, j] = torch.linalg.norm(w).item()
            V.append(w / H[j + 1, j])
            e = np.zeros(j + 2)
            e[0] = beta.item()
            s, _, _, _ = np.linalg.lstsq(H[:j + 2, :j + 1], e, rcond=None)
            if np.linalg.norm(e - H[:j + 2, :j + 1] @ s) <= 0.3 * tol * bn.item():
                break
        for c, zv in zip(s, Zs):
            x = x + float(c) * zv
        r = b - A(x)
    return x


def exact(case, seed):
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["call"] == "eigs" or case["call"] != "apply" and (_Precond.bytes_of(case) > 24e9 or _unknowns(case) > 3.4e6):
        return None  # over the time: nested solves, or the 1D decompositions of the large grids
    prob = _Problem(case, dev)
    v = _input(_unknowns(case), seed).to(dev)
    if case["call"] == "apply":
        return prob.apply(case["E"], v)
    try:
        P = _Precond(prob, case["E"], strict=case["call"] == "precond")
    except ValueError:
        return None  # complex or degenerate 1D modes: the preconditioner then depends on the basis chosen for them
    if case["call"] == "precond":
        return P(v)
    return _gmres(lambda u: prob.apply(case["E"], u), P, v, 1e-13)
