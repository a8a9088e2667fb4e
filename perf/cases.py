"""The work a user of the library has it do, as measurable cases: block matvecs in each
precision and boundary condition, true residuals, batched stored matvecs, whole solves,
whole requests (discretise, right-hand sides, solve) and off-surface fields, through the
Python binding of the C ABI.

Shapes follow the library's own workloads (disk, star, kite, ellipse, random stars) and the
served range (random stars, 1..64 directions, 8 to 16 nodes per wavelength).  The reference
values (`exact`) are plain torch in 64 bits: Kress's rule, dense sums, LU.
"""
import math
import random

import torch

from paper_1408_1578_gb300 import cfie

DEV = "cuda"
EULER = 0.57721566490153286061


# ---------------------------------------------------------------------------
# cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the plain FP64 matvec of one incident wave on a small obstacle: latency and launches
        {"name": "disk-fp64", "kind": "apply", "precision": "fp64", "bc": "soft",
         "curve": "circle", "shape": 0, "n": 1024, "omega": 64.0, "nrhs": 1},
        # the plain FP64 sound-hard matvec, 16 directions
        {"name": "star-fp64-hard", "kind": "apply", "precision": "fp64", "bc": "hard",
         "curve": "star5", "shape": 0, "n": 4096, "omega": 256.0, "nrhs": 16},
        # the inner block matvec of the headline solve: 64 directions on a large kite
        {"name": "kite-fp32", "kind": "apply", "precision": "fp32", "bc": "soft",
         "curve": "kite", "shape": 0, "n": 32768, "omega": 2048.0, "nrhs": 64},
        # the inner block matvec of a mid-size sound-hard solve
        {"name": "star-fp32-hard", "kind": "apply", "precision": "fp32", "bc": "hard",
         "curve": "star5", "shape": 0, "n": 4096, "omega": 256.0, "nrhs": 16},
        # one direction on the large ellipse, sound hard, 8 nodes per wavelength
        {"name": "ellipse-fp32-hard", "kind": "apply", "precision": "fp32", "bc": "hard",
         "curve": "ellipse", "shape": 0, "n": 32768, "omega": 5313.0, "nrhs": 1},
        # one lockstep matvec of a batch of stored operators, 32 directions each
        {"name": "stars-stored", "kind": "batch", "precision": "tensor", "bc": "soft",
         "curve": "stars", "shape": 1408, "n": 16384, "count": 32, "nrhs": 32},
        # the true residual of the headline solve (once per refinement step)
        {"name": "kite-residual", "kind": "residual", "precision": "fp32", "bc": "soft",
         "curve": "kite", "shape": 0, "n": 32768, "omega": 2048.0, "nrhs": 64},
        # the true residual of a sound-hard solve
        {"name": "star-residual-hard", "kind": "residual", "precision": "fp32", "bc": "hard",
         "curve": "star5", "shape": 0, "n": 4096, "omega": 256.0, "nrhs": 16},
        # a whole unrestarted FP64 solve of a small problem, one direction
        {"name": "disk-solve", "kind": "solve", "precision": "fp64", "bc": "soft",
         "curve": "circle", "shape": 0, "n": 1024, "omega": 64.0, "nrhs": 1},
        # a whole refined solve of 64 directions, operator kept
        {"name": "kite-solve", "kind": "solve", "precision": "fp32", "bc": "soft",
         "curve": "kite", "shape": 0, "n": 8192, "omega": 512.0, "nrhs": 64},
        # a whole request: a new sound-hard obstacle, discretised, solved and dropped; ragged sizes
        {"name": "star-request-hard", "kind": "request", "precision": "fp32", "bc": "hard",
         "curve": "star8", "shape": 1578, "n": 6002, "omega": 480.0, "nrhs": 33},
        # the scattered field of 16 densities at 20000 points after a solve
        {"name": "star-field", "kind": "field", "precision": "fp64", "bc": "hard",
         "curve": "star5", "shape": 0, "n": 4096, "omega": 256.0, "nrhs": 16, "npts": 20000},
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


# largest n drawn per kind (and precision): what one pass of the listed cases costs at most
_NMAX = {"apply": 32768, "residual": 16384, "solve": 4096, "request": 6144, "field": 8192}


def draw(rng):
    kind = rng.choice(["apply", "apply", "apply", "residual", "residual", "solve", "request",
                       "field", "batch"])
    if kind == "batch":
        return {"kind": kind, "precision": "tensor", "bc": "soft", "curve": "stars",
                "shape": rng.randrange(1 << 20), "n": 2 * int(_log(rng, 1024, 16384) / 2),
                "count": rng.randint(2, 24), "nrhs": rng.randint(1, 64)}
    prec = rng.choice(["fp64", "fp32", "fp32"]) if kind in ("apply", "solve", "field") else "fp32"
    nmax = _NMAX[kind] if prec == "fp32" else min(_NMAX[kind], 2048 if kind == "solve" else 6144)
    curve = rng.choice(["circle", "ellipse", "star5", "star8", "star8", "kite"])
    shape = rng.randrange(1 << 20)
    n = 2 * int(_log(rng, 512, nmax) / 2)
    c = {"kind": kind, "precision": prec, "bc": rng.choice(["soft", "hard"]), "curve": curve,
         "shape": shape, "n": n, "nrhs": int(_log(rng, 1, 64.99))}
    c["omega"] = round(2 * math.pi * n / (rng.uniform(8.0, 16.0) * _perimeter(curve, shape)), 3)
    if kind == "field":
        c["npts"] = int(_log(rng, 64, 20000))
    return c


# ---------------------------------------------------------------------------
# curves: parameters and samples
# ---------------------------------------------------------------------------
def _star8(shape):
    r = random.Random(int(shape))
    return ([r.uniform(-0.05, 0.05) for _ in range(8)], [r.uniform(-0.05, 0.05) for _ in range(8)])


def _params(curve, shape):
    if curve == "circle":
        return "circle", {}
    if curve == "ellipse":
        return "ellipse", {"a": 1.0, "b": 0.5}
    if curve == "kite":
        return "kite", {}
    if curve == "star5":
        return "star", {"a": [0, 0, 0, 0, 0.3], "b": [0, 0, 0, 0, 0]}
    a, b = _star8(shape)
    return "star", {"a": a, "b": b}


def _curve(curve, shape, n):
    """z, z', z'' (n x 2, FP64) at t_j = 2 pi j / n."""
    t = 2 * math.pi * torch.arange(n, dtype=torch.float64) / n
    kind, p = _params(curve, shape)
    co, si = torch.cos(t), torch.sin(t)
    if kind == "circle":
        q = ((co, si), (-si, co), (-co, -si))
    elif kind == "ellipse":
        a, b = p["a"], p["b"]
        q = ((a * co, b * si), (-a * si, b * co), (-a * co, -b * si))
    elif kind == "kite":
        q = ((co + 0.65 * torch.cos(2 * t) - 0.65, 1.5 * si),
             (-si - 1.3 * torch.sin(2 * t), 1.5 * co),
             (-co - 2.6 * torch.cos(2 * t), -1.5 * si))
    else:
        r, r1, r2 = torch.ones_like(t), torch.zeros_like(t), torch.zeros_like(t)
        for k, (a, b) in enumerate(zip(p["a"], p["b"]), 1):
            ck, sk = torch.cos(k * t), torch.sin(k * t)
            r += a * ck + b * sk
            r1 += k * (b * ck - a * sk)
            r2 -= k * k * (a * ck + b * sk)
        q = ((r * co, r * si), (r1 * co - r * si, r1 * si + r * co),
             (r2 * co - 2 * r1 * si - r * co, r2 * si + 2 * r1 * co - r * si))
    return [torch.stack(v, 1) for v in q]


def _perimeter(curve, shape):
    return float(_curve(curve, shape, 2048)[1].norm(dim=1).sum()) * 2 * math.pi / 2048


def _stars(case):
    """(shape, n, omega) of a batch's operators: random stars, n log-uniform up to case["n"],
    10 nodes per wavelength."""
    r = random.Random(int(case["shape"]))
    out = []
    for _ in range(case["count"]):
        s = r.randrange(1 << 20)
        n = 2 * int(_log(r, max(512, case["n"] // 32), case["n"]) / 2)
        out.append((s, n, 2 * math.pi * n / (10.0 * _perimeter("star8", s))))
    return out


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cpu")
    g.manual_seed(int(seed) % (1 << 62))
    return g


def _density(z, omega, nrhs, g):
    """Densities as a solve meets them (incident data, Krylov vectors): each column a random
    superposition of 24 plane waves on the curve, unit rms."""
    th = 2 * math.pi * torch.rand(nrhs, 24, generator=g, dtype=torch.float64)
    c = torch.randn(nrhs, 24, generator=g, dtype=torch.complex128).to(DEV)
    th, z = th.to(DEV), z.to(DEV)
    x = torch.zeros(nrhs, z.shape[0], dtype=torch.complex128, device=DEV)
    for m in range(24):
        ph = omega * (torch.outer(torch.cos(th[:, m]), z[:, 0]) +
                      torch.outer(torch.sin(th[:, m]), z[:, 1]))
        x += c[:, m, None] * torch.polar(torch.ones_like(ph), ph)
    return (x / math.sqrt(24.0)).contiguous()


def _angles(case, g):
    """Evenly spaced incidence angles from a random first one."""
    k = case["nrhs"]
    first = float(torch.rand(1, generator=g, dtype=torch.float64))
    return [2 * math.pi * (m + first) / k for m in range(k)]


def _points(z, npts, g):
    """Field points on random rays, 0.3 to 3 beyond a circle around the obstacle."""
    th = 2 * math.pi * torch.rand(npts, generator=g, dtype=torch.float64)
    r = float(z.norm(dim=1).max()) + 0.3 + 2.7 * torch.rand(npts, generator=g, dtype=torch.float64)
    return torch.polar(r, th).to(DEV).contiguous()


def _rtol(case):
    # refined solves two digits beyond the 1e-8 of the served requests, so that what is
    # returned is the solution and not the stopping rule's remainder
    return 1e-10


def prepare(case, seed):
    g = _gen(seed)
    ctx = cfie.Context(0, stream=torch.cuda.current_stream())
    s = {"case": case, "ctx": ctx}
    if case["kind"] == "batch":
        ops, xs = [], []
        for sh, n, om in _stars(case):
            op = ctx.geometry("star", **_params("star8", sh)[1]).discretise(
                n, om, bc="soft", precision="tensor", layout="stored")
            ops.append(op)
            xs.append(_density(_curve("star8", sh, n)[0], om, case["nrhs"], g).reshape(-1))
        s["ops"] = ops
        s["batch"] = cfie.Batch(ctx, ops, [case["nrhs"]] * len(ops))
        s["x"] = torch.cat(xs)
        s["y"] = torch.empty_like(s["x"])
        return s
    n, nrhs = case["n"], case["nrhs"]
    kind, par = _params(case["curve"], case["shape"])
    z = _curve(case["curve"], case["shape"], n)[0]
    if case["kind"] == "request":
        s["theta"] = _angles(case, g)
        s["geometry"] = (kind, par)
        return s
    op = ctx.geometry(kind, **par).discretise(n, case["omega"], bc=case["bc"],
                                              precision=case["precision"])
    s["op"] = op
    if case["kind"] == "solve":
        s["f"] = torch.empty(nrhs, n, dtype=torch.complex128, device=DEV)
        op.rhs_plane_waves(_angles(case, g), s["f"])
        s["q"] = torch.empty_like(s["f"])
    else:
        s["x"] = _density(z, case["omega"], nrhs, g)
        if case["kind"] == "field":
            s["pts"] = _points(z, case["npts"], g)
            s["u"] = torch.empty(nrhs, case["npts"], dtype=torch.complex128, device=DEV)
        else:
            s["y"] = torch.empty_like(s["x"])
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "apply":
        s["op"].apply(s["x"], s["y"])
        # the FP32 matvec's caller (an FP32 Krylov basis) keeps complex64
        return s["y"] if case["precision"] == "fp64" else s["y"].to(torch.complex64)
    if kind == "residual":
        s["op"].apply_residual(s["x"], s["y"])
        return s["y"]
    if kind == "batch":
        s["batch"].apply(s["x"], s["y"])
        return s["y"].to(torch.complex64)
    if kind == "field":
        s["op"].field_eval(s["x"], s["pts"], s["u"])
        return s["u"]
    if kind == "solve":
        s["q"].zero_()
        s["op"].gmres_solve(s["f"], s["q"], rtol=_rtol(case), restart=80, maxit=2000)
        return s["q"]
    g = s["ctx"].geometry(s["geometry"][0], **s["geometry"][1])
    op = g.discretise(case["n"], case["omega"], bc=case["bc"], precision=case["precision"])
    f = torch.empty(case["nrhs"], case["n"], dtype=torch.complex128, device=DEV)
    op.rhs_plane_waves(s["theta"], f)
    q = torch.zeros_like(f)
    op.gmres_solve(f, q, rtol=_rtol(case), restart=80, maxit=2000)
    op.close()
    g.close()
    return q


# ---------------------------------------------------------------------------
# work of one pass
# ---------------------------------------------------------------------------
def work(case):
    if case["kind"] == "batch":
        shapes = _stars(case)
        entries = sum(n * n for _, n, _ in shapes)
        vec = sum(n for _, n, _ in shapes) * case["nrhs"]
        return {"bytes": 8.0 * entries + 32.0 * vec, "flops": 8.0 * entries * case["nrhs"]}
    n, r = case["n"], case["nrhs"]
    vec = 16.0 * n * r
    if case["kind"] == "field":
        # one kernel value per (point, node) and a complex multiply-add per density
        return {"bytes": vec + 48.0 * n + 16.0 * case["npts"] * (r + 1),
                "flops": 1.0 * n * case["npts"] * (60 + 8 * r)}
    # one entry evaluation per pair (about 60 operations) and one complex multiply-add per
    # right-hand side and sum: one sum (soft), or S u and the rest (hard)
    sums = 1 if case["bc"] == "soft" else 2
    mv = {"bytes": 2 * vec + 48.0 * n, "flops": 1.0 * n * n * (60 + 8 * r * sums)}
    if case["kind"] in ("apply", "residual"):
        return mv
    # GMRES to 1e-10: the steps grow about like n^0.3 (soft, eta = omega); two products with the
    # basis per step
    its = 27.0 * (n / 512.0) ** 0.305
    return {"bytes": its * mv["bytes"] + its * its * vec, "flops": its * mv["flops"]}


# ---------------------------------------------------------------------------
# the same in 64 bits, plain torch
# ---------------------------------------------------------------------------
def _bessel(a):
    """J0, Y0, J1, Y1 of a > 0 in 64 bits: Hankel's asymptotic expansion for a >= 25, Miller's
    backward recurrence with Neumann's series below (torch.special's lose digits around a = 5)."""
    t = 1.0 / a
    t2 = t * t
    amp = torch.sqrt(2 / math.pi * t)
    chi = a - math.pi / 4
    co, si = torch.cos(chi) * amp, torch.sin(chi) * amp
    out = []
    for nu in (0, 1):
        c = [1.0]
        for k in range(1, 24):
            c.append(c[-1] * (4 * nu * nu - (2 * k - 1) ** 2) / (8 * k))
        P = torch.full_like(a, c[22] * (-1) ** 11)
        Q = torch.full_like(a, c[23] * (-1) ** 11)
        for k in range(10, -1, -1):
            P = P * t2 + c[2 * k] * (-1) ** k
            Q = Q * t2 + c[2 * k + 1] * (-1) ** k
        Q = Q * t
        out += [P * co - Q * si, P * si + Q * co] if nu == 0 else [P * si + Q * co, Q * si - P * co]
    near = (a < 25.0).nonzero(as_tuple=True)
    x = a[near]
    if x.numel():
        up, cur = torch.zeros_like(x), torch.full_like(x, 1e-280)
        even, y0, y1 = torch.zeros_like(x), torch.zeros_like(x), torch.zeros_like(x)
        for k in range(72, 0, -1):
            # cur = J_k, up = J_(k+1), unnormalised
            m = k // 2
            if k % 2 == 0:
                even = even + cur
                y0 = y0 + (-1) ** m / m * cur
                # (-1)^m (J_(2m-1) - J_(2m+1)) / m, J_(2m-1) = (4 m / x) J_2m - J_(2m+1)
                y1 = y1 + (-1) ** m / m * (2 * k / x * cur - 2 * up)
            if k == 1:
                one = cur
            up, cur = cur, 2 * k / x * cur - up
            s = torch.where(cur.abs() > 1e150, 1e-150, 1.0)
            up, cur, even, y0, y1 = up * s, cur * s, even * s, y0 * s, y1 * s
            if k == 1:
                one = one * s
        nrm = 1.0 / (cur + 2 * even)
        j0, j1 = cur * nrm, one * nrm
        lg = torch.log(x / 2) + EULER
        v = (j0, 2 / math.pi * (lg * j0 - 2 * y0 * nrm), j1,
             2 / math.pi * (lg * j1 - j0 / x + y1 * nrm))
        for o, q in zip(out, v):
            o[near] = q
    return out


class _Curve:
    def __init__(self, curve, shape, n, omega):
        z, d, dd = [v.to(DEV) for v in _curve(curve, shape, n)]
        self.n, self.w, self.h = n, omega, 2 * math.pi / n
        self.x, self.y = z[:, 0].contiguous(), z[:, 1].contiguous()
        self.s = d.norm(dim=1)
        self.n1, self.n2 = d[:, 1].contiguous(), -d[:, 0]
        self.l2 = (d[:, 1] * dd[:, 0] - d[:, 0] * dd[:, 1]) / (4 * math.pi * self.s ** 2)
        # Kress weights R_d = -(2 pi / N) sum_{m<N} cos(m t_d) / m - (pi / N^2) cos(N t_d), n = 2 N
        N = n // 2
        c = torch.zeros(n, dtype=torch.float64, device=DEV)
        m = torch.arange(1, N, device=DEV)
        c[1:N] = 1.0 / m.double()
        c[N] = 1.0 / n
        R = -(2 * math.pi / N) * torch.fft.fft(c).real
        td = math.pi * torch.arange(n, dtype=torch.float64, device=DEV) / n
        self.wd = R.clone()
        self.wd[1:] -= self.h * torch.log(4 * torch.sin(td[1:]) ** 2)
        self.R0 = R[0]

    def rows(self, i0, i1, what):
        """Rows i0..i1 of the soft matrix ("soft") or of S and D' ("hard"); eta = omega."""
        i = torch.arange(i0, i1, device=DEV)
        j = torch.arange(self.n, device=DEV)
        dx = self.x[i, None] - self.x[None, :]
        dy = self.y[i, None] - self.y[None, :]
        r = torch.sqrt(dx * dx + dy * dy)
        diag = (torch.arange(i1 - i0, device=DEV), i)
        r[diag] = 1.0
        a = self.w * r
        J0, Y0, J1, Y1 = _bessel(a)
        w = self.wd[(i[:, None] - j[None, :]) % self.n]
        h, s, om = self.h, self.s, self.w
        q = 1 / (4 * math.pi)
        m2 = 0.25j - EULER / (2 * math.pi) - torch.log(om * s[i] / 2) / (2 * math.pi)
        Sd = (-self.R0 * q + h * m2) * s[i]
        if what == "soft":
            c = om * (dx * self.n1 + dy * self.n2) / r
            es = om * s[None, :]
            A = torch.complex(h / 4 * (es * J0 - c * Y1) - w * q * c * J1,
                              h / 4 * (c * J1 + es * Y0) + w * q * es * J0)
            A[diag] = 0.5 + h * self.l2[i] - 1j * om * Sd
            return A
        S = torch.complex((-h / 4 * Y0 - w * q * J0) * s, h / 4 * J0 * s)
        S[diag] = Sd
        c = -om * (dx * self.n1[i, None] + dy * self.n2[i, None]) / r * s / s[i, None]
        D = torch.complex(-h / 4 * c * Y1 - w * q * c * J1, h / 4 * c * J1)
        D[diag] = (h * self.l2[i]).to(D.dtype)
        return S, D

    def dt(self, v):
        """(1/|z'|) d/dt along the last axis, spectral, Nyquist mode zero."""
        k = torch.fft.fftfreq(self.n, 1.0 / self.n, dtype=torch.float64, device=DEV)
        k[self.n // 2] = 0
        return torch.fft.ifft(1j * k * torch.fft.fft(v)) / self.s

    def _blocks(self):
        step = max(1, min(self.n, (1 << 25) // self.n))
        for i0 in range(0, self.n, step):
            yield i0, min(self.n, i0 + step)

    def apply(self, bc, x):
        """A x for the rows of x."""
        xt = x.T.contiguous()
        if bc == "soft":
            return torch.cat([self.rows(a, b, bc) @ xt for a, b in self._blocks()]).T
        k, om = x.shape[0], self.w
        n1, n2 = self.n1 / self.s, self.n2 / self.s
        v = torch.cat([self.dt(x), n1 * x, n2 * x]).T.contiguous()
        S, D = [], []
        for a, b in self._blocks():
            p, q = self.rows(a, b, bc)
            S.append(p @ v)
            D.append(q @ xt)
        S, D = torch.cat(S).T, torch.cat(D).T
        return 0.5 * x - D + (self.dt(S[:k]) + om ** 2 * (n1 * S[k:2 * k] + n2 * S[2 * k:])) / (1j * om)

    def matrix(self, bc):
        if bc == "soft":
            return torch.cat([self.rows(a, b, bc) for a, b in self._blocks()])
        p = [self.rows(a, b, bc) for a, b in self._blocks()]
        S, D = torch.cat([v[0] for v in p]), torch.cat([v[1] for v in p])
        n1, n2 = self.n1 / self.s, self.n2 / self.s
        om = self.w
        # S (1/s) Dt as a matrix: rows times the derivative, whose transpose is -Dt
        k = torch.fft.fftfreq(self.n, 1.0 / self.n, dtype=torch.float64, device=DEV)
        k[self.n // 2] = 0
        T = torch.fft.ifft(-1j * k * torch.fft.fft(S / self.s))
        T = self.dt(T.T.contiguous()).T
        A = (T + om ** 2 * (n1[:, None] * S * n1 + n2[:, None] * S * n2)) / (1j * om) - D
        A.diagonal().add_(0.5)
        return A

    def plane_waves(self, bc, theta):
        d = torch.tensor([[math.cos(t), math.sin(t)] for t in theta], dtype=torch.float64,
                         device=DEV)
        ph = self.w * (d[:, :1] * self.x + d[:, 1:] * self.y)
        u = torch.polar(torch.ones_like(ph), ph)
        if bc == "soft":
            return -u
        return -1j * self.w * (d[:, :1] * self.n1 + d[:, 1:] * self.n2) / self.s * u

    def field(self, bc, q, pts):
        out = []
        step = max(1, (1 << 25) // self.n)
        for p in pts.split(step):
            dx, dy = p.real[:, None] - self.x, p.imag[:, None] - self.y
            r = torch.sqrt(dx * dx + dy * dy)
            a = self.w * r
            J0, Y0, J1, Y1 = _bessel(a)
            S = torch.complex(-0.25 * Y0 * self.s, 0.25 * J0 * self.s)
            c = 0.25 * self.w * (dx * self.n1 + dy * self.n2) / r
            D = torch.complex(-c * Y1, c * J1)
            K = D - 1j * self.w * S if bc == "soft" else D / (1j * self.w) - S
            out.append(self.h * (K @ q.T))
        return torch.cat(out).T.contiguous()


def exact(case, seed):
    g = _gen(seed)
    if case["kind"] == "batch":
        out = []
        for sh, n, om in _stars(case):
            x = _density(_curve("star8", sh, n)[0], om, case["nrhs"], g)
            out.append(_Curve("star8", sh, n, om).apply("soft", x).reshape(-1))
        return torch.cat(out)
    c = _Curve(case["curve"], case["shape"], case["n"], case["omega"])
    if case["kind"] in ("solve", "request"):
        f = c.plane_waves(case["bc"], _angles(case, g))
        return torch.linalg.solve(c.matrix(case["bc"]), f.T).T.contiguous()
    z = _curve(case["curve"], case["shape"], case["n"])[0]
    x = _density(z, case["omega"], case["nrhs"], g)
    if case["kind"] == "field":
        return c.field(case["bc"], x, _points(z, case["npts"], g))
    return c.apply(case["bc"], x).contiguous()
