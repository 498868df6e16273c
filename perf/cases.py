"""The work that programs have this library do, as cases that can be timed and checked.

A case is one call (or one short sequence of calls) of the public binding, `aim.Context` and
`aim.matvec_multi`, on a seeded contour: products with the operators of an EFIE solve, whole
GMRES solves, several contexts in one launch, the bare grid product, and the setup of a new
geometry. Lengths follow the library's serving stream: ten segments per wavelength, a grid whose
spacing is about 0.16 wavelengths, alpha = min(8k, (2/3) pi / eps).

`exact` restates the method in plain torch (float64 and complex128) without the library: nodes ->
projections -> grid kernel -> FFT product -> interpolation, plus the near field from Gauss
quadrature, the Gram inverse from a cyclic tridiagonal solve, and dense solves.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2606_10784_gb300 import aim

S, QP = 4, 4                        # stencil points per axis, Gauss nodes per segment
PREC = {"fp64": aim.FP64, "mixed": aim.MIXED}


# ----------------------------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------------------------
def listed() -> list:
    te = {"kind": "product", "form": "te", "k": 2.0 * math.pi}
    return [
        # the smallest TE system a server accepts (5 wavelengths): one product is all launches
        {"name": "calderon_n64", **te, "perimeter": 5.0, "n": 64, "m": 32, "op": "calderon_alpha", "nrhs": 2,
         "precision": "fp64"},
        # TM-EFIE of a cylinder of about one wavelength radius, solved to the end: Arnoldi steps of
        # small kernels, one host read per iteration
        {"name": "tm_solve_n256", "kind": "solve", "form": "tm", "k": 2.0 * math.pi, "perimeter": 6.3, "n": 256, "m": 64,
         "op": "efie", "nrhs": 1, "precision": "fp64", "tol": 1e-11, "restart": 200},
        # the middle of the serving stream: 40 wavelengths, a handful of incidence angles, complex64 grid
        {"name": "serve_n400_mixed", **te, "perimeter": 40.0, "n": 400, "m": 128, "op": "calderon_alpha", "nrhs": 7,
         "precision": "mixed"},
        # sizes that are no powers of two, unfiltered (near field in both factors)
        {"name": "ragged_n733", **te, "perimeter": 73.3, "n": 733, "m": 201, "op": "calderon", "nrhs": 3,
         "precision": "fp64"},
        # the upper part of the serving stream, one incidence angle in full precision
        {"name": "serve_n1500", **te, "perimeter": 150.0, "n": 1500, "m": 512, "op": "calderon_alpha", "nrhs": 1,
         "precision": "fp64"},
        # eight small requests of the serving stream in one multi-context call
        {"name": "multi8_mixed", "kind": "multi", "form": "te", "k": 2.0 * math.pi, "count": 8, "longest": 100.0,
         "op": "calderon_alpha", "precision": "mixed"},
        # one GMRES iteration's product at the benchmark's size (1000 wavelengths), both precisions
        {"name": "single_n10000", **te, "perimeter": 1000.0, "n": 10000, "m": 2048, "op": "calderon_alpha", "nrhs": 1,
         "precision": "fp64"},
        {"name": "single_n10000_mixed", **te, "perimeter": 1000.0, "n": 10000, "m": 2048, "op": "calderon_alpha",
         "nrhs": 1, "precision": "mixed"},
        # the benchmark's batching workload: 64 incidence angles in every launch
        {"name": "batch64_n4000_mixed", **te, "perimeter": 400.0, "n": 4000, "m": 1024, "op": "calderon_alpha",
         "nrhs": 64, "precision": "mixed"},
        # Eq. 8 / Eq. 10 alone on full grids
        {"name": "grid_m500", "kind": "grid", "form": "te", "k": 2.0 * math.pi, "perimeter": 140.0, "n": 1400, "m": 500,
         "nrhs": 3, "precision": "fp64", "filtered": True},
        # a served request: mixed-precision refinement of the Calderon system, four angles
        {"name": "solve_n600_mixed", "kind": "solve", "form": "te", "k": 2.0 * math.pi, "perimeter": 60.0, "n": 600,
         "m": 192, "op": "calderon", "nrhs": 4, "precision": "mixed", "tol": 1e-10, "restart": 200},
        # a geometry that has not been seen: setup, excitation, its first product, release
        {"name": "setup_n1500", "kind": "setup", "form": "te", "k": 2.0 * math.pi, "perimeter": 150.0, "n": 1500, "m": 512,
         "op": "calderon_alpha", "nrhs": 2, "precision": "fp64"},
    ]


def _log_uniform(rng, lo: float, hi: float) -> float:
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid_side(perimeter_wl: float, rng) -> int:
    """Grid points per side for a spacing of about 0.16 wavelengths: the smallest power of two the
    server would take, or a size just as fine as needed."""
    need = 1.25 * perimeter_wl / math.pi / 0.16 + 8
    m = max(32, int(math.ceil(need * rng.uniform(1.0, 1.15))))
    if rng.random() < 0.5:
        m = 1 << (m - 1).bit_length()
    return min(m, 2048)


def draw(rng) -> dict:
    kind = rng.choices(["product", "solve", "multi", "grid", "setup"], [10, 3, 2, 2, 1])[0]
    k = rng.uniform(math.pi, 4.0 * math.pi)
    wl = 2.0 * math.pi / k
    precision = rng.choice(["fp64", "mixed"])
    if kind == "multi":
        return {"kind": kind, "form": "te", "k": k, "count": rng.randint(2, 10), "longest": rng.uniform(20.0, 110.0),
                "op": rng.choice(["calderon_alpha", "calderon", "N", "S_alpha"]), "precision": precision}
    if kind == "solve":
        per = _log_uniform(rng, 5.0, 70.0)
        tm = rng.random() < 0.4
        per = min(per, 20.0) if tm else per
        n = max(50, int(round((40.0 if tm else 10.0) * per)))
        return {"kind": kind, "form": "tm" if tm else "te", "k": k, "perimeter": per * wl, "n": n,
                "m": _grid_side(per * (2.5 if tm else 1.0), rng), "op": "efie" if tm else "calderon",
                "nrhs": rng.randint(1, 6), "precision": precision, "tol": 1e-11 if precision == "fp64" else 1e-10,
                "restart": 200}
    per = _log_uniform(rng, 5.0, 1000.0 if kind == "product" else 300.0)
    n = max(50, int(round(10.0 * per)))
    m = _grid_side(per, rng)
    case = {"kind": kind, "form": "te", "k": k, "perimeter": per * wl, "n": n, "m": m, "precision": precision}
    # right-hand sides: as many as keep the pass below the batching workload's
    cells = 4 * float(_embed(m)) ** 2 * (4 if precision == "fp64" else 1)
    most = max(1, min(64, int(1.0e9 / cells)))
    if kind == "grid":
        return {**case, "nrhs": rng.randint(1, max(1, min(6, most))), "filtered": rng.random() < 0.5}
    nrhs = int(round(_log_uniform(rng, 1.0, most))) if rng.random() < 0.6 else 1
    op = rng.choice(["calderon_alpha", "calderon_alpha", "calderon", "N", "S_alpha", "S", "N_alpha", "calderon_alpha2"])
    return {**case, "op": op if kind == "product" else "calderon_alpha", "nrhs": max(1, min(most, nrhs))}


# ----------------------------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------------------------
def _star(seed: int, perimeter: float, n: int) -> np.ndarray:
    """n vertices at equal arc length of a closed smooth curve r(phi) = 1 + sum eps_m cos(m phi + th_m)."""
    rng = np.random.default_rng(seed)
    eps, th = rng.uniform(0.0, 0.08, 8), rng.uniform(0.0, 2.0 * math.pi, 8)
    fine = max(4096, 16 * n)
    phi = 2.0 * math.pi * np.arange(fine + 1) / fine
    r = 1.0 + sum(e * np.cos((i + 1) * phi + t) for i, (e, t) in enumerate(zip(eps, th)))
    x, y = r * np.cos(phi), r * np.sin(phi)
    s = np.concatenate([[0.0], np.cumsum(np.hypot(np.diff(x), np.diff(y)))])
    at = s[-1] * np.arange(n) / n
    return np.stack([np.interp(at, s, x), np.interp(at, s, y)], axis=1) * (perimeter / s[-1])


def _embed(m: int) -> int:
    P = 64
    while P < 2 * m - 1:
        P *= 2
    return P


def _half_side(nodes: np.ndarray, m: int) -> float:
    return float(np.max(np.abs(nodes))) / (1.0 - (S + 2.0) / (m - 1.0))


def _alpha(nodes: np.ndarray, k: float, m: int) -> float:
    eps = 2.0 * _half_side(nodes, m) / (m - 1)
    return max(1.05 * k, min(8.0 * k, (2.0 / 3.0) * math.pi / eps))


def _random(shape, seed: int) -> np.ndarray:
    rng = np.random.default_rng([seed, 1])
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)) / math.sqrt(2.0)


def _requests(case: dict, seed: int) -> list:
    """The contexts of a case: (nodes, k, m, alpha, right-hand sides) each."""
    if case["kind"] != "multi":
        nodes = _star(seed, case["perimeter"], case["n"])
        return [(nodes, case["k"], case["m"], _alpha(nodes, case["k"], case["m"]), case["nrhs"])]
    out = []
    rng = np.random.default_rng(case["count"])      # the mix is the case's; contours and vectors the seed's
    for i in range(case["count"]):
        per = math.exp(rng.uniform(math.log(5.0), math.log(case["longest"])))
        k = case["k"] * rng.uniform(0.7, 1.4)
        m, nrhs = 32, int(rng.integers(1, 17))
        while m < 256 and 1.25 * per / math.pi / (m - 8) > 0.16:
            m *= 2
        nodes = _star(seed * 64 + i, per * 2.0 * math.pi / k, max(50, int(round(10.0 * per))))
        out.append((nodes, k, m, _alpha(nodes, k, m), nrhs))
    return out


def _angles(case: dict, seed: int) -> np.ndarray:
    return 2.0 * math.pi * np.random.default_rng([seed, 2]).uniform(size=case["nrhs"])


def _form(case: dict) -> int:
    return aim.TE if case["form"] == "te" else aim.TM


def prepare(case: dict, seed: int) -> dict:
    """A user's program before the call: contexts of its geometries and its vectors on the GPU."""
    kind, prec = case["kind"], PREC[case["precision"]]
    req = _requests(case, seed)
    st = {"case": case, "prec": prec}
    if kind == "setup":
        nodes, k, m, alpha, nrhs = req[0]
        st.update(nodes=nodes, k=k, m=m, alpha=alpha, angles=_angles(case, seed),
                  rhs=torch.empty((nrhs, len(nodes)), dtype=torch.complex128, device="cuda"),
                  y=torch.empty((nrhs, len(nodes)), dtype=torch.complex128, device="cuda"))
        return st
    ctxs = [aim.Context(nodes, k, _form(case), m, alpha=alpha) for nodes, k, m, alpha, _ in req]
    st["ctxs"] = ctxs
    if kind == "grid":
        nrhs, m = case["nrhs"], case["m"]
        u = torch.from_numpy(_random((nrhs, m, m), seed)).cuda()
        lo, hi = ctxs[0].info()["row_lo"], ctxs[0].info()["row_hi"]
        u[:, :lo] = 0                     # the product is defined on the context's rows, and 0 beyond them
        u[:, hi + 1:] = 0
        st.update(u=u, v=torch.empty_like(u))
        return st
    for ctx, r in zip(ctxs, req):
        ctx.reserve(r[4], prec)
    if kind == "solve":
        rhs = torch.empty((case["nrhs"], case["n"]), dtype=torch.complex128, device="cuda")
        ctxs[0].rhs_planewave(_angles(case, seed), rhs)
        st.update(rhs=rhs, x=torch.zeros_like(rhs), stream=torch.cuda.Stream())
        return st
    st["x"] = [torch.from_numpy(_random((r[4], len(r[0])), seed + i)).cuda() for i, r in enumerate(req)]
    st["y"] = [torch.empty_like(x) for x in st["x"]]
    return st


def _result(y: torch.Tensor, st: dict) -> torch.Tensor:
    # a program that asks for complex64 grid arithmetic holds the product as complex64
    return y.to(torch.complex64) if st["prec"] == aim.MIXED else y


def run(st: dict):
    case = st["case"]
    kind = case["kind"]
    if kind == "product":
        st["ctxs"][0].matvec(case["op"], st["x"][0], st["y"][0], precision=st["prec"])
        return _result(st["y"][0], st)
    if kind == "multi":
        aim.matvec_multi(st["ctxs"], [case["op"]] * len(st["ctxs"]), st["x"], st["y"], precision=st["prec"])
        return [_result(y, st) for y in st["y"]]
    if kind == "grid":
        st["ctxs"][0].grid_product(st["u"], st["v"], case["filtered"], precision=st["prec"])
        return _result(st["v"], st)
    if kind == "solve":
        st["ctxs"][0].solve(case["op"], st["rhs"], st["x"], tol=case["tol"], restart=case["restart"], max_iter=1000,
                            precision=st["prec"], stream=st["stream"])
        return st["x"]
    with aim.Context(st["nodes"], st["k"], _form(case), st["m"], alpha=st["alpha"]) as ctx:
        ctx.rhs_planewave(st["angles"], st["rhs"])
        ctx.matvec(case["op"], st["rhs"], st["y"], precision=st["prec"])
        torch.cuda.synchronize()          # the context's buffers are released below
    return [st["rhs"], _result(st["y"], st)]


def work(case: dict) -> dict:
    """Bytes: vectors in and out, projection lists, near field, Gram band and spectra, each once.
    Flops: pruned row and column transforms of every channel (5 L log2 L for each length-L line),
    spectral products, interpolation; products of a solve times a nominal iteration count."""
    el = 16 if case["precision"] == "fp64" else 8

    def grid_flops(m, channels):
        P = float(_embed(m))
        lines = 2 * m + 2 * P             # row transforms there and back, column transforms there and back
        return channels * (lines * 5 * P * math.log2(P) / 2 * 2 / 2 + 6 * P * P)

    def product(n, m, nrhs, op):
        passes = {"calderon": (3, 1), "calderon_alpha": (3, 1), "calderon_alpha2": (3, 1), "N": (3,), "N_alpha": (3,),
                  "S": (1,), "S_alpha": (1,), "efie": (1,)}[op]
        b = 2.0 * 16 * n * nrhs
        f = 0.0
        for ch in passes:
            b += n * 45 * 2 * (4 + 8 * ch) + n * 20 * (4 + el) + (_embed(m) // 2 + 1) ** 2 * el
            f += grid_flops(m, ch * nrhs) + nrhs * n * 45 * 8 * ch
        if op.startswith("calderon"):
            b += 81 * 8 * n
            f += 2 * nrhs * n * 81 * 4
        return b, f

    kind = case["kind"]
    if kind == "grid":
        b, f = 2.0 * 16 * case["nrhs"] * case["m"] ** 2 + (_embed(case["m"]) // 2 + 1) ** 2 * el, grid_flops(case["m"], case["nrhs"])
    elif kind == "multi":
        parts = [product(len(q[0]), q[2], q[4], case["op"]) for q in _requests(case, 0)]
        b, f = sum(p[0] for p in parts), sum(p[1] for p in parts)
    else:
        b, f = product(case["n"], case["m"], case["nrhs"], case["op"])
        if kind == "solve":
            it = 60
            b, f = b + it * it * case["n"] * case["nrhs"] * 16, it * f + 16.0 * it * it * case["n"] * case["nrhs"]
        if kind == "setup":
            b += 2 * 40 * (_embed(case["m"]) // 2 + 1) ** 2
            f += 50.0 * (_embed(case["m"]) // 2 + 1) ** 2 + case["n"] * 30 * 256 * 60
    return {"bytes": b, "flops": f}


# ----------------------------------------------------------------------------------------------
# the same values in plain torch, 64 bits
# ----------------------------------------------------------------------------------------------
def _dev():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _gauss(n: int):
    x, w = np.polynomial.legendre.leggauss(n)
    return torch.from_numpy(0.5 * (x + 1.0)), torch.from_numpy(0.5 * w)


def _bessel0(x: torch.Tensor):
    """J0 and Y0 of x > 0 (torch.special's are good to 1e-7 only around x = 5): power series below 2,
    Miller's backward recurrence with Neumann's series below 25, Hankel's expansion above."""
    J, Y = torch.empty_like(x), torch.empty_like(x)
    small, big = x < 2.0, x > 25.0
    mid = ~(small | big)
    z = x[small]
    t, j, s, harm = torch.ones_like(z), torch.ones_like(z), torch.zeros_like(z), 0.0
    for i in range(1, 20):
        t = t * (-z * z / (4.0 * i * i))
        harm += 1.0 / i
        j, s = j + t, s - harm * t
    J[small], Y[small] = j, (2.0 / math.pi) * ((torch.log(0.5 * z) + np.euler_gamma) * j + s)
    z = x[mid]
    up, cur, even, neu = torch.zeros_like(z), torch.full_like(z, 1e-150), torch.zeros_like(z), torch.zeros_like(z)
    for i in range(84, 0, -1):
        up, cur = cur, (2.0 * i / z) * cur - up                 # J_{i-1}, unnormalised
        if i > 1 and (i - 1) % 2 == 0:
            even, neu = even + cur, neu + (-1.0 if ((i - 1) >> 1) & 1 else 1.0) / ((i - 1) >> 1) * cur
    norm = cur + 2.0 * even
    j = cur / norm
    J[mid], Y[mid] = j, (2.0 / math.pi) * ((torch.log(0.5 * z) + np.euler_gamma) * j - 2.0 * neu / norm)
    z = x[big]
    a, p, q = torch.ones_like(z), torch.ones_like(z), torch.zeros_like(z)
    for i in range(1, 21):
        a = a * (-(2 * i - 1) ** 2) / (8.0 * i * z)
        sign = -1.0 if (i >> 1) & 1 else 1.0
        p, q = (p, q + sign * a) if i & 1 else (p + sign * a, q)
    c, s, amp = torch.cos(z), torch.sin(z), torch.sqrt(1.0 / (math.pi * z))
    J[big], Y[big] = amp * (p * (c + s) - q * (s - c)), amp * (p * (s - c) + q * (c + s))
    return J, Y


def _green(k: float, r: torch.Tensor) -> torch.Tensor:
    """-(j/4) H0^(2)(k r), r > 0."""
    x = (k * r).reshape(-1)
    out = []
    for v in torch.split(x, 1 << 23):
        j0, y0 = _bessel0(v)
        out.append(torch.complex(-0.25 * y0, -0.25 * j0))
    return torch.cat(out).reshape(r.shape) if out else torch.zeros(r.shape, dtype=torch.complex128, device=r.device)


class _Method:
    """The AIM operators of one context."""

    def __init__(self, nodes: np.ndarray, k: float, m: int, alpha: float, te: bool, near: bool):
        dev = _dev()
        self.k, self.m, self.n, self.te, self.P = k, m, len(nodes), te, _embed(m)
        self.L = _half_side(nodes, m)
        self.eps = 2.0 * self.L / (m - 1)
        self.v0 = torch.from_numpy(nodes).to(dev)
        self.v1 = torch.roll(self.v0, -1, 0)
        self.d = self.v1 - self.v0
        self.h = torch.hypot(self.d[:, 0], self.d[:, 1])
        t = self.d / self.h[:, None]
        self.nrm = torch.stack([t[:, 1], -t[:, 0]], 1)
        H = self.P // 2
        i = torch.arange(H + 1, dtype=torch.float64, device=dev)
        r = self.eps * torch.sqrt(i[:, None] ** 2 + i[None, :] ** 2)
        r[0, 0] = 1.0
        self.quarter = _green(k, r)
        self.quarter[0, 0] = 0.0
        cell = torch.arange(self.P, device=dev)
        cell = torch.minimum(cell, self.P - cell)
        self.hat = torch.fft.fft2(self.quarter[cell[:, None], cell[None, :]])
        c = cell.double()
        kappa = (2.0 * math.pi / (self.P * self.eps)) * torch.sqrt(c[:, None] ** 2 + c[None, :] ** 2)
        self.hat_alpha = torch.where(kappa <= alpha, self.hat, torch.zeros_like(self.hat))
        self._projections()
        if near:
            self._near()

    def _stencil(self, pts: torch.Tensor):
        """Grid indices and weights, (..., S) per axis, of the Lagrange stencils of points (..., 2)."""
        xi = (pts + self.L) / self.eps
        base = torch.floor(xi).long() - S // 2 + 1
        loc = xi - base
        w = torch.ones(xi.shape + (S,), dtype=torch.float64, device=pts.device)
        for a in range(S):
            for b in range(S):
                if b != a:
                    w[..., a] *= (loc - b) / (a - b)
        return base, w

    def _box(self, pts: torch.Tensor, vals: torch.Tensor):
        """Per unknown, the accumulated stencils of its points (n, u, 2) with values (n, u, q) in a
        common box: (origin (n, 2), weights (n, B, B, q))."""
        base, w = self._stencil(pts)
        org = base.amin(1)
        off = base - org[:, None, :]
        B = int(off.max()) + S
        W = torch.zeros((pts.shape[0], B * B, vals.shape[-1]), dtype=torch.float64, device=pts.device)
        a = torch.arange(S, device=pts.device)
        cell = (off[..., 1, None, None] + a[:, None]) * B + off[..., 0, None, None] + a[None, :]
        val = (w[..., 1, :, None] * w[..., 0, None, :])[..., None] * vals[:, :, None, None, :]
        n = pts.shape[0]
        W.scatter_add_(1, cell.reshape(n, -1, 1).expand(-1, -1, vals.shape[-1]), val.reshape(n, -1, vals.shape[-1]))
        yy, xx = torch.meshgrid(torch.arange(B, device=pts.device), torch.arange(B, device=pts.device), indexing="ij")
        pos = torch.stack([org[:, 0, None] + xx.reshape(-1), org[:, 1, None] + yy.reshape(-1)], -1)   # (n, B*B, 2)
        return pos.clamp(0, self.m - 1), W      # cells past the edge carry no weight

    def _projections(self):
        x, w = _gauss(QP)
        x, w = x.to(self.v0.device), w.to(self.v0.device)
        pts = self.v0[:, None, :] + x[None, :, None] * self.d[:, None, :]        # (n, QP, 2)
        wq = w[None, :] * self.h[:, None]
        if not self.te:
            self.src = self._box(pts, wq[..., None])
            mid = (0.5 * (self.v0 + self.v1))[:, None, :]
            self.tst = self._box(mid, torch.ones(mid.shape[:2] + (1,), dtype=torch.float64, device=mid.device))
            return
        def piece(phi, slope):
            return torch.stack([wq * phi, wq * slope / self.h[:, None], wq * phi * self.nrm[:, :1],
                                wq * phi * self.nrm[:, 1:]], -1)
        fall, rise = piece(1.0 - x[None, :], -1.0), piece(x[None, :], 1.0)
        prev = lambda t: torch.roll(t, 1, 0)  # noqa: E731
        self.src = self.tst = self._box(torch.cat([pts, prev(pts)], 1), torch.cat([fall, prev(rise)], 1))

    def _grid(self, u: torch.Tensor, hat: torch.Tensor) -> torch.Tensor:
        return torch.fft.ifft2(torch.fft.fft2(u, s=(self.P, self.P)) * hat)[..., :self.m, :self.m]

    def _pass(self, x: torch.Tensor, hat: torch.Tensor, proj, coef) -> torch.Tensor:
        y = torch.zeros_like(x)
        (sp, sw), (tp, tw) = self.src, self.tst
        at, to = sp[..., 1] * self.m + sp[..., 0], tp[..., 1] * self.m + tp[..., 0]
        for r in range(x.shape[0]):
            for q, c in zip(proj, coef):
                u = torch.zeros((self.m * self.m, 2), dtype=torch.float64, device=x.device)
                u.index_add_(0, at.reshape(-1), torch.view_as_real(x[r][:, None] * sw[..., q]).reshape(-1, 2))
                v = self._grid(torch.view_as_complex(u).reshape(self.m, self.m), hat).reshape(-1)
                y[r] += c * (v[to] * tw[..., q]).sum(1)
        return y

    def apply(self, op: str, x: torch.Tensor) -> torch.Tensor:
        k2 = self.k * self.k
        if op in ("S", "S_alpha"):
            y = self._pass(x, self.hat if op == "S" else self.hat_alpha, (0,), (1.0,))
            return y + self._near_add(0, x) if op == "S" else y
        if op in ("N", "N_alpha"):
            y = self._pass(x, self.hat if op == "N" else self.hat_alpha, (1, 2, 3), (1.0, -k2, -k2))
            return y + self._near_add(1, x) if op == "N" else y
        if op == "efie":
            return 1j * self.k * (self._pass(x, self.hat, (0,), (1.0,)) + self._near_add(0, x))
        first = "N_alpha" if op == "calderon_alpha2" else "N"
        second = "S" if op == "calderon" else "S_alpha"
        return self.gram_solve(self.apply(second, self.gram_solve(self.apply(first, x))))

    def gram_solve(self, b: torch.Tensor) -> torch.Tensor:
        """G^-1 b, G cyclic tridiagonal: Thomas elimination and the Sherman-Morrison corner."""
        h = self.h.cpu().numpy()
        n, rhs = self.n, b.cpu().numpy().T.copy()
        diag, up = (np.roll(h, 1) + h) / 3.0, h / 6.0
        low = np.roll(up, 1)
        g = -diag[0]
        dd = diag.copy()
        dd[0] -= g
        dd[-1] -= up[-1] * up[-1] / g
        u = np.zeros((n, 1))
        u[0], u[-1] = g, up[-1]
        z = np.concatenate([rhs, u], 1)
        cp = np.zeros(n)
        cp[0] = up[0] / dd[0]
        z[0] = z[0] / dd[0]
        for i in range(1, n):
            den = dd[i] - low[i] * cp[i - 1]
            cp[i] = up[i] / den
            z[i] = (z[i] - low[i] * z[i - 1]) / den
        for i in range(n - 2, -1, -1):
            z[i] -= cp[i] * z[i + 1]
        v = z[0] + up[-1] / g * z[-1]
        x = z[:, :-1] - np.outer(z[:, -1], v[:-1] / (1.0 + v[-1]))
        return torch.from_numpy(np.ascontiguousarray(x.T)).to(b.device)

    # ---- near field: exact entries minus their grid values
    def _dist(self, p, a, b):
        e = b - a
        t = (((p - a) * e).sum(-1) / (e * e).sum(-1)).clamp(0.0, 1.0)
        return torch.linalg.vector_norm(p - (a + t[..., None] * e), dim=-1)

    def _near(self):
        n, rad, dev = self.n, S * self.eps, self.v0.device
        a, b = self.v0, self.v1
        pairs = []
        for at in range(0, n, 256):
            s = slice(at, min(n, at + 256))
            if self.te:
                d = torch.minimum(torch.minimum(self._dist(a[s, None], a[None], b[None]), self._dist(b[s, None], a[None], b[None])),
                                  torch.minimum(self._dist(a[None], a[s, None], b[s, None]), self._dist(b[None], a[s, None], b[s, None])))
            else:
                d = self._dist((0.5 * (a + b))[s, None], a[None], b[None])
            i, j = torch.nonzero(d <= rad, as_tuple=True)
            pairs.append(torch.stack([i + at, j], 1))
        pr = torch.cat(pairs)
        if self.te:       # segment pair (e, f) touches hats {e, e+1} x {f, f+1}
            e, f = pr[:, 0], pr[:, 1]
            e1, f1 = (e + 1) % n, (f + 1) % n
            key = torch.unique(torch.cat([e * n + f, e * n + f1, e1 * n + f, e1 * n + f1]))
            pr = torch.stack([key // n, key % n], 1)
        self.ni, self.nj = pr[:, 0], pr[:, 1]
        nq = 4 if self.te else 1
        A = torch.empty((len(pr), nq), dtype=torch.complex128, device=dev)
        (sp, sw), (tp, tw) = self.src, self.tst
        step = max(1, (1 << 24) // (sp.shape[1] * tp.shape[1]))
        for at in range(0, len(pr), step):
            i, j = self.ni[at:at + step], self.nj[at:at + step]
            off = (tp[i][:, :, None, :] - sp[j][:, None, :, :]).abs()
            T = self.quarter[off[..., 1], off[..., 0]]
            A[at:at + step] = torch.einsum("paq,pab,pbq->pq", tw[i].to(T.dtype), T, sw[j].to(T.dtype))
        if not self.te:
            self.nv = [self._tm_entries() - A[:, 0]]
            return
        St, N = self._te_entries()
        k2 = self.k ** 2
        self.nv = [St - A[:, 0], N - (A[:, 1] - k2 * (A[:, 2] + A[:, 3]))]

    def _near_add(self, which: int, x: torch.Tensor) -> torch.Tensor:
        out = torch.empty_like(x)
        for r in range(x.shape[0]):
            y = torch.zeros((self.n, 2), dtype=torch.float64, device=x.device)
            y.index_add_(0, self.ni, torch.view_as_real(self.nv[which] * x[r][self.nj]))
            out[r] = torch.view_as_complex(y)
        return out

    def _quad(self, r: torch.Tensor, w: torch.Tensor) -> torch.Tensor:
        """sum over points u of g(r[p, u]) w[p, u, ...] for each pair p, in blocks."""
        out = []
        step = max(1, (1 << 23) // r.shape[1])
        for at in range(0, r.shape[0], step):
            ww = w[at:at + step] if w.shape[0] == r.shape[0] else w
            out.append(torch.einsum("pu,puq->pq", _green(self.k, r[at:at + step]), ww.to(torch.complex128).expand(len(r[at:at + step]), -1, -1)))
        return torch.cat(out)

    def _te_entries(self):
        """Exact S and N (Maue form) of the hat pairs from I_ab = int_e int_f psi_a g psi_b."""
        n, dev = self.n, self.v0.device
        prev = lambda t: (t + n - 1) % n  # noqa: E731
        e4 = torch.stack([self.ni, self.ni, prev(self.ni), prev(self.ni)], 1)
        f4 = torch.stack([self.nj, prev(self.nj), self.nj, prev(self.nj)], 1)
        key, inv = torch.unique((e4 * n + f4).reshape(-1), return_inverse=True)
        e, f = key // n, key % n
        I = torch.zeros((len(key), 4), dtype=torch.complex128, device=dev)      # [00, 01, 10, 11]
        hh = (self.h[e] * self.h[f])[:, None]
        x, w = (t.to(dev) for t in _gauss(24))
        same, nxt, prv = e == f, f == (e + 1) % n, e == (f + 1) % n
        # one segment: reduce to t = |sigma - tau|, graded t = u^6
        t, wt = x ** 6, 6.0 * x ** 5 * w
        q11 = 2.0 * ((1 - t) ** 3 / 3.0 + t * (1 - t) ** 2 / 2.0)
        q01 = (1.0 - t ** 3) / 3.0
        wgt = (wt[:, None] * torch.stack([q11, q01, q01, q11], 1))[None]
        I[same] = self._quad(self.h[e[same]][:, None] * t[None, :], wgt)
        # a shared vertex: Duffy, radial X = u^4
        xa, wa = (v.to(dev) for v in _gauss(16))
        X, wX = (x ** 4)[:, None].expand(-1, 16).reshape(-1), (4.0 * x ** 3 * w)[:, None].expand(-1, 16).reshape(-1)
        Y, wY = xa[None, :].expand(24, -1).reshape(-1), wa[None, :].expand(24, -1).reshape(-1)
        back, ahead = torch.cat([X, X * Y]), torch.cat([X * Y, X])     # distances from the vertex, as fractions
        jac = torch.cat([X * wX * wY] * 2)
        for sel, flip in ((nxt & ~same, False), (prv & ~same & ~nxt, True)):
            if not bool(sel.any()):
                continue
            a, b = (f[sel], e[sel]) if flip else (e[sel], f[sel])      # a ends where b begins
            r = torch.linalg.vector_norm(back[None, :, None] * self.d[a][:, None] + ahead[None, :, None] * self.d[b][:, None], dim=-1)
            pa, pb = (back, 1.0 - back), (1.0 - ahead, ahead)          # psi_0, psi_1 on each segment
            ww = torch.stack([jac * pa[c] * pb[g] for c in (0, 1) for g in (0, 1)], 1)[None]
            v = self._quad(r, ww)
            I[sel] = v[:, [0, 2, 1, 3]] if flip else v
        # apart: tensor Gauss
        sel = ~(same | nxt | prv)
        sg, tg = xa[:, None].expand(-1, 16).reshape(-1), xa[None, :].expand(16, -1).reshape(-1)
        w2 = (wa[:, None] * wa[None, :]).reshape(-1)
        ww = torch.stack([w2 * ps * pt for ps in (1 - sg, sg) for pt in (1 - tg, tg)], 1)[None]
        es, fs = e[sel], f[sel]
        got = []
        for at in range(0, len(es), 1 << 15):
            i, j = es[at:at + (1 << 15)], fs[at:at + (1 << 15)]
            r = torch.linalg.vector_norm((self.v0[i][:, None] + sg[None, :, None] * self.d[i][:, None])
                                         - (self.v0[j][:, None] + tg[None, :, None] * self.d[j][:, None]), dim=-1)
            got.append(self._quad(r, ww))
        if got:
            I[sel] = torch.cat(got)
        I = (I * hh)[inv].reshape(-1, 4, 4)                            # (pair, piece, ab)
        # pieces: (falling, falling), (falling, rising), (rising, falling), (rising, rising)
        St = I[:, 0, 0] + I[:, 1, 1] + I[:, 2, 2] + I[:, 3, 3]
        slope = torch.tensor([1.0, -1.0, -1.0, 1.0], device=dev, dtype=torch.float64)[None, :] / (self.h[e4] * self.h[f4])
        nn = (self.nrm[e4] * self.nrm[f4]).sum(-1)
        own = torch.stack([I[:, c, c] for c in range(4)], 1)
        N = (slope * I.sum(2) - self.k ** 2 * nn * own).sum(1)
        return St, N

    def _tm_entries(self):
        dev = self.v0.device
        mid = 0.5 * (self.v0 + self.v1)
        out = torch.zeros(len(self.ni), dtype=torch.complex128, device=dev)
        x, w = (t.to(dev) for t in _gauss(24))
        own = self.ni == self.nj
        h = self.h[self.nj]
        out[own] = self._quad(0.5 * h[own][:, None] * (x ** 6)[None, :], (6.0 * x ** 5 * w)[None, :, None])[:, 0] * h[own]
        i, j = self.ni[~own], self.nj[~own]
        r = torch.linalg.vector_norm(mid[i][:, None] - (self.v0[j][:, None] + x[None, :, None] * self.d[j][:, None]), dim=-1)
        out[~own] = self._quad(r, w[None, :, None])[:, 0] * h[~own]
        return out

    def planewave(self, angles: np.ndarray) -> torch.Tensor:
        rows = []
        x, w = (t.to(self.v0.device) for t in _gauss(16))
        for a in angles:
            ca, sa = math.cos(a), math.sin(a)
            if not self.te:
                mid = 0.5 * (self.v0 + self.v1)
                rows.append(torch.exp(-1j * self.k * (ca * mid[:, 0] + sa * mid[:, 1])))
                continue
            pts = self.v0[:, None] + x[None, :, None] * self.d[:, None]
            e = torch.exp(-1j * self.k * (ca * pts[..., 0] + sa * pts[..., 1])) * (ca * self.d[:, 1] - sa * self.d[:, 0])[:, None] * w[None, :]
            rows.append(1j * self.k * ((e * (1 - x)).sum(1) + torch.roll((e * x).sum(1), 1, 0)))
        return torch.stack(rows)


def exact(case: dict, seed: int):
    kind, te = case["kind"], case["form"] == "te"
    ops = case.get("op", "")
    near = kind != "grid" and ops not in ("S_alpha", "N_alpha", "calderon_alpha2")
    made = [(q, _Method(*q[:4], te, near)) for q in _requests(case, seed)]
    q, M = made[0]
    dev = M.v0.device
    if kind == "grid":
        u = torch.from_numpy(_random((case["nrhs"], case["m"], case["m"]), seed)).to(dev)
        rows = torch.unique(M.tst[0][..., 1][M.tst[1].abs().amax(-1) > 0])
        lo, hi = int(rows.min()), int(rows.max())
        u[:, :lo] = 0
        u[:, hi + 1:] = 0
        v = M._grid(u, M.hat_alpha if case["filtered"] else M.hat).clone()
        v[:, :lo] = 0
        v[:, hi + 1:] = 0
        return v
    if kind == "setup":
        rhs = M.planewave(_angles(case, seed))
        return [rhs, M.apply(ops, rhs)]
    if kind == "solve":
        rhs = M.planewave(_angles(case, seed))
        A = M.apply(ops, torch.eye(M.n, dtype=torch.complex128, device=dev)).T
        if te:      # the library solves G^-1 S G^-1 N x = G^-1 S G^-1 E
            rhs = M.gram_solve(M.apply("S", M.gram_solve(rhs)))
        return torch.linalg.solve(A, rhs.T).T
    got = [m.apply(ops, torch.from_numpy(_random((r[4], m.n), seed + i)).to(dev)) for i, (r, m) in enumerate(made)]
    return got[0] if kind == "product" else got
