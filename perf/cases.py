"""The performance cases of the tensor-product multigrid: what a host model has the
library do, from the smallest solve to the operational grid.

`listed()` names the cases, `draw(rng)` makes more of the same ranges, `prepare` builds
what a program holds before the call (the fields and the handle), `run` is one pass
through the package's entry points, `work` what a pass cannot do without, and `exact` the
same outputs from plain torch in 64 bits.

Inputs are the lat-lon pressure-correction system of the repository's workloads: cell-centred
finite volumes on a spherical shell (6371 km, 80 km deep, quadratic stretching, Courant
number 10), every cell's coefficients multiplied by the exponential of a smoothed Gaussian
field of deviation `sigma`, right-hand sides uniform in [-1, 1].  They are drawn on the GPU
so that the operational size is made in a second.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2307_04528_gb300.solver import MGBatch, MGHandle, NSHandle, mg_solve_fn

RADIUS, TOP, COURANT = 6371.0e3, 80.0e3, 10.0
TOL = 1e-10
# iterations that take the residual from 1 to 1e-10 at the rate these systems show
# (about a quarter per V-cycle-preconditioned iteration)
NEEDED = 16


# ----------------------------------------------------------------- cases
def listed():
    return [
        # The smallest solve in use: a coarse grid in FP64 (a test model, a column of an
        # intercomparison); latency and launches.
        dict(name="fp64_64x32x16", kind="solve", prec="fp64", nlon=64, nlat=32, nz=16, sigma=0.1),
        # One pressure solve per time step of a low-resolution climate member.
        dict(name="mixed_256x192x70", kind="solve", prec="mixed", nlon=256, nlat=192, nz=70,
             sigma=0.1),
        # A regional-climate grid with nothing a round number: odd layers, rows that are no
        # multiple of a warp, a coarsest level 11 columns wide.
        dict(name="mixed_352x226x37", kind="solve", prec="mixed", nlon=352, nlat=226, nz=37,
             sigma=0.2),
        # The ordinary solve of a time step at mid resolution.
        dict(name="mixed_512x384x70", kind="solve", prec="mixed", nlon=512, nlat=384, nz=70,
             sigma=0.1),
        # The operational grid: the headline solve, the largest case.
        dict(name="mixed_1536x1152x70", kind="solve", prec="mixed", nlon=1536, nlat=1152, nz=70,
             sigma=0.2),
        # The same method in double precision throughout (reference runs, validation).
        dict(name="fp64_1024x768x70", kind="solve", prec="fp64", nlon=1024, nlat=768, nz=70,
             sigma=0.1),
        # The shallow hierarchy of four levels with a Chebyshev coarsest-level solve, the
        # paper's configuration.
        dict(name="shallow_512x384x70", kind="shallow", nlon=512, nlat=384, nz=70, sigma=0.1),
        # Parameter estimation: one forward and one adjoint solve with the gradients of all
        # four coefficient fields, the hierarchy built anew for the new coefficients.
        dict(name="grad_256x128x32", kind="grad", nlon=256, nlat=128, nz=32, sigma=0.1),
        # Directed couplings (transport): one FP32 V-cycle and one FP64 application of the
        # system and of its transpose, the steps of a forward and of an adjoint model's own
        # Krylov solver.
        dict(name="ns_512x384x70", kind="ns", prec="fp32", nlon=512, nlat=384, nz=70, sigma=0.1),
        # An ensemble of uneven members solved together.
        dict(name="ensemble_5", kind="ensemble", nlon=1024, nlat=768, nz=70, sigma=0.1, large=1,
             half=2, quarter=2),
        # One FP32 V-cycle, the preconditioner inside a host model's own Krylov solver.
        dict(name="vcycle_fp32_1024x768x70", kind="vcycle", prec="fp32", nlon=1024, nlat=768,
             nz=70, sigma=0.1),
        # One operator application in FP64, the same solver's other half, at the operational
        # size.
        dict(name="apply_1536x1152x70", kind="apply", nlon=1536, nlat=1152, nz=70, sigma=0.2),
    ]


def _draw_nlon(rng, lo, hi):
    """An even number of longitudes in [lo, hi], uniform in the logarithm, that halves down
    to a dozen columns or fewer (an odd factor up to 11)."""
    while True:
        want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
        odd = rng.choice([1, 3, 5, 7, 9, 11])
        n = odd * 2 ** max(2, round(math.log2(want / odd)))
        if lo <= n <= hi and n >= 4 * odd:
            return n


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "solve", "shallow", "grad", "ns", "ensemble",
                       "vcycle", "apply"])
    hi = {"solve": 1408, "shallow": 768, "grad": 384, "ns": 768, "ensemble": 896,
          "vcycle": 1536, "apply": 1536}[kind]
    lo = {"ensemble": 256, "shallow": 128}.get(kind, 64)
    nlon = _draw_nlon(rng, lo, hi)
    nlat = 2 * max(8, round(nlon * rng.uniform(0.5, 0.75) / 2))
    nz = rng.choice([16, 32, 37, 50, 63, 70, 70, 70, rng.randrange(12, 71)])
    case = dict(kind=kind, nlon=nlon, nlat=nlat, nz=nz, sigma=rng.choice([0.1, 0.2]))
    if kind == "solve":
        case["prec"] = "fp64" if nlon <= 896 and rng.random() < 0.4 else "mixed"
    elif kind in ("vcycle", "ns"):
        case["prec"] = rng.choice(["fp32", "fp64"])
    elif kind == "ensemble":
        # members of nlon/2 and nlon/4 longitudes keep at least four halvings
        case["nlat"] = nlat - nlat % 8 or 8
        case.update(large=rng.randrange(0, 2), half=rng.randrange(1, 3),
                    quarter=rng.randrange(1, 4))
    return case


def _members(case):
    """(nlon, nlat, nz) of an ensemble's systems."""
    out = []
    for div, count in ((1, case["large"]), (2, case["half"]), (4, case["quarter"])):
        nlat = 2 * (case["nlat"] // div // 2)
        out += [(case["nlon"] // div, nlat, case["nz"])] * count
    return out


# ----------------------------------------------------------------- inputs
def _smooth(g):
    """Three-point running means along longitude (periodic), latitude and height."""
    g = (torch.roll(g, 1, 2) + g + torch.roll(g, -1, 2)) / 3.0
    for axis in (1, 0):
        n = g.shape[axis]
        if n == 1:
            continue
        out = g.clone()
        out.narrow(axis, 1, n - 1).add_(g.narrow(axis, 0, n - 1))
        out.narrow(axis, 0, n - 1).add_(g.narrow(axis, 1, n - 1))
        out.narrow(axis, 0, 1).div_(2.0)
        out.narrow(axis, n - 1, 1).div_(2.0)
        if n > 2:
            out.narrow(axis, 1, n - 2).div_(3.0)
        g = out
    return g


def _rows(nlon, nlat, nz):
    """Latitude faces, row centres, layer faces and layer centres (numpy)."""
    faces = -0.5 * np.pi + np.arange(nlat + 1) * (np.pi / nlat)
    faces[0], faces[-1] = -0.5 * np.pi, 0.5 * np.pi
    centres = -0.5 * np.pi + (np.arange(nlat) + 0.5) * (np.pi / nlat)
    rf = RADIUS + TOP * (np.arange(nz + 1) / nz) ** 2
    return faces, centres, rf, 0.5 * (rf[:-1] + rf[1:])


def _fields(nlon, nlat, nz, sigma, gen):
    """(tx, ty, tz, h) on the GPU, [nz, nlat, nlon] float64."""
    dlon, dlat = 2.0 * np.pi / nlon, np.pi / nlat
    K = (COURANT * RADIUS * dlon) ** 2
    faces, centres, rf, rc = _rows(nlon, nlat, nz)
    sin_f, cos_f = np.sin(faces), np.cos(faces)
    sin_f[0], sin_f[-1], cos_f[0], cos_f[-1] = -1.0, 1.0, 0.0, 0.0
    ds, cos_c = np.diff(sin_f), np.cos(centres)
    half = 0.5 * (rf[1:] ** 2 - rf[:-1] ** 2)[:, None]
    tx2 = K * dlat * half / (rc[:, None] * cos_c[None, :] * dlon)
    ty2 = K * cos_f[None, 1:] * dlon * half / (rc[:, None] * dlat)
    tz2 = np.zeros((nz, nlat))
    tz2[:-1] = K * rf[1:-1, None] ** 2 * dlon * ds[None, :] / np.diff(rc)[:, None]
    h2 = ((rf[1:] ** 3 - rf[:-1] ** 3) / 3.0)[:, None] * dlon * ds[None, :]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()[:, :, None]
    g = sigma * _smooth(torch.randn((nz, nlat, nlon), generator=gen, device="cuda",
                                    dtype=torch.float64))
    h = torch.exp(g) * dev(h2)
    tx = torch.exp(0.5 * (g + torch.roll(g, -1, 2))) * dev(tx2)
    ty, tz = torch.zeros_like(h), torch.zeros_like(h)
    ty[:, :-1] = torch.exp(0.5 * (g[:, :-1] + g[:, 1:])) * dev(ty2)[:, :-1]
    tz[:-1] = torch.exp(0.5 * (g[:-1] + g[1:])) * dev(tz2)[:-1]
    return tx, ty, tz, h


def _transport(fields, nlon, nlat, nz, gen, pe=0.3):
    """The seven arrays (h, tx, ty, tz, txr, tyr, tzr): upwind transport by a divergence-free
    flow of two stream functions, a fraction pe of each layer's longitude coupling."""
    tx, ty, tz, h = fields
    faces, centres, _, _ = _rows(nlon, nlat, nz)
    randn = lambda *shape: _smooth(torch.randn(shape, generator=gen, device="cuda",
                                               dtype=torch.float64))
    s = tx.reshape(nz, -1).median(dim=1).values[:, None, None]
    cos_f = torch.from_numpy(np.cos(faces)).cuda()[None, :, None]
    cos_c = torch.from_numpy(np.cos(centres)).cuda()[None, :, None]
    p1 = pe * s * cos_f * randn(nz, nlat + 1, nlon)
    p1[:, 0] = p1[:, nlat] = 0.0
    p2 = pe * torch.cat([s[:1], s]) * cos_c * randn(nz + 1, nlat, nlon)
    p2[0] = p2[nz] = 0.0
    fx = (p1[:, 1:] - p1[:, :-1]) + (p2[1:] - p2[:-1])
    fy = -(p1[:, 1:] - torch.roll(p1[:, 1:], 1, 2))
    fz = -(p2[1:] - torch.roll(p2[1:], 1, 2))
    fy[:, nlat - 1] = 0.0
    fz[nz - 1] = 0.0
    own = [t + torch.clamp(-f, min=0.0) for t, f in ((tx, fx), (ty, fy), (tz, fz))]
    back = [t + torch.clamp(f, min=0.0) for t, f in ((tx, fx), (ty, fy), (tz, fz))]
    return (h, *own, *back)


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _uniform(shape, gen, dtype=torch.float64):
    return torch.rand(shape, generator=gen, device="cuda", dtype=dtype) * 2.0 - 1.0


def _inputs(case, seed):
    """(coefficient tuples, right-hand sides, output gradient or None)."""
    gen = _gen(seed)
    grids = (_members(case) if case["kind"] == "ensemble" else
             [(case["nlon"], case["nlat"], case["nz"])])
    coeffs, rhs = [], []
    for nlon, nlat, nz in grids:
        c = _fields(nlon, nlat, nz, case["sigma"], gen)
        if case["kind"] == "ns":
            c = _transport(c, nlon, nlat, nz, gen)
        single = case["kind"] in ("vcycle", "ns") and case["prec"] == "fp32"
        coeffs.append(c)
        rhs.append(_uniform((nz, nlat, nlon), gen, torch.float32 if single else torch.float64))
    second = _uniform(rhs[0].shape, gen) if case["kind"] in ("grad", "ns") else None
    return coeffs, rhs, second


# ----------------------------------------------------------------- the calls
# four levels, 24 Chebyshev steps on the coarsest, up to 40 FP32 iterations a refinement step
SHALLOW = dict(levels=4, coarse_method=2, coarse_iters=24, inner_maxit=40)


def prepare(case, seed):
    coeffs, rhs, second = _inputs(case, seed)
    kind = case["kind"]
    state = dict(kind=kind, prec=case.get("prec"), b=rhs[0])
    if kind == "grad":
        tx, ty, tz, h = coeffs[0]
        state["args"] = [t.requires_grad_() for t in (rhs[0], h, tx, ty, tz)]
        state["gx"] = second
    elif kind == "ns":
        state["handle"] = NSHandle(*coeffs[0], mixed=int(case["prec"] == "fp32"))
        state["x"] = second
    elif kind == "ensemble":
        state["handle"] = MGBatch(coeffs, mixed=1)
        state["b"] = rhs
    elif kind == "shallow":
        state["handle"] = MGHandle(*coeffs[0], mixed=1, **SHALLOW)
    else:
        state["handle"] = MGHandle(*coeffs[0], mixed=int(case.get("prec") in ("mixed", "fp32")))
    return state


def run(state):
    kind, b, H = state["kind"], state["b"], state.get("handle")
    if kind == "solve":
        x, _ = H.solve_mixed(b, tol=TOL) if state["prec"] == "mixed" else H.solve(b, tol=TOL)
        return x
    if kind == "shallow":
        return H.solve_mixed(b, tol=TOL)[0]
    if kind == "grad":
        x = mg_solve_fn(*state["args"], tol=TOL)
        return [x, *torch.autograd.grad(x, state["args"], state["gx"])]
    if kind == "ns":
        p, x = int(state["prec"] == "fp32"), state["x"]
        return [H.vcycle(b, prec=p), H.vcycle(b, transpose=True, prec=p), H.apply(x),
                H.apply(x, transpose=True)]
    if kind == "ensemble":
        return H.solve(b, tol=TOL)[0]
    if kind == "vcycle":
        return H.vcycle(b, prec=1 if state["prec"] == "fp32" else 0)
    return H.apply(b)


def work(case):
    """Bytes: every field the call is given read once, every field it returns written once
    (8 bytes a value, 4 in single precision).  Operations: one operator application is 20
    flops a cell; a V-cycle with its transfers and coarser levels about 80; an iteration of a
    solve one of each and 6 for its vectors, NEEDED of them for ten digits."""
    kind = case["kind"]
    if kind == "ensemble":
        n = sum(a * b * c for a, b, c in _members(case))
    else:
        n = case["nlon"] * case["nlat"] * case["nz"]
    solve = 106 * NEEDED
    if kind == "apply":
        return dict(bytes=6 * 8 * n, flops=20 * n)
    if kind == "vcycle":
        # read: four coefficient fields and the residual
        return dict(bytes=6 * (4 if case["prec"] == "fp32" else 8) * n, flops=80 * n)
    if kind == "grad":
        # read: b, four coefficients, dL/dx; written: x and five gradients
        return dict(bytes=12 * 8 * n, flops=(2 * solve + 13) * n)
    if kind == "ns":
        # V-cycles: seven arrays and r read, two results written; applications the same
        single = 4 if case["prec"] == "fp32" else 8
        return dict(bytes=10 * (single + 8) * n, flops=200 * n)
    return dict(bytes=6 * 8 * n, flops=solve * n)


# ----------------------------------------------------------------- the same in plain torch
def _north(a):
    out = torch.zeros_like(a)
    out[:, :-1] = a[:, 1:]
    return out


def _south(a):
    out = torch.zeros_like(a)
    out[:, 1:] = a[:, :-1]
    return out


def _up(a):
    out = torch.zeros_like(a)
    out[:-1] = a[1:]
    return out


def _down(a):
    out = torch.zeros_like(a)
    out[1:] = a[:-1]
    return out


def _apply(arrays, u):
    """H u of the seven directed arrays (h, own couplings, couplings back)."""
    h, tx, ty, tz, txr, tyr, tzr = arrays
    y = h * u
    y += tx * (u - torch.roll(u, -1, 2))
    y += torch.roll(txr, 1, 2) * (u - torch.roll(u, 1, 2))
    y += ty * (u - _north(u))
    y += _south(tyr) * (u - _south(u))
    y += tz * (u - _up(u))
    y += _down(tzr) * (u - _down(u))
    return y


def _transposed(arrays):
    h, tx, ty, tz, txr, tyr, tzr = arrays
    ht = h + (tx - txr) + torch.roll(txr - tx, 1, 2) + (ty - tyr) + _south(tyr - ty)
    ht += (tz - tzr) + _down(tzr - tz)
    return (ht, txr, tyr, tzr, tx, ty, tz)


def _merge_rows(south, north, nlon_c, alpha_c=0.6):
    """Row groups (first, count) of the coarser level: pairs merged from the equator poleward
    while the merged cell keeps cos(theta) dlon / dlat >= alpha_c, mirrored at the equator."""
    n, groups, merging = len(south), [], True
    q = n // 2
    while q < n:
        if merging and q + 1 < n:
            a, b = south[q], north[q + 1]
            if math.cos(0.5 * (a + b)) * (2.0 * math.pi / nlon_c) / (b - a) >= alpha_c:
                groups.append((q, 2))
                q += 2
                continue
            merging = False
        groups.append((q, 1))
        q += 1
    return [(n - first - cnt, cnt) for first, cnt in reversed(groups)] + groups


class _Levels:
    """The V(1,1)-cycle in float64 of an operator given by its seven directed arrays (equal
    couplings both ways: the symmetric one): block-Jacobi sweeps on the column tridiagonals
    (relaxation 0.85), bilinear transfers, rediscretised coarse operators, 12 sweeps on the
    coarsest level."""

    OMEGA, COARSE_SWEEPS = 0.85, 12

    def __init__(self, arrays):
        self.lev = []
        h, tx, ty, tz, txr, tyr, tzr = arrays
        nlat = h.shape[1]
        south = [-0.5 * math.pi + j * (math.pi / nlat) for j in range(nlat)]
        north = south[1:] + [0.5 * math.pi]
        while True:
            s = h + tx + torch.roll(txr, 1, 2) + ty + _south(tyr)
            m, dq = torch.empty_like(h), torch.empty_like(h)
            q = s[0]
            for k in range(h.shape[0]):
                if k:
                    q = s[k] + tzr[k - 1] * dq[k - 1]
                m[k] = 1.0 / (q + tz[k])
                dq[k] = q * m[k]
            L = dict(tx=tx, ty=ty, txr=txr, tyr=tyr, tzr=tzr, m=m, dq=dq)
            L["big"] = max(float(a.max()) for a in (h, tx, ty, tz, txr, tyr, tzr))
            self.lev.append(L)
            nlon = h.shape[2]
            if nlon % 2 or nlon // 2 < 4:
                return
            g = _merge_rows(south, north, nlon // 2)
            mid = lambda a, b: [0.5 * (x + y) for x, y in zip(a, b)]
            cs, cn = [south[f] for f, _ in g], [north[f + c - 1] for f, c in g]
            fc, cc = mid(south, north), mid(cs, cn)
            # prolongation in latitude, fine rows x coarse rows
            P = np.zeros((len(south), len(g)))
            sy = np.zeros(len(g))
            for J, (f, c) in enumerate(g):
                for j in range(f, f + c):
                    d = fc[j] - cc[J]
                    Jn = J + 1 if d > 0 else J - 1
                    if d == 0.0 or not 0 <= Jn < len(g):
                        P[j, J] = 1.0
                    else:
                        P[j, Jn] = d / (cc[Jn] - cc[J])
                        P[j, J] = 1.0 - P[j, Jn]
                if J + 1 < len(g):
                    sy[J] = (fc[f + c] - fc[f + c - 1]) / (cc[J + 1] - cc[J])
            L["P"] = torch.from_numpy(P).cuda()
            first = torch.tensor([f for f, _ in g], device="cuda")
            last = torch.tensor([f + c - 1 for f, c in g], device="cuda")
            two = torch.tensor([float(c == 2) for _, c in g], device="cuda",
                               dtype=torch.float64)[None, :, None]
            ratio = torch.from_numpy(sy).cuda()[None, :, None]
            rows = lambda a: a[:, first] + two * a[:, last]
            pairs = lambda a: a[:, :, 0::2] + a[:, :, 1::2]
            h, tz, tzr = (rows(pairs(a)) for a in (h, tz, tzr))
            tx, txr = (0.5 * rows(a[:, :, 1::2]) for a in (tx, txr))
            ty, tyr = (ratio * pairs(a[:, last]) for a in (ty, tyr))
            south, north = cs, cn

    def _across(self, L, v, u):
        """v plus the four horizontal couplings of u."""
        return (v + L["tx"] * torch.roll(u, -1, 2) + torch.roll(L["txr"], 1, 2) *
                torch.roll(u, 1, 2) + L["ty"] * _north(u) + _south(L["tyr"]) * _south(u))

    def _sweep(self, L, b, u):
        v = b if u is None else self._across(L, b, u)
        y = torch.empty_like(b)
        for k in range(b.shape[0]):
            y[k] = (v[k] + (L["tzr"][k - 1] * y[k - 1] if k else 0.0)) * L["m"][k]
        for k in range(b.shape[0] - 2, -1, -1):
            y[k] = y[k + 1] + (y[k] - L["dq"][k] * y[k + 1])
        y *= self.OMEGA
        return y if u is None else y + (1.0 - self.OMEGA) * u

    def cycle(self, b, level=0):
        L = self.lev[level]
        u = self._sweep(L, b, None)
        if level + 1 == len(self.lev):
            for _ in range(self.COARSE_SWEEPS - 1):
                u = self._sweep(L, b, u)
            return u
        r = self._across(L, (1.0 - self.OMEGA) * b, u)
        even, odd = r[:, :, 0::2], r[:, :, 1::2]
        r = 0.75 * (even + odd) + 0.25 * (torch.roll(odd, 1, 2) + torch.roll(even, -1, 2))
        e = L["P"] @ self.cycle(L["P"].T @ r, level + 1)
        fine = torch.empty_like(u)
        fine[:, :, 0::2] = 0.75 * e + 0.25 * torch.roll(e, 1, 2)
        fine[:, :, 1::2] = 0.75 * e + 0.25 * torch.roll(e, -1, 2)
        return self._sweep(L, b, u + fine)

    def single(self, e, other=None):
        """e of a V-cycle in single precision, whose arrays are the float64 ones over the
        power of two above the largest of them (of both operators where there are two)."""
        big = max(L["big"] for v in (self, other) if v for L in v.lev)
        return e * 2.0 ** math.frexp(big)[1]


def _dot(a, b):
    return float(torch.dot(a.reshape(-1), b.reshape(-1)))


def _cg(arrays, levels, b):
    """H x = b by preconditioned conjugate gradients, run until rounding stops them."""
    x, r = torch.zeros_like(b), b.clone()
    z = levels.cycle(r)
    d, rz, bb = z.clone(), _dot(r, z), _dot(b, b)
    for _ in range(60):
        q = _apply(arrays, d)
        a = rz / _dot(d, q)
        x += a * d
        r -= a * q
        if _dot(r, r) <= 1e-28 * bb:
            break
        z = levels.cycle(r)
        old, rz = rz, _dot(r, z)
        d = z + (rz / old) * d
    return x


def exact(case, seed):
    coeffs, rhs, second = _inputs(case, seed)
    kind = case["kind"]
    single = case.get("prec") == "fp32"
    if kind == "ns":
        A = coeffs[0]
        T = _transposed(A)
        L, LT = _Levels(A), _Levels(T)
        out = [L.cycle(rhs[0].double()), LT.cycle(rhs[0].double())]
        if single:
            out = [L.single(e, LT) for e in out]
        return out + [_apply(A, second), _apply(T, second)]
    out = []
    for (tx, ty, tz, h), b in zip(coeffs, rhs):
        A = (h, tx, ty, tz, tx, ty, tz)
        if kind == "apply":
            return _apply(A, b)
        levels = _Levels(A)
        if kind == "vcycle":
            e = levels.cycle(b.double())
            return levels.single(e) if single else e
        x = _cg(A, levels, b)
        if kind != "grad":
            out.append(x)
            continue
        lam = _cg(A, levels, second)
        east = lambda a: torch.roll(a, -1, 2)
        gty = -(lam - _north(lam)) * (x - _north(x))
        gtz = -(lam - _up(lam)) * (x - _up(x))
        gty[:, -1] = 0.0
        gtz[-1] = 0.0
        return [x, lam, -lam * x, -(lam - east(lam)) * (x - east(x)), gty, gtz]
    return out if kind == "ensemble" else out[0]
