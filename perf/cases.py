"""The measured workloads: what programs that use the library have it do.

A program that uses this library runs a particle-in-cell code, or answers Poisson solves on pipes
of many shapes.  Its calls are those of the cases below: a solve on a hierarchy that it keeps
(every time step), the operator, hierarchy and solve of a geometry that it has not seen, a
hierarchy rebuilt on known aggregates when the grid spacing follows the bunch, one V-cycle used as
a preconditioner in the program's own Krylov loop, many small solves in one call, and the charge
deposition, the field and its gather at the particles around each solve.  Grids go from 32^3 to
256^3, odd and non-cubic ones among them; bunches from ten thousand to ten million particles.

Each case is a dict of plain values; prepare() makes what the program holds before the call (from
the seed alone), run() is one pass through the public calls, exact() the same outputs from plain
torch in 64 bits, written from the paper's equations.
"""
import math
import random

import torch

from paper_0907_4863_gb300 import saamg as S

MODES = {"constant": S.BC_CONSTANT, "linear": S.BC_LINEAR, "quadratic": S.BC_QUADRATIC}
PRECISIONS = {"fp64": S.PREC_FP64, "fp32": S.PREC_FP32, "bf16": S.PREC_FP32_BF16}
# wall: semi-axes of the cross-section at the first plane, and its scale at the last
WALLS = {"cylinder": (0.45, 0.45, 1.0), "pipe": (0.45, 0.30, 1.0), "taper": (0.45, 0.45, 0.30 / 0.45)}
RTOL = 1e-8


def listed():
    def solve(name, path, nx, ny, nz, wall, mode, precision, max_coarse, max_levels=10):
        return dict(name=name, path=path, nx=nx, ny=ny, nz=nz, wall=wall, mode=mode,
                    precision=precision, max_coarse=max_coarse, max_levels=max_levels)

    def pic(name, path, n, particles):
        return dict(name=name, path=path, nx=n, ny=n, nz=n, wall="pipe", particles=particles,
                    order="random")

    return [
        # the smallest grid: a time step's solve where every launch counts
        solve("solve_32", "solve", 32, 32, 32, "cylinder", "constant", "fp64", 1000, 3),
        # a time step's solve on the large elliptic pipe, whole method in FP64
        solve("solve_256", "solve", 256, 256, 256, "pipe", "linear", "fp64", 4096),
        # the same grid with quadratic extrapolation at the wall and the V-cycle in FP32
        solve("solve_256_quadratic_fp32", "solve", 256, 256, 256, "pipe", "quadratic", "fp32", 4096),
        # an uneven grid on a narrowing pipe, coarse operators stored in BF16
        solve("solve_taper_bf16", "solve", 141, 97, 203, "taper", "linear", "bf16", 1000),
        # a geometry not seen before: operator, hierarchy (with a coarsest level of more than a
        # thousand unknowns) and first solve
        solve("geometry_128", "geometry", 128, 128, 128, "pipe", "linear", "fp64", 4096),
        # the same on the large grid
        solve("geometry_256", "geometry", 256, 256, 256, "pipe", "linear", "fp64", 4096),
        # the grid spacing follows the bunch along z: the operator changes on the same unknowns
        # and the hierarchy is rebuilt on the aggregates it has, then one solve
        solve("respaced_fp32", "respaced", 183, 160, 171, "cylinder", "linear", "fp32", 1000),
        # one V-cycle on an uneven grid, as another Krylov loop calls it
        solve("vcycle_uneven", "vcycle", 193, 131, 160, "pipe", "linear", "fp64", 1000),
        # a stack of small uneven geometries with two right-hand sides each, in one call
        dict(name="batch_small", path="batch", instances=16, rhs=2, lo=32, hi=64, mode="linear",
             precision="fp32"),
        # the charges of a large bunch onto the grid, before the solve
        pic("deposit_256", "deposit", 256, 10_000_000),
        # the field of the solved potential, after it
        pic("field_256", "field", 256, 0),
        # the field at the particles
        pic("gather_256", "gather", 256, 10_000_000),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["solve", "solve", "geometry", "respaced", "vcycle", "batch", "deposit",
                       "field", "gather"])
    if path == "batch":
        lo = _log_int(rng, 32, 48)
        return dict(path=path, instances=rng.randint(2, 16), rhs=rng.randint(1, 2), lo=lo,
                    hi=rng.randint(lo, 64), mode=rng.choice(list(MODES)),
                    precision=rng.choice(list(PRECISIONS)))
    nx, ny, nz = (_log_int(rng, 32, 256) for _ in range(3))
    # a narrowing pipe's unknowns need not survive another spacing along z
    wall = rng.choice(["cylinder", "pipe"] if path == "respaced" else list(WALLS))
    if path in ("deposit", "field", "gather"):
        return dict(path=path, nx=nx, ny=ny, nz=nz, wall=wall,
                    particles=0 if path == "field" else _log_int(rng, 10_000, 10_000_000),
                    order=rng.choice(["random", "cells"]))
    # a V-cycle is returned in FP64 and called in FP64 by other Krylov loops
    precision = "fp64" if path == "vcycle" else rng.choice(list(PRECISIONS))
    return dict(path=path, nx=nx, ny=ny, nz=nz, wall=wall, mode=rng.choice(list(MODES)),
                precision=precision, max_coarse=1000, max_levels=10)


# ---------------------------------------------------------------------------------------------
# inputs, from the seed alone
# ---------------------------------------------------------------------------------------------
def _spacing(case):
    return [1.0 / case["nx"], 1.0 / case["ny"], 1.0 / case["nz"]]


def _axes(case, h=None):
    n = (case["nx"], case["ny"], case["nz"])
    h = h or _spacing(case)
    return [-0.5 + 0.5 / n[d] + torch.arange(n[d], dtype=torch.float64, device="cuda") * h[d]
            for d in range(3)]


def _bunch_centre(seed, k=0):
    rng = random.Random(1000 * seed + k)
    return [c + rng.uniform(-0.02, 0.02) for c in (0.08, 0.04, 0.10)]


def _charge(case, seed, k=0):
    """Gaussian bunch of charge on the box (x fastest), sigma 0.1, 0.1, 0.2, jittered centre."""
    c = _bunch_centre(seed, k)
    g = [torch.exp(-0.5 * ((x - c[d]) / s) ** 2)
         for d, (x, s) in enumerate(zip(_axes(case), (0.1, 0.1, 0.2)))]
    return (g[2][:, None, None] * g[1][None, :, None] * g[0][None, None, :]).reshape(-1).contiguous()


def _particles(case, seed):
    """A bunch inside the box: normal positions cut at the outermost nodes, equal charges; in the
    order they were made ("random") or by lattice cell ("cells"), as a code that sorts holds them."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    n = case["particles"]
    c = _bunch_centre(seed)
    pos = []
    for d, (x, s) in enumerate(zip(_axes(case), (0.1, 0.1, 0.2))):
        lo, hi = (0.5 + 0.5 * math.erf((float(x[e]) - c[d]) / (s * math.sqrt(2.0))) for e in (0, -1))
        u = lo + (hi - lo) * torch.rand(n, dtype=torch.float64, device="cuda", generator=gen)
        p = c[d] + s * math.sqrt(2.0) * torch.erfinv(2.0 * u - 1.0)
        pos.append(p.clamp_(float(x[0]), float(x[-1]) - 1e-9))
    if case["order"] == "cells":
        h, key = _spacing(case), torch.zeros(n, dtype=torch.int64, device="cuda")
        for d, m in ((2, 1), (1, case["ny"]), (0, case["nx"])):
            key = key * m + torch.floor((pos[d] + 0.5 - 0.5 * h[d]) / h[d]).to(torch.int64)
        at = torch.argsort(key)
        pos = [p[at].contiguous() for p in pos]
    q = torch.full((n,), 1.0 / n, dtype=torch.float64, device="cuda")
    return pos[0], pos[1], pos[2], q


def _potential(case, seed):
    """A smooth potential on the box, as a solve leaves it at the unknowns."""
    c = _bunch_centre(seed)
    x, y, z = _axes(case)
    r2 = ((x - c[0])[None, None, :] ** 2 + (y - c[1])[None, :, None] ** 2
          + 0.3 * (z - c[2])[:, None, None] ** 2)
    return (1.0 / (0.05 + r2)).reshape(-1).contiguous()


def _field(case, seed):
    """A smooth vector field on the box, as field_gradient leaves it."""
    c = _bunch_centre(seed)
    x, y, z = _axes(case)
    dx, dy, dz = (x - c[0])[None, None, :], (y - c[1])[None, :, None], (z - c[2])[:, None, None]
    w = 1.0 / (0.05 + dx ** 2 + dy ** 2 + 0.3 * dz ** 2) ** 2
    return [(f * w).reshape(-1).contiguous() for f in (dx, dy, 0.3 * dz)]


def _instances(case, seed):
    """The geometries of a batch: sizes uniform per axis, cylinder / pipe / taper in turn.  The
    sizes are the case's; the seed moves the bunches."""
    rng = random.Random(4321)
    out = []
    for k in range(case["instances"]):
        n = [rng.randint(case["lo"], case["hi"]) for _ in range(3)]
        out.append(dict(nx=n[0], ny=n[1], nz=n[2], wall=list(WALLS)[k % 3], mode=case["mode"],
                        precision=case["precision"], max_coarse=1000, max_levels=10))
    return out


# ---------------------------------------------------------------------------------------------
# the calls
# ---------------------------------------------------------------------------------------------
def _grid(case, h=None):
    n = (case["nx"], case["ny"], case["nz"])
    h = h or _spacing(case)
    g = S.Grid()
    for d in range(3):
        g.n[d], g.h[d], g.origin[d] = n[d], h[d], -0.5 + 0.5 / n[d]
    return g


def _operator(case, h=None):
    a, b, taper = WALLS[case["wall"]]
    return S.build_operator(S.Domain(a, b, taper, 0.0, 0.0, S.Z_ROBIN, 1), _grid(case, h),
                            MODES[case.get("mode", "linear")])


def _params(case):
    mixed = case["precision"] != "fp64"
    return S.params_default(precision=PRECISIONS[case["precision"]], beta_rule=1 if mixed else 0,
                            max_coarse=case["max_coarse"], max_levels=case["max_levels"])


def _respaced(case):
    """The z spacing of a bunch that has grown by a seventh; the wall of a straight pipe does not
    depend on z, so the unknowns stay."""
    h = _spacing(case)
    return [h[0], h[1], h[2] * 8.0 / 7.0]


def prepare(case, seed):
    S.use_torch_allocator()
    path, st = case["path"], dict(case=case)
    if path == "batch":
        st.update(hs=[], rho=[], phi=[])
        for k, inst in enumerate(_instances(case, seed)):
            h = S.setup(_operator(inst), _params(inst))
            for r in range(case["rhs"]):
                st["hs"].append(h)
                st["rho"].append(_charge(inst, seed, 16 * k + r))
                st["phi"].append(torch.zeros_like(st["rho"][-1]))
        return st
    if path in ("deposit", "gather"):
        st["grid"] = _grid(case)
        st["particles"] = _particles(case, seed)
        if path == "deposit":
            st["rho"] = torch.empty(case["nx"] * case["ny"] * case["nz"], dtype=torch.float64,
                                    device="cuda")
        else:
            st["field"] = _field(case, seed)
            st["at"] = [torch.empty_like(st["particles"][0]) for _ in range(3)]
        return st
    if path == "field":
        st["op"] = _operator(case)
        st["phi"] = _potential(case, seed)
        st["field"] = [torch.empty_like(st["phi"]) for _ in range(3)]
        return st
    if path in ("solve", "vcycle", "respaced"):
        st["h"] = S.setup(_operator(case), _params(case))
    if path == "vcycle":
        gen = torch.Generator(device="cuda")
        gen.manual_seed(seed)
        n = st["h"].op.size()[0]
        st["r"] = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)
        st["z"] = torch.empty_like(st["r"])
        return st
    st["rho"] = _charge(case, seed)
    st["phi"] = torch.zeros_like(st["rho"])
    return st


def run(st):
    case = st["case"]
    path = case["path"]
    if path == "deposit":
        x, y, z, q = st["particles"]
        S.deposit_cic(st["grid"], x, y, z, q, st["rho"])
        return st["rho"]
    if path == "gather":
        x, y, z, _ = st["particles"]
        S.gather_cic(st["grid"], *st["field"], x, y, z, *st["at"])
        return st["at"]
    if path == "field":
        S.field_gradient(st["op"], st["phi"], *st["field"])
        return st["field"]
    if path == "vcycle":
        S.vcycle(st["h"], st["r"], st["z"])
        return st["z"]
    if path == "batch":
        for p in st["phi"]:
            p.zero_()
        S.solve_batched(st["hs"], st["rho"], st["phi"], rtol=RTOL)
        return st["phi"]
    st["phi"].zero_()
    if path == "solve":
        S.solve(st["h"], st["rho"], st["phi"], rtol=RTOL)
        return st["phi"]
    if path == "geometry":
        op = _operator(case)
        h = S.setup(op, _params(case))
    else:  # respaced
        op = _operator(case, _respaced(case))
        h = S.setup_reuse(op, st["h"], _params(case))
    S.solve(h, st["rho"], st["phi"], rtol=RTOL)
    h.free()
    op.free()
    return st["phi"]


# ---------------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------------
def _unknowns(case):
    a, b, t = WALLS[case["wall"]]
    return case["nx"] * case["ny"] * case["nz"] * math.pi * a * b * (1.0 + t + t * t) / 3.0


def _vcycle_work(n, precision):
    """Bytes and operations of one V-cycle of degree 2 on n unknowns: on the finest level four
    passes with the seven-point rows (two vectors read, one written), the transfers' 3.4 entries a
    row, and on the coarser levels about three stored entries per unknown, read four times."""
    v, e = (8, 10) if precision == "fp64" else (4, 6) if precision == "fp32" else (4, 4)
    return n * (4 * 3 * v + 2 * (3.4 * (4 + v) + 2 * v) + 4 * 3 * e), n * (4 * 15 + 2 * 6.8 + 4 * 6)


def _solve_work(case):
    n = _unknowns(case)
    nbox = case["nx"] * case["ny"] * case["nz"]
    its = round(6 + 1.9 * math.log2(nbox ** (1.0 / 3.0)))  # what this method takes to 1e-8
    vb, vf = _vcycle_work(n, case["precision"])
    return 16.0 * n + 8.0 * nbox + its * (88.0 * n + vb), its * (25.0 * n + vf)


def work(case):
    path = case["path"]
    if path == "batch":
        b, f = (sum(x) * case["rhs"] for x in zip(*(_solve_work(i) for i in _instances(case, 0))))
        return dict(bytes=b, flops=f)
    nbox = case["nx"] * case["ny"] * case["nz"]
    if path == "deposit":
        return dict(bytes=32.0 * case["particles"] + 8.0 * nbox, flops=40.0 * case["particles"])
    if path == "gather":
        return dict(bytes=48.0 * case["particles"] + 24.0 * min(nbox, 8 * case["particles"]),
                    flops=70.0 * case["particles"])
    n = _unknowns(case)
    if path == "field":
        return dict(bytes=8.0 * n + 24.0 * nbox, flops=6.0 * n)
    if path == "vcycle":
        b, f = _vcycle_work(n, case["precision"])
        return dict(bytes=b, flops=f)
    b, f = _solve_work(case)
    if path != "solve":
        # the operator's 7 entries a row, P and R (3.4 each), A P (9) and the next A (3) written
        # once and read by the product after them; eleven passes of the power iteration
        b += n * (2 * 12 * (7 + 2 * 3.4 + 9 + 3) + 11 * (16 + 3 * 10))
        f += n * (2 * (7 * 3.4 + 3.4 * 9) + 11 * (15 + 6))
    return dict(bytes=b, flops=f)


# ---------------------------------------------------------------------------------------------
# the same outputs in 64 bits, from the equations
# ---------------------------------------------------------------------------------------------
def _shift(t, axis, step, fill):
    """t at the neighbour `step` (+1 or -1) along axis (0 = x), `fill` beyond the box."""
    dim = 2 - axis
    out = torch.full_like(t, fill)
    m = t.shape[dim]
    out.narrow(dim, 0 if step > 0 else 1, m - 1).copy_(t.narrow(dim, 1 if step > 0 else 0, m - 1))
    return out


class _Lattice:
    """Inside test and boundary fractions of an elliptic pipe on the case's box (Sec. 2, 4.1)."""

    def __init__(self, case, h=None):
        self.case = case
        self.h = h or _spacing(case)
        self.a, self.b, self.taper = WALLS[case["wall"]]
        x, y, z = _axes(case, self.h)
        self.x, self.y, self.z = x[None, None, :], y[None, :, None], z[:, None, None]
        self.zlo, self.zhi = z[0], z[-1]
        self.sg = 1.0 + (self.taper - 1.0) * (self.z - self.zlo) / (self.zhi - self.zlo)
        u, v = self.x / (self.a * self.sg), self.y / (self.b * self.sg)
        self.inside = (u * u + v * v) - 1.0 < 0.0

    def neighbour(self, axis, step):
        return _shift(self.inside, axis, step, False)

    def fraction(self, axis, step):
        """0 < s <= 1: distance to the wall along the axis over the spacing (where it is outside)."""
        tiny = 2.0 ** -20
        if axis == 2:
            if self.taper == 1.0:
                return torch.ones_like(self.inside, dtype=torch.float64)
            q = torch.sqrt((self.x / self.a) ** 2 + (self.y / self.b) ** 2)
            d = step * (self.zlo + (q - 1.0) / (self.taper - 1.0) * (self.zhi - self.zlo) - self.z)
            return torch.where(d > 0, (d / self.h[2]).clamp(tiny, 1.0), torch.ones_like(d))
        p, o, pa, oa = (self.x, self.y, self.a, self.b) if axis == 0 else (self.y, self.x, self.b, self.a)
        w = pa * self.sg * torch.sqrt((1.0 - (o / (oa * self.sg)) ** 2).clamp(min=0.0))
        return ((w - step * p) / self.h[axis]).clamp(tiny, 1.0)


def _rows(lat):
    """Diagonal, six couplings (-x, +x, -y, +y, -z, +z) and the factor of the right-hand side of the
    finite-difference rows, Eqs. (6)-(12), Robin rows halved."""
    mode = lat.case["mode"]
    inside, nz = lat.inside, lat.inside.shape[0]
    diag = torch.zeros_like(inside, dtype=torch.float64)
    off = []
    for ax in range(3):
        c = 1.0 / (lat.h[ax] * lat.h[ax])
        m, p = lat.neighbour(ax, -1), lat.neighbour(ax, 1)
        s, t = lat.fraction(ax, -1), lat.fraction(ax, 1)
        f = torch.where(m, t, s)  # the one-sided fraction
        both, one = m & p, m ^ p
        unit = torch.ones_like(diag)
        if mode == "constant":
            dd, oo = 2.0 * unit, -unit
        elif mode == "linear":
            dd = torch.where(one, 1.0 + 1.0 / f, 1.0 / s + 1.0 / t)
            oo = -unit
        else:
            dd = torch.where(one, 2.0 / f, 2.0 / (s * t))
            oo = torch.where(one, -2.0 / (f + 1.0), -unit)
        dd = torch.where(both, 2.0 * unit, dd) * c
        om = torch.where(m, oo * c, 0.0 * unit)
        op = torch.where(p, oo * c, 0.0 * unit)
        if ax == 2:  # Robin planes, Eq. (11)
            robin = 2.0 * lat.h[2] / (0.5 * (nz - 1) * lat.h[2])
            for k, has, fr, mine, other in ((0, p, t, op, om), (nz - 1, m, s, om, op)):
                lone = 2.0 * unit[k] if mode == "constant" else 2.0 / fr[k]
                dd[k] = (torch.where(has[k], 2.0 * unit[k], lone) + robin) * c
                mine[k] = torch.where(has[k], -2.0 * c * unit[k], 0.0 * unit[k])
                other[k] = 0.0
        diag += dd
        off += [om, op]
    factor = torch.ones_like(diag)
    for k in (0, nz - 1):
        for t in [diag, factor] + off:
            t[k] *= 0.5
    out = ~inside
    diag[out] = 1.0
    factor[out] = 0.0
    for t in off:
        t[out] = 0.0
    return diag, off, factor


def _tight_solution(case, rho, h=None):
    """phi with A phi = rho to 1e-13, by conjugate gradients on the symmetric rows and BiCGStab on
    the quadratic ones, scaled by the diagonal; None if that does not get there."""
    lat = _Lattice(case, h)
    diag, off, factor = _rows(lat)
    sc = torch.where(lat.inside, 1.0 / torch.sqrt(diag), torch.zeros_like(diag))
    sxy = case["nx"] * case["ny"]
    steps = [-1, 1, -case["nx"], case["nx"], -sxy, sxy]
    scaled = []
    for q, t in enumerate(off):
        t = t * sc * _shift(sc, q // 2, 1 if q % 2 else -1, 0.0)
        scaled.append(t.reshape(-1))
    on = lat.inside.to(torch.float64).reshape(-1)
    b = (sc * factor).reshape(-1) * rho
    sc = sc.reshape(-1)
    del diag, off, factor

    def mul(v):
        y = v * on
        for t, d in zip(scaled, steps):
            if d > 0:
                y[:-d].addcmul_(t[:-d], v[d:])
            else:
                y[-d:].addcmul_(t[-d:], v[:d])
        return y

    x = torch.zeros_like(b)
    r = b.clone()
    goal = 1e-13 * float(b.norm())
    if case["mode"] != "quadratic":
        p, rr = r.clone(), r.dot(r)
        for k in range(4000):
            q = mul(p)
            alpha = rr / p.dot(q)
            x.addcmul_(p, alpha)
            r.addcmul_(q, -alpha)
            new = r.dot(r)
            if k % 16 == 15 and float(new) <= goal * goal:
                return x * sc
            p.mul_(new / rr).add_(r)
            rr = new
        return None
    best = None
    for _ in range(6):  # restarted from the true residual
        r = b - mul(x)
        if float(r.norm()) <= goal:
            return x * sc
        r0, p, rr = r.clone(), r.clone(), r.dot(r)
        for k in range(1500):
            v = mul(p)
            alpha = rr / r0.dot(v)
            s = r - alpha * v
            t = mul(s)
            om = t.dot(s) / t.dot(t)
            x.addcmul_(p, alpha).addcmul_(s, om)
            r = s - om * t
            new = r0.dot(r)
            p = r + (new / rr) * (alpha / om) * (p - om * v)
            rr = new
            if k % 16 == 15 and not float(r.norm()) > 0.5 * goal:
                break
        if not math.isfinite(float(x.norm())):
            return None
        best = x
    r = b - mul(best)
    return best * sc if float(r.norm()) <= 10.0 * goal else None


def _corners(case, x, y, z):
    """The eight (node, weight) pairs of each particle's cell; a node outside the box has weight 0."""
    n, h, o = (case["nx"], case["ny"], case["nz"]), _spacing(case), [-0.5 + 0.5 * e for e in _spacing(case)]
    cell, frac = [], []
    for d, p in enumerate((x, y, z)):
        u = (p - o[d]) / h[d]
        cell.append(torch.floor(u).to(torch.int64))
        frac.append(u - torch.floor(u))
    for k in (0, 1):
        for j in (0, 1):
            for i in (0, 1):
                at = [cell[0] + i, cell[1] + j, cell[2] + k]
                w = ((frac[0] if i else 1.0 - frac[0]) * (frac[1] if j else 1.0 - frac[1])
                     * (frac[2] if k else 1.0 - frac[2]))
                for d in range(3):
                    w = torch.where((at[d] >= 0) & (at[d] < n[d]), w, torch.zeros_like(w))
                    at[d] = at[d].clamp(0, n[d] - 1)
                yield at[0] + n[0] * (at[1] + n[1] * at[2]), w


def exact(case, seed):
    path = case["path"]
    if path == "vcycle":
        return None  # the multigrid hierarchy itself would have to be formed again
    if path == "batch":
        return [_tight_solution(inst, _charge(inst, seed, 16 * k + r))
                for k, inst in enumerate(_instances(case, seed)) for r in range(case["rhs"])]
    if path == "deposit":
        x, y, z, q = _particles(case, seed)
        rho = torch.zeros(case["nx"] * case["ny"] * case["nz"], dtype=torch.float64, device="cuda")
        h = _spacing(case)
        for at, w in _corners(case, x, y, z):
            rho.index_add_(0, at, w * (q / (h[0] * h[1] * h[2])))
        return rho
    if path == "gather":
        x, y, z, _ = _particles(case, seed)
        field = _field(case, seed)
        out = [torch.zeros_like(x) for _ in range(3)]
        for at, w in _corners(case, x, y, z):
            for e, f in zip(out, field):
                e.addcmul_(w, f[at])
        return out
    if path == "field":
        lat = _Lattice(case)
        phi = _potential(case, seed).reshape(lat.inside.shape)
        nz, out = case["nz"], []
        for ax in range(3):
            m, p = lat.neighbour(ax, -1), lat.neighbour(ax, 1)
            zero = torch.zeros_like(phi)
            # the derivative of the quadratic through the node and its two neighbours, an outside
            # neighbour being the wall point (value 0) at its boundary fraction
            hm = torch.where(m, 1.0 + zero, lat.fraction(ax, -1)) * lat.h[ax]
            hp = torch.where(p, 1.0 + zero, lat.fraction(ax, 1)) * lat.h[ax]
            vm = torch.where(m, _shift(phi, ax, -1, 0.0), zero)
            vp = torch.where(p, _shift(phi, ax, 1, 0.0), zero)
            e = -(hm * hm * vp - hp * hp * vm + (hp * hp - hm * hm) * phi) / (hm * hp * (hm + hp))
            if ax == 2:
                d = 0.5 * (nz - 1) * lat.h[2]
                e[0], e[nz - 1] = -phi[0] / d, phi[nz - 1] / d
            out.append(torch.where(lat.inside, e, zero).reshape(-1))
        return out
    h = _respaced(case) if path == "respaced" else None
    return _tight_solution(case, _charge(case, seed), h)
