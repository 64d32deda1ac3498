"""PIC transfers at the edges of their kernels: spacings whose division takes the correction step,
the exact reciprocal or the plain division, lines of fewer than 32 nodes and blocks of unfinished
lines, zero, subnormal, huge and non-finite potentials, particles on nodes, on the box faces, far
outside and not a number, charges from the subnormal to the huge."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_0907_4863_gb300 import inputs as I
from tests.oracle_cases import oracle_operator

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def S():
    import torch
    from paper_0907_4863_gb300 import build
    build.build()
    from paper_0907_4863_gb300 import saamg
    assert torch.cuda.is_available()
    torch.cuda.set_device(0)
    saamg.use_torch_allocator()
    return saamg


def dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a, np.float64)).cuda()


WORKLOADS = [
    I.Workload("pow2_spacing", I.cell_centred_grid(32), I.Domain(0.45, 0.30), I.LINEAR),
    I.Workload("short_lines", I.cell_centred_grid(13, 7, 5), I.Domain(0.45, 0.45), I.LINEAR),
    I.Workload("long_lines", I.cell_centred_grid(131, 11, 9), I.Domain(0.45, 0.30, taper=0.6),
               I.QUADRATIC),
    I.Workload("whole_box", I.vertex_grid(17), I.Domain(5.0, 5.0, zbc=I.Z_DIRICHLET), I.LINEAR),
    I.Workload("two_planes", I.cell_centred_grid(33, 35, 2), I.Domain(0.45, 0.45), I.CONSTANT),
]


@pytest.mark.parametrize("values", ["plain", "special"])
@pytest.mark.parametrize("w", WORKLOADS, ids=lambda w: w.name)
def test_gradient_bitwise(S, w, values):
    import torch
    o = oracle_operator(w)
    rng = np.random.default_rng(11)
    phi = rng.standard_normal(w.grid.nbox)
    if values == "special":
        pick = rng.integers(0, 12, w.grid.nbox)
        for k, v in enumerate([0.0, -0.0, 1e300, -1e305, 5e-324, 1e-310, 3e-200, np.inf, np.nan]):
            phi[pick == k] = v
    with np.errstate(all="ignore"):
        ref = O.field_gradient(o, phi)
    op = S.build_operator(S.make_domain(w.domain), S.make_grid(w.grid), w.mode)
    e = [torch.full((w.grid.nbox,), 7.0, dtype=torch.float64, device="cuda") for _ in range(3)]
    S.field_gradient(op, dev(phi), *e)
    for a, b in zip(e, ref):
        assert np.array_equal(a.cpu().numpy(), b, equal_nan=True)


@pytest.mark.parametrize("w", WORKLOADS, ids=lambda w: w.name)
def test_gradient_signs_of_zeros(S, w):
    """Potentials of zeros of either sign and few other values: differences that vanish, beside the
    wall too, keep the reference's sign."""
    import torch
    o = oracle_operator(w)
    rng = np.random.default_rng(12)
    op = S.build_operator(S.make_domain(w.domain), S.make_grid(w.grid), w.mode)
    for values in ([0.0], [-0.0], [0.0, -0.0, 1.0, -1.0]):
        phi = rng.choice(values, w.grid.nbox)
        ref = O.field_gradient(o, phi)
        e = [torch.empty(w.grid.nbox, dtype=torch.float64, device="cuda") for _ in range(3)]
        S.field_gradient(op, dev(phi), *e)
        for a, b in zip(e, ref):
            assert np.array_equal(a.cpu().numpy().view(np.int64), b.view(np.int64))


def edge_particles(g, rng):
    """Positions on nodes, on cell edges' neighbours, on and beyond the faces, far outside."""
    lo, h, n = np.array(g.origin), np.array(g.h), np.array(g.n)
    hi = lo + (n - 1) * h
    pts = [lo + rng.integers(0, n, size=(64, 3)) * h]                    # on nodes
    p = lo + rng.integers(0, n, size=(64, 3)) * h
    pts += [np.nextafter(p, -9.0), np.nextafter(p, 9.0)]                 # one unit beside them
    pts += [lo - h * rng.uniform(0, 1, (64, 3)), hi + h * rng.uniform(0, 1, (64, 3))]
    mix = rng.uniform(lo - 2 * h, hi + 2 * h, size=(512, 3))
    far = mix[:32].copy()
    far[:16, 0] = 1e12
    far[16:, 1] = -1e300
    pts += [mix, far, np.array([lo, hi, lo - h, hi + h, lo - 1e-18, 0.5 * (lo + hi)])]
    return [np.ascontiguousarray(c) for c in np.concatenate(pts).T]


GRIDS = [I.cell_centred_grid(32), I.cell_centred_grid(23, 37, 5), I.cell_centred_grid(2, 1, 3),
         I.Grid((40, 9, 11), (0.3, 0.125, 1e-3), (-3.0, 2.0, 100.0))]


@pytest.mark.parametrize("g", GRIDS, ids=lambda g: "x".join(map(str, g.n)))
def test_gather_bitwise(S, g):
    import torch
    rng = np.random.default_rng(5)
    e = [rng.standard_normal(g.nbox) for _ in range(3)]
    e[1][rng.integers(0, 3, g.nbox) == 0] = -0.0
    x, y, z = edge_particles(g, rng)
    ref = O.gather_cic(g, e, x, y, z)
    x, y, z = (np.append(c, np.nan) for c in (x, y, z))  # touches no node
    out = [torch.empty(len(x), dtype=torch.float64, device="cuda") for _ in range(3)]
    S.gather_cic(S.make_grid(g), *[dev(c) for c in e], dev(x), dev(y), dev(z), *out)
    for a, b in zip(out, ref):
        a = a.cpu().numpy()
        assert np.array_equal(a[:-1], b) and a[-1] == 0.0
        assert not np.any(np.signbit(a) & (a == 0.0))  # a sum from +0 never ends at -0


@pytest.mark.parametrize("special", [-0.0, 5e-324, -1e-310, 2.2250738585072014e-308, 1e-305, 1e300,
                                     -1.7976931348623157e308, np.inf, np.nan], ids=str)
@pytest.mark.parametrize("g", GRIDS[:2], ids=lambda g: "x".join(map(str, g.n)))
def test_gather_special_fields(S, g, special):
    """Field values whose products with the weights the integer multiplication hands back, or rounds
    at an end of the exponent range, in every component."""
    import torch
    rng = np.random.default_rng(9)
    e = [rng.standard_normal(g.nbox) for _ in range(3)]
    for c in e:
        c[rng.integers(0, 6, g.nbox) == 0] = special
    lo, h, n = np.array(g.origin), np.array(g.h), np.array(g.n)
    inner = rng.uniform(lo, lo + (n - 1) * h, size=(4096, 3)).T
    x, y, z = (np.concatenate(p) for p in zip(inner, edge_particles(g, rng)))
    with np.errstate(all="ignore"):
        ref = O.gather_cic(g, e, x, y, z)
    out = [torch.empty(len(x), dtype=torch.float64, device="cuda") for _ in range(3)]
    S.gather_cic(S.make_grid(g), *[dev(c) for c in e], dev(x), dev(y), dev(z), *out)
    for a, b in zip(out, ref):
        assert np.array_equal(a.cpu().numpy(), b, equal_nan=True)


@pytest.mark.parametrize("scale", [1.0, 1e-280, 1e-320, 1e250])
@pytest.mark.parametrize("g", GRIDS, ids=lambda g: "x".join(map(str, g.n)))
def test_deposit_edges(S, g, scale):
    """Against the oracle; the fixed-point unit is at most 2^-60 of the summed charge density, a
    node takes at most one unit of error from each particle, and the oracle's own sums (one rounding
    per contribution, as many products) 2^-50 of the node's absolute sum."""
    import torch
    rng = np.random.default_rng(6)
    x, y, z = edge_particles(g, rng)
    q = rng.standard_normal(len(x)) * scale
    q[::7] = 0.0
    ref = O.deposit_cic(g, x, y, z, q)
    bound = O.deposit_cic(g, x, y, z, np.abs(q))
    total = np.sum(np.abs(q) / ((g.h[0] * g.h[1]) * g.h[2]))
    x, y, z, q = np.append(x, np.nan), np.append(y, 0.0), np.append(z, 0.0), np.append(q, 0.0)
    rho = torch.full((g.nbox,), 7.0, dtype=torch.float64, device="cuda")
    S.deposit_cic(S.make_grid(g), dev(x), dev(y), dev(z), dev(q), rho)
    got = rho.cpu().numpy()
    tol = len(x) * 2.0 ** -60 * total + 2.0 ** -50 * bound + len(x) * 5e-324
    assert np.all(np.abs(got - ref) <= tol)


@pytest.mark.parametrize("count", [32, 33, 96, 1000])
@pytest.mark.parametrize("scale", [1.0, 1e-300, 1e200])
def test_deposit_of_one_cell(S, scale, count):
    """Particles that share a cell, warp by warp, and the same ones in turn with those of other
    cells (a corner cell of the box, one across its face): the sums are of integers, so the bits
    do not depend on the order."""
    import torch
    g = I.Grid((40, 9, 11), (0.3, 0.125, 1e-3), (-3.0, 2.0, 100.0))
    rng = np.random.default_rng(count)
    lo, h = np.array(g.origin), np.array(g.h)
    cells = np.array([[17, 4, 6], [38, 7, 9], [0, 0, 0], [39, 3, 3]])
    pts = lo + (cells[:, None, :] + rng.uniform(0, 1, (4, count, 3))) * h   # cell by cell
    q = rng.uniform(-1.0, 1.0, (4, count)) * scale
    sums = []
    for order in (lambda a: a, lambda a: np.swapaxes(a, 0, 1)):
        p, c = order(pts).reshape(-1, 3), order(q).reshape(-1)
        rho = torch.full((g.nbox,), 7.0, dtype=torch.float64, device="cuda")
        S.deposit_cic(S.make_grid(g), *[dev(p[:, d]) for d in range(3)], dev(c), rho)
        sums.append(rho.cpu().numpy())
    assert np.array_equal(sums[0].view(np.int64), sums[1].view(np.int64))
    x, y, z = (np.ascontiguousarray(pts.reshape(-1, 3)[:, d]) for d in range(3))
    ref = O.deposit_cic(g, x, y, z, q.reshape(-1))
    bound = O.deposit_cic(g, x, y, z, np.abs(q.reshape(-1)))
    total = np.sum(np.abs(q) / ((g.h[0] * g.h[1]) * g.h[2]))
    assert np.all(np.abs(sums[0] - ref) <= q.size * 2.0 ** -60 * total + 2.0 ** -50 * bound)


def test_deposit_single_charges_to_the_unit(S):
    """One particle: every node within one fixed-point unit (2^-60 of the density) of the exact
    product, which integers of any size give."""
    import torch
    from fractions import Fraction as F
    g = I.cell_centred_grid(16)
    rng = np.random.default_rng(8)
    for _ in range(20):
        p = rng.uniform(-0.45, 0.45, 3)
        q = float(rng.uniform(0.1, 3.0)) * (1 if rng.integers(2) else -1)
        rho = torch.empty(g.nbox, dtype=torch.float64, device="cuda")
        S.deposit_cic(S.make_grid(g), *[dev([c]) for c in p], dev([q]), rho)
        got = rho.cpu().numpy().reshape(16, 16, 16)
        u = [(p[d] - g.origin[d]) / g.h[d] for d in range(3)]
        c = [int(np.floor(v)) for v in u]
        f = [F(u[d]) - c[d] for d in range(3)]
        v = F(q / ((g.h[0] * g.h[1]) * g.h[2]))
        for k in range(8):
            b = (k & 1, (k >> 1) & 1, k >> 2)
            w = v
            for d in range(3):
                w *= f[d] if b[d] else 1 - f[d]
            # plus the rounding of the result to a double
            unit = abs(float(v)) * 2.0 ** -59 + abs(float(w)) * 2.0 ** -53
            assert abs(F(float(got[c[2] + b[2], c[1] + b[1], c[0] + b[0]])) - w) <= F(unit)
