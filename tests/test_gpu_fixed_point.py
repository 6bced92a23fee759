"""The FP64 strips' fixed-point form (csrc/m1_fx.cuh) where it can go wrong:
neighbours of very unequal size (each cell's block has its own exponent), unequal
cell sides in both directions, c != 1, fluxes of full length along the axes, the
tile edges (30 columns, the strip heights), and cells no block can hold, whose
strips take the FP64 form.  Against the oracle, cell by cell.

Tolerance: both sides evaluate the same operator in 53 bits or more, so a result
differs from the oracle's by a few roundings of the largest term of its own stencil:
1e-12 of that term (the bound of the other kernel tests, taken locally)."""
import math

import numpy as np
import pytest

from oracle import oracle as O
from oracle import oracle3d as O3
from paper_2208_14703_gb300 import inputs
from tests.test_oracle3d import opacities, random_state3

pytestmark = pytest.mark.gpu

m1 = pytest.importorskip("paper_2208_14703_gb300.m1")


def _case(nx, ny, ly, c, spread, bc, seed, tiny=0):
    case = inputs.random_admissible_2d(nx, ny, seed, fmax=1.0, cfl=30, bc=bc)
    rng = np.random.default_rng(seed)
    s = case["state"]
    s[:3] *= 10.0 ** rng.uniform(-spread, spread, (ny, nx)) if spread else 1.0
    ax = rng.integers(0, 8, (ny, nx))                 # a quarter of the cells: f = 1 along an axis
    for k, (fx, fy) in enumerate([(1, 0), (0, -1)]):
        s[1][ax == k], s[2][ax == k] = fx * s[0][ax == k], fy * s[0][ax == k]
    if tiny:                                          # cells below a block's range, at rest
        j, i = rng.integers(0, ny, tiny), rng.integers(0, nx, tiny)
        s[0][j, i], s[1][j, i], s[2][j, i] = 1e-170, 0.0, 0.0
    s[1:3] *= c
    case["desc"].update(c=c, ly=ly)
    if case["inflow"] is not None:
        case["inflow"][:, 1:] *= c
    return case


def _local(x, bc):
    """Largest magnitude over each cell and its four neighbours (walls: itself)."""
    p = np.pad(np.abs(x), 1, mode="wrap" if bc[0] == "periodic" else "edge")
    return np.max([p[1:-1, 1:-1], p[:-2, 1:-1], p[2:, 1:-1], p[1:-1, :-2], p[1:-1, 2:]], axis=0)


CASES = [
    ("square", dict(nx=61, ny=33, ly=33 / 61, c=1.0, spread=0, bc=("reflect",) * 4, seed=1)),
    ("unequal", dict(nx=64, ny=34, ly=34 / 64, c=1.0, spread=40, bc=("periodic",) * 4, seed=2)),
    ("wide-cells", dict(nx=31, ny=47, ly=0.3, c=1.0, spread=3, bc=("neumann",) * 4, seed=3)),
    ("tall-cells", dict(nx=90, ny=16, ly=5.0, c=1.0, spread=3, bc=("reflect",) * 4, seed=4)),
    ("light-speed", dict(nx=40, ny=24, ly=0.7, c=2.9979e3, spread=2, seed=5,
                         bc=("inflow", "reflect", "neumann", "inflow"))),
    ("out-of-range", dict(nx=70, ny=40, ly=40 / 70, c=1.0, spread=1, bc=("reflect",) * 4, seed=6,
                          tiny=5)),
    ("no-blocks", dict(nx=40, ny=18, ly=0.5, c=1e61, spread=1, bc=("reflect",) * 4, seed=8)),
]


@pytest.mark.parametrize("name,kw", CASES)
def test_fixed_point_strips_match_oracle(name, kw):
    case = _case(**kw)
    g = O.Grid.from_case(case)
    desc = m1.desc_from_case(case, lmax=1)
    dt, c, s = case["dt"], case["desc"]["c"], case["state"]
    sig = np.stack([case["sa"], case["ss"]])
    b = O.rhs_of(g, s)
    scale = _local(s[0], kw["bc"])
    wall = 1.0 if case["inflow"] is not None else 0.0
    d = 1.0 + c * dt * (s.shape[2] / case["desc"]["lx"] + s.shape[1] / case["desc"]["ly"])
    stiff = 1.0 + c * dt * (case["sa"] + case["ss"])

    # A(u): terms of size (diag + k) E of the stencil (T: its own row's terms)
    got, _ = m1.m1_op_level(desc, dt, sig, s, mode=m1.OP_APPLY, inflow=case["inflow"])
    ref = O.apply_A(g, dt, case["sa"], case["ss"], s)
    big = (d + stiff) * (np.maximum(scale, wall) + s[3] ** 4)
    for f, unit in enumerate((1.0, c, c)):
        assert np.max(np.abs(got[f] - ref[f]) / (big * unit)) <= 1e-12, (name, f)
    assert np.max(np.abs(got[3] - ref[3]) / (big + s[3])) <= 1e-12

    # one Jacobi sweep: E, F on the scale of the stencil and of the gas; T by its row
    # C_v T - k (E - T^4) = b_T, whose terms are of that size times k
    got, fails = m1.m1_op_level(desc, dt, sig, s, b, mode=m1.OP_JACOBI, inflow=case["inflow"])
    ref, it = O.jacobi_sweep(g, dt, case["sa"], case["ss"], b, s)
    assert it >= 0 and fails == 0
    big = np.maximum(scale, wall) + s[3] + ref[3] ** 4
    for f, unit in enumerate((1.0, c, c)):
        assert np.max(np.abs(got[f] - ref[f]) / (big * unit)) <= 1e-12, (name, f)
    ka, T = c * dt * case["sa"], got[3]
    row = T - ka * (got[0] - T ** 4) - b[3]
    assert np.max(np.abs(row) / (T + ka * (big + T ** 4) + b[3])) <= 1e-12


def test_strips_with_nan_stay_local():
    """A NaN in the right-hand side of the state reaches its neighbours only (the
    strip takes the FP64 form), as in FP64 arithmetic throughout."""
    case = _case(64, 40, 40 / 64, 1.0, 0, ("reflect",) * 4, 7)
    desc = m1.desc_from_case(case, lmax=1)
    sig = np.stack([case["sa"], case["ss"]])
    s = case["state"].copy()
    clean, _ = m1.m1_op_level(desc, case["dt"], sig, s, mode=m1.OP_APPLY)
    s[0, 20, 31] = np.nan
    got, _ = m1.m1_op_level(desc, case["dt"], sig, s, mode=m1.OP_APPLY)
    near = np.zeros(s.shape[1:], bool)
    near[20, 30:33] = near[19:22, 31] = True
    assert np.isnan(got[0][near]).all()
    far = ~near
    assert np.isfinite(got[:, far]).all()
    big = np.abs(clean).max()
    assert np.max(np.abs(got[:, far] - clean[:, far])) <= 1e-12 * big


def _local3(x, bc):
    p = np.pad(np.abs(x), 1, mode="wrap" if bc[0] == "periodic" else "edge")
    c = slice(1, -1)
    return np.max([p[c, c, c], p[:-2, c, c], p[2:, c, c], p[c, :-2, c], p[c, 2:, c], p[c, c, :-2],
                   p[c, c, 2:]], axis=0)


@pytest.mark.parametrize("name,dims,lengths,c,spread,bc,tiny", [
    ("equal", (33, 5, 4), (33.0, 5.0, 4.0), 1.0, 0, ("reflect",) * 6, 0),
    ("unequal-cells", (9, 31, 3), (1.0, 0.7, 2.0), 1.0, 2, ("periodic",) * 6, 0),
    ("unequal-states", (16, 8, 8), (16.0, 8.0, 8.0), 1.0, 40, ("neumann",) * 6, 0),
    ("light-speed", (7, 6, 20), (1.0, 1.0, 1.0), 2.9979e3, 1, ("reflect",) * 6, 0),
    ("out-of-range", (12, 11, 9), (1.2, 1.1, 0.9), 1.0, 1, ("reflect",) * 6, 6),
    ("no-blocks", (12, 6, 5), (1.0, 1.0, 1.0), 1e61, 1, ("reflect",) * 6, 0),
])
def test_fixed_point_3d_matches_oracle(name, dims, lengths, c, spread, bc, tiny):
    """A(u) and two Jacobi sweeps in 3D, on the scale of each cell's stencil."""
    nx, ny, nz = dims
    h = [lengths[a] / dims[a] for a in range(3)]
    dt = 3.0 * min(h) / c
    g = O3.Grid3(nx, ny, nz, *h, bc, c)
    d = m1.make_desc3(nx, ny, nz, *lengths, bc, c)
    rng = np.random.default_rng(11)
    s, b = random_state3(nx, ny, nz, 50, fmax=1.0), random_state3(nx, ny, nz, 51, fmax=0.95)
    if spread:
        s[:4] *= 10.0 ** rng.uniform(-spread, spread, (nz, ny, nx))
    if tiny:
        k, j, i = (rng.integers(0, n, tiny) for n in (nz, ny, nx))
        s[0][k, j, i], s[1:4, k, j, i] = 1e-170, 0.0
    s[1:4] *= c
    b[1:4] *= c
    sa, ss = opacities((nz, ny, nx), 52)
    sa, ss = sa / c, ss / c
    sig = np.stack([sa, ss])
    stiff = 1.0 + 3.0 * sum(min(h) / x for x in h) + c * dt * (sa + ss)
    got, _ = m1.m1_op_level3(d, dt, sig, s, mode=m1.OP3_APPLY)
    ref = O3.apply_A(g, dt, sa, ss, s)
    big = stiff * (_local3(s[0], bc) + s[4] ** 4 + s[4])
    for f, unit in enumerate((1.0, c, c, c, 1.0)):
        assert np.max(np.abs(got[f] - ref[f]) / (big * unit)) <= 1e-12, (name, f)
    # two sweeps: the second takes the blocks the first one wrote; E and F on the scale
    # of the stencil of the first one's result, T by its row
    got, _ = m1.m1_op_level3(d, dt, sig, s, rhs=b, mode=m1.OP3_JACOBI, sweeps=2)
    one, _ = O3.jacobi_sweep(g, dt, sa, ss, b, s)
    ref, _ = O3.jacobi_sweep(g, dt, sa, ss, b, one)
    big = _local3(_local3(s[0], bc) + b[0] + b[4], bc) + ref[4] ** 4
    for f, unit in enumerate((1.0, c, c, c)):
        assert np.max(np.abs(got[f] - ref[f]) / (big * unit)) <= 1e-12, (name, f)
    ka, T = c * dt * sa, got[4]
    row = T - ka * (got[0] - T ** 4) - b[4]
    assert np.max(np.abs(row) / (T + ka * (big + T ** 4) + b[4])) <= 1e-12


@pytest.mark.parametrize("power", [-2, -1, 0, 1, 3])
def test_local_solve_near_powers_of_two(power):
    """A gas at or close to rest at T near a power of two, where the fixed-point root's
    significand is at either end of its range: one Jacobi sweep against the oracle.
    A dozen roundings of the row's right-hand side R reach T (R's relative error bounds
    T's: g' T >= R) and E: 1e-14 of their sizes, taken ten times."""
    nx, ny = 60, 32
    rng = np.random.default_rng(20 + power)
    case = inputs.random_admissible_2d(nx, ny, 1, fmax=0.0, cfl=100, bc=("reflect",) * 4)
    off = rng.choice([-1.0, 1.0], (ny, nx)) * 10.0 ** rng.uniform(-17, -3, (ny, nx))
    T = 2.0 ** power * (1.0 + off)
    case["state"] = np.stack([T ** 4, 0.0 * T, 0.0 * T, T])
    g = O.Grid.from_case(case)
    s, dt = case["state"], case["dt"]
    b = O.rhs_of(g, s)
    desc = m1.desc_from_case(case, lmax=1)
    got, fails = m1.m1_op_level(desc, dt, np.stack([case["sa"], case["ss"]]), s, b, mode=m1.OP_JACOBI)
    ref, it = O.jacobi_sweep(g, dt, case["sa"], case["ss"], b, s)
    assert it >= 0 and fails == 0
    assert np.max(np.abs(got[3] / ref[3] - 1.0)) <= 1e-13
    assert np.max(np.abs(got[0] / ref[0] - 1.0)) <= 1e-13


@pytest.mark.parametrize("name", ["2d", "3d"])
def test_sums_carry_no_bias(name):
    """Radiation in vacuum within periodic walls keeps its total energy: Jacobi sweeps map a
    state of the total of b to one of it (sizes and time steps whose coefficients are exact).
    Rounding to nearest adds 2^-53 / sqrt(cells) a sweep at random, below 1e-16 over either
    run; a bias of 2^-58 of the sums in one direction adds 1e-14.  Bound: 3e-15."""
    rng = np.random.default_rng(3)
    if name == "2d":                                  # ten steps of some hundred sweeps
        case = inputs.riemann_2d(128, cfl=150.0, lmax=1, tol=5e-3)
        g = m1.grid_from_case(case)
        e0 = math.fsum(case["state"][0].ravel())
        for _ in range(10):
            g.implicit_step(case["dt"], m1.m1_default_params(tol=5e-3))
        e1 = math.fsum(np.asarray(g.get_state()[0]).ravel())
        g.close()
    else:                                             # one long run of sweeps
        n = 32
        E = 1.0 + rng.random((n, n, n))
        F = 0.1 * rng.standard_normal((3, n, n, n)) * E
        F *= np.minimum(1.0, 0.9 * E / np.linalg.norm(F, axis=0))
        s = np.concatenate([E[None], F, np.ones((1, n, n, n))])
        d = m1.make_desc3(n, n, n, 1.0, 1.0, 1.0, ("periodic",) * 6)
        out, _ = m1.m1_op_level3(d, 3000.0 / n, np.zeros((2, n, n, n)), s, rhs=s,
                                 mode=m1.OP3_JACOBI, sweeps=3000)
        e0, e1 = math.fsum(E.ravel()), math.fsum(np.asarray(out)[0].ravel())
    assert abs(e1 / e0 - 1.0) <= 3e-15


@pytest.mark.parametrize("name", ["2d", "3d"])
def test_scaled_sums_carry_no_bias(name):
    """test_sums_carry_no_bias with unequal cell sides (ratio 2, so that every coefficient
    is exact): the pairs of the longer sides are scaled.  20000 sweeps: a bias of half a unit of such a sum adds 5e-15 or more.  Same
    bound."""
    rng = np.random.default_rng(4)
    if name == "2d":
        nx, ny = 64, 64
        E = 1.0 + rng.random((ny, nx))
        F = 0.1 * rng.standard_normal((2, ny, nx)) * E
        F *= np.minimum(1.0, 0.9 * E / np.linalg.norm(F, axis=0))
        d = m1.make_desc(2, nx, ny, 1.0, 0.5, ("periodic",) * 4, 1)
        g = m1.Grid(d)
        zero = np.zeros((ny, nx))
        g.set_state(E, F[0], F[1], np.ones((ny, nx)), zero, zero)
        g.jacobi(3000.0 / nx, 20000)
        e1 = math.fsum(np.asarray(g.get_state()[0]).ravel())
        g.close()
    else:
        nx, ny, nz = 32, 32, 32
        E = 1.0 + rng.random((nz, ny, nx))
        F = 0.1 * rng.standard_normal((3, nz, ny, nx)) * E
        F *= np.minimum(1.0, 0.9 * E / np.linalg.norm(F, axis=0))
        s = np.concatenate([E[None], F, np.ones((1, nz, ny, nx))])
        d = m1.make_desc3(nx, ny, nz, 1.0, 0.5, 1.0, ("periodic",) * 6)
        out, _ = m1.m1_op_level3(d, 3000.0 / nx, np.zeros((2, nz, ny, nx)), s, rhs=s,
                                 mode=m1.OP3_JACOBI, sweeps=20000)
        e1 = math.fsum(np.asarray(out)[0].ravel())
    assert abs(e1 / math.fsum(E.ravel()) - 1.0) <= 3e-15


@pytest.mark.parametrize("ly", [0.4, 1.3])
def test_scaled_pairs_keep_zero(ly):
    """Unequal sides and a state uniform along one axis without flux in that direction: that
    flux stays exactly zero, as sums of zeros do."""
    nx = ny = 48
    rng = np.random.default_rng(6)
    desc = m1.make_desc(2, nx, ny, 1.0, ly, ("reflect",) * 4, 1)
    for axis in (0, 1):                               # uniform along y, then along x
        line = lambda lo, hi: np.broadcast_to((lambda v: v if axis == 0 else v[:, None])(
            rng.uniform(lo, hi, nx)), (ny, nx)).copy()
        E, f, T = line(0.5, 2), line(-0.9, 0.9), line(0.5, 2)
        s = np.stack([E, f * E if axis == 0 else 0 * E, f * E if axis else 0 * E, T])
        got, _ = m1.m1_op_level(desc, 10.0 / nx, np.stack([line(0.1, 1), line(0.1, 1)]), s, s,
                                mode=m1.OP_JACOBI)
        assert np.all(got[2 - axis] == 0.0)


def rows_exact(s, sig, dt, h, c):
    """A(u) on periodic walls (c_v = a_r = 1) in 80 bits and, for each value, the sum of the
    sizes of its terms.  Axes as in s: [E, F of the last axis, ..., T] over (.., y, x)."""
    L = np.longdouble
    d = s.ndim - 1
    s, sig = s.astype(L), sig.astype(L)
    E, F, T = s[0], s[1:1 + d], s[-1]
    f2 = sum(x * x for x in F) / (L(c) * E) ** 2
    root = np.sqrt(4 - 3 * f2)
    iso, q = (root - 1) / 3 * E, 3 / (2 + root) / (L(c) ** 2 * E)
    P = [[q * F[a] * F[b] + (iso if a == b else 0) for b in range(d)] for a in range(d)]
    beta = [L(dt) / (2 * L(x)) for x in h]
    diag = 1 + 2 * L(c) * sum(beta)
    ka, kt = L(c) * L(dt) * sig[0], L(c) * L(dt) * (sig[0] + sig[1])
    src = ka * (E - T ** 4)
    out = [diag * E + src] + [(diag + kt) * F[a] for a in range(d)] + [T - src]
    size = [np.abs(diag * E) + ka * (E + T ** 4)] + [np.abs((diag + kt) * F[a]) for a in range(d)] + [
        T + ka * (E + T ** 4)]
    for a in range(d):
        ax = d - 1 - a
        for side in (1, -1):                          # the low neighbour, then the high one
            n = lambda x: np.roll(x, side, axis=ax)
            out[0] = out[0] - beta[a] * (L(c) * n(E) + side * n(F[a]))
            size[0] = size[0] + beta[a] * (L(c) * n(E) + np.abs(n(F[a])))
            for b in range(d):
                out[1 + b] = out[1 + b] - L(c) * beta[a] * (n(F[b]) + side * L(c) * n(P[a][b]))
                size[1 + b] = size[1 + b] + L(c) * beta[a] * (np.abs(n(F[b])) + L(c) * np.abs(n(P[a][b])))
    return np.stack(out), np.stack(size)


@pytest.mark.parametrize("flux", [0.9, 1e-6, 1e-13])
@pytest.mark.parametrize("sides", [(1, 1), (1, 2.5), (5, 1), (1, 300), (3e4, 1), (1, 1e9), (1, 1, 3),
                                   (2, 1, 300), (1, 1e9, 1e3), (1, 1e21, 1)])
def test_rows_to_the_roundings_of_their_own_terms(sides, flux):
    """Each row of A(u), flux rows among them, to a few roundings (16) of its own terms, as
    FP64 arithmetic gives it, whatever the ratio of the cell sides and however small the
    fluxes beside E."""
    d = len(sides)
    shape = (24, 40) if d == 2 else (7, 9, 16)
    rng = np.random.default_rng(12)
    E = 10.0 ** rng.uniform(-1, 1, shape)
    F = rng.standard_normal((d,) + shape)
    F *= flux * rng.uniform(0, 1, shape) * E / np.linalg.norm(F, axis=0)
    s = np.concatenate([E[None], F, 10.0 ** rng.uniform(-0.3, 0.3, (1,) + shape)])
    sig = 10.0 ** rng.uniform(-2, 1, (2,) + shape)
    n = shape[::-1]
    h = [sides[a] / n[0] for a in range(d)]
    dt = 3.0 * min(h)
    if d == 2:
        desc = m1.make_desc(2, *n, h[0] * n[0], h[1] * n[1], ("periodic",) * 4, 1)
        got, _ = m1.m1_op_level(desc, dt, sig, s, mode=m1.OP_APPLY)
    else:
        desc = m1.make_desc3(*n, *(h[a] * n[a] for a in range(3)), ("periodic",) * 6)
        got, _ = m1.m1_op_level3(desc, dt, sig, s, mode=m1.OP3_APPLY)
    ref, size = rows_exact(s, sig, dt, h, 1.0)
    err = np.max(np.abs(got - ref) / size, axis=tuple(range(1, d + 1)))
    assert np.all(err <= 16 * 2.0 ** -53), err * 2.0 ** 53


@pytest.mark.parametrize("size", [1.0, 1e-9, 1e-20, 1e-200])
@pytest.mark.parametrize("shape", [(96,), (20, 70), (6, 10, 40)])
def test_small_fluxes_keep_their_bits(shape, size):
    """E varies along x only; the fluxes along x are of its size, those across it (Fy of a 1D
    grid too) far below.  The pressures of the pairs across x cancel exactly, so a row of A(u)
    across x holds fluxes and what goes with them alone: to a few roundings (16) of those terms,
    as in FP64 throughout.  Periodic walls, 80-bit reference with P split into E / 3 and the
    rest."""
    L, d = np.longdouble, len(shape)
    k = 2 if d == 1 else d                            # flux components
    rng = np.random.default_rng(13)
    E = np.broadcast_to(10.0 ** rng.uniform(-1, 1, shape[-1]), shape).copy()
    F = np.stack([E * rng.uniform(0.2, 0.5, shape) * (1 if a == 0 else size) for a in range(k)])
    for a in range(k):                                # the same on every line along x
        F[a] = F[a][(0,) * (d - 1)]
    T, sig = np.ones(shape), 10.0 ** rng.uniform(-2, 1, (2,) + shape)
    h, n = 1.0 / shape[-1], shape[::-1]
    dt = 3.0 * h
    if d < 3:
        desc = m1.make_desc(d, n[0], n[1] if d == 2 else 1, 1.0, n[1] * h if d == 2 else 1.0,
                            ("periodic",) * 4, 1)
        full = (n[1] if d == 2 else 1, n[0])
        s = np.concatenate([E[None], F, T[None]]).reshape((4,) + full)
        got, _ = m1.m1_op_level(desc, dt, sig.reshape((2,) + full), s, mode=m1.OP_APPLY)
        got = got.reshape((4,) + shape)
    else:
        desc = m1.make_desc3(*n, *(h * x for x in n), ("periodic",) * 6)
        got, _ = m1.m1_op_level3(desc, dt, sig, np.concatenate([E[None], F, T[None]]), mode=m1.OP3_APPLY)
    E, F = E.astype(L), F.astype(L)
    A = [1.5 * F[a] * F / (E + np.sqrt(E * E - 0.75 * (F * F).sum(0))) for a in range(k)]
    beta = L(dt) / (2 * L(h))
    dF = 1 + 2 * d * beta + L(dt) * (sig[0].astype(L) + sig[1].astype(L))
    for b in range(1, k):                             # the rows across x
        ref, terms = dF * F[b], dF * np.abs(F[b])
        for a in range(d):
            for side in (1, -1):
                near = lambda x: np.roll(x, side, axis=d - 1 - a)
                rest = 0 * E if a == b else A[a][b]   # its own pair's pressures cancel
                ref = ref - beta * (near(F[b]) + side * near(rest))
                terms = terms + beta * (np.abs(near(F[b])) + np.abs(near(rest)))
        assert np.max(np.abs(got[1 + b] - ref) / terms) <= 16 * 2.0 ** -53
