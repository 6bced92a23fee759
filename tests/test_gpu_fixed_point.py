"""The FP64 strips' fixed-point form (csrc/m1_fx.cuh) where it can go wrong:
neighbours of very unequal size (each cell's block has its own exponent), unequal
cell sides in both directions, c != 1, fluxes of full length along the axes, the
tile edges (30 columns, the strip heights), and cells no block can hold, whose
strips take the FP64 form.  Against the oracle, cell by cell.

Tolerance: both sides evaluate the same operator in 53 bits or more, so a result
differs from the oracle's by a few roundings of the largest term of its own stencil:
1e-12 of that term (the bound of the other kernel tests, taken locally)."""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2208_14703_gb300 import inputs

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
