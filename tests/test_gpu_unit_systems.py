"""The step in unit systems far from c = 1 and E of order one: the same problems with E,
F, T, c, a_r and dt rescaled (CGS-like: c = 3e10, E near 1e12; and small: c = 1e-12,
E near 1e-11), where the limiter of the pseudo-time step and the damping of the
prolongation have to bind as often as in the units of the paper.  Against the oracle
in the same units.

Tolerances: those of the same comparisons at c = 1 (tests/test_gpu_kernels.py,
test_gpu_step.py, test_gpu_grid3.py), each field taken in its own unit; the scaling
changes no conditioning."""
import numpy as np
import pytest

from oracle import oracle as O
from oracle import oracle3d as O3
from paper_2208_14703_gb300 import inputs
from tests.test_gpu_grid3 import mixed_walls_case

pytestmark = pytest.mark.gpu

m1 = pytest.importorskip("paper_2208_14703_gb300.m1")

UNITS = {"cgs": dict(e=1e12, c=2.99792458e10), "small": dict(e=1e-11, c=1e-12)}


def rescale(case, e, c):
    """The case with energies and temperatures in units of 1/e (C_v stays one) and light
    speed c."""
    d = case["desc"] = dict(case["desc"])
    assert d["c"] == d["a_r"] == d["c_v"] == 1.0
    s = case["state"] = np.array(case["state"])
    s[0] *= e
    s[1:-1] *= e * c
    s[-1] *= e
    d.update(c=c, a_r=e ** -3)
    case["dt"] = case["dt"] / c
    return case


def rel(got, ref, c):
    nE = np.linalg.norm(ref[0])
    return max(np.linalg.norm(got[0] - ref[0]) / nE,
               np.linalg.norm(got[1:-1] - ref[1:-1]) / (c * nE),
               np.linalg.norm(got[-1] - ref[-1]) / np.linalg.norm(ref[-1]))


@pytest.mark.parametrize("units", UNITS)
def test_pseudo_step_limited_as_in_the_oracle(units):
    """One pseudo-time step of sources that would carry cells far beyond the cone or below
    E = 0, T = 0: a limiter that misses them leaves E, F or T off by their own size."""
    case = rescale(inputs.random_admissible_2d(64, 48, 3, fmax=0.99, cfl=30, bc=("reflect",) * 4),
                   **UNITS[units])
    c = UNITS[units]["c"]
    g = O.Grid.from_case(case)
    rng = np.random.default_rng(5)
    f = rng.standard_normal((4, 48, 64)) * case["state"][0] * 10.0 ** rng.uniform(-2, 1, (48, 64))
    f[1:3] *= c
    desc = m1.desc_from_case(case, lmax=1)
    sig = np.stack([case["sa"], case["ss"]])
    for dtau in (1e-3, 0.3):
        ref, it = O.pseudo_time_smooth(g, case["dt"], case["sa"], case["ss"], f, case["state"], dtau,
                                       m=1, nu=1, theta=0.5)
        got, fails = m1.m1_op_level(desc, case["dt"], sig, case["state"], f, mode=m1.OP_PSEUDO,
                                    dtau=dtau, theta=0.5)
        assert it >= 0 and fails == 0
        free, _ = m1.m1_op_level(desc, case["dt"], sig, case["state"], 1e-6 * f, mode=m1.OP_PSEUDO,
                                 dtau=dtau, theta=0.5)
        assert rel(ref, free, c) > 1e-3                # the sources matter
        assert rel(got, ref, c) <= 1e-12


@pytest.mark.parametrize("units", UNITS)
def test_prolongation_damps_the_same_cells(units):
    case = rescale(inputs.random_admissible_2d(64, 48, 3, fmax=0.99, cfl=30, bc=("reflect",) * 4),
                   **UNITS[units])
    g = O.Grid.from_case(case)
    c = UNITS[units]["c"]
    rng = np.random.default_rng(4)
    vc = O.restrict_state(g, case["state"])
    d = rng.normal(0, 0.6, vc.shape) * vc[0]
    d[1:3] *= c
    got, nd = m1.m1_op_prolong_correct(m1.desc_from_case(case, lmax=2), vc + d, vc, case["state"])
    ref, nd_ref = O.prolong_correct(g, vc + d, vc, case["state"])
    assert nd == nd_ref and nd > 0
    assert rel(got, ref, c) <= 1e-13


@pytest.mark.parametrize("units", UNITS)
@pytest.mark.parametrize("lmax,shape,nx,ny", [(3, 0, 272, 192), (4, 1, 64, 48)])
def test_step_matches_oracle(units, lmax, shape, nx, ny):
    """2D steps with the coarse levels in launches (272 x 192) and in one launch: cycles,
    history, damped cells and state."""
    case = rescale(inputs.random_admissible_2d(nx, ny, seed=9, fmax=0.99, cfl=20,
                                               bc=("reflect",) * 4, lmax=lmax), **UNITS[units])
    g = O.Grid.from_case(case)
    ref, ost, ohist, _ = O.implicit_step(
        g, case["dt"], case["sa"], case["ss"], case["state"],
        O.SolveParams(lmax=lmax, tol=1e-10, cycle=shape, max_cycles=4, dtau0=10.0))
    grid = m1.grid_from_case(case)
    st = grid.implicit_step(case["dt"], m1.m1_default_params(tol=1e-10, cycle=shape, max_cycles=4,
                                                             dtau0=10.0), allow_not_converged=True)
    out = np.stack(grid.get_state())
    hist, _ = grid.step_history(st.cycles + 1)
    grid.close()
    assert st.cycles == ost["cycles"]
    assert st.damped == ost["damped"] > 0
    np.testing.assert_allclose(hist, ohist, rtol=1e-9, atol=1e-13 * ohist[0])
    assert rel(out, ref, case["desc"]["c"]) <= 1e-10


@pytest.mark.parametrize("units", UNITS)
def test_step3_matches_oracle(units):
    case = mixed_walls_case()
    F = case["state"][1:4]                                # fluxes at the cone
    case["state"][1:4] = 0.999 * case["state"][0] * F / np.linalg.norm(F, axis=0)
    case["dt"] *= 0.1
    case = rescale(case, **UNITS[units])
    d = case["desc"]
    g = O3.Grid3(d["nx"], d["ny"], d["nz"], d["lx"] / d["nx"], d["ly"] / d["ny"], d["lz"] / d["nz"],
                 tuple(d["bc"]), d["c"], d["a_r"], d["c_v"], None)
    ref, ost, ohist = O3.implicit_step(g, case["dt"], case["sa"], case["ss"], case["state"],
                                       O3.SolveParams3(lmax=3, tol=1e-10, max_cycles=8, dtau0=10.0))
    grid = m1.grid3_from_case(case, lmax=3)
    st = grid.implicit_step(case["dt"], m1.m1_default_params(tol=1e-10, max_cycles=8, dtau0=10.0),
                            allow_not_converged=True)
    out = grid.get_state()
    hist, _ = grid.step_history(st.cycles + 1)
    grid.close()
    assert st.cycles == ost["cycles"]
    assert st.damped == ost["damped"] > 0
    np.testing.assert_allclose(hist, ohist, rtol=1e-8, atol=1e-12 * ohist[0])
    assert rel(out, ref, d["c"]) <= 1e-10


def fallback(case, kind):
    """The case where no block holds a cell (c = 1e61), where the cells are too long for the
    fixed-point sums, or with a dark region (E = 1e-170) in vacuum, wide enough for coarse cells
    that are dark too, beside regular ones."""
    d = case["desc"] = dict(case["desc"])
    s = case["state"]
    if kind == "far":
        return rescale(case, e=1.0, c=1e61)
    if kind == "long":
        d["ly"] *= 5.0
        return case
    dark = tuple(slice(n // 8, n // 8 + 3 * n // 4) for n in s.shape[1:])
    s[0][dark] = 1e-170
    for k in range(1, len(s) - 1):
        s[k][dark] = 0.0
    case["sa"][dark] = case["ss"][dark] = 0.0
    return case


@pytest.mark.parametrize("kind", ["far", "long", "dark"])
@pytest.mark.parametrize("lmax,shape,nx,ny", [(3, 0, 272, 192), (4, 1, 64, 48)])
def test_step_in_the_fallback_forms(kind, lmax, shape, nx, ny):
    """Whole 2D steps through the FP64 strips and, in the coarse levels' one launch, the FP64
    sums.  Bounds of test_step_matches_oracle."""
    case = fallback(inputs.random_admissible_2d(nx, ny, seed=9, fmax=0.99, cfl=20,
                                                bc=("reflect",) * 4, lmax=lmax), kind)
    g = O.Grid.from_case(case)
    ref, ost, ohist, _ = O.implicit_step(g, case["dt"], case["sa"], case["ss"], case["state"],
                                         O.SolveParams(lmax=lmax, tol=1e-10, cycle=shape, max_cycles=4))
    grid = m1.grid_from_case(case)
    st = grid.implicit_step(case["dt"], m1.m1_default_params(tol=1e-10, cycle=shape, max_cycles=4),
                            allow_not_converged=True)
    out = np.stack(grid.get_state())
    hist, _ = grid.step_history(st.cycles + 1)
    grid.close()
    assert (st.cycles, st.damped, st.newton_fail) == (ost["cycles"], ost["damped"], 0)
    np.testing.assert_allclose(hist, ohist, rtol=1e-9, atol=1e-13 * ohist[0])
    assert rel(out, ref, case["desc"]["c"]) <= 1e-10


@pytest.mark.parametrize("kind", ["far", "long", "dark"])
def test_step3_in_the_fallback_forms(kind):
    """Whole 3D steps: the FP64 sums in place of the blocks (far, dark), the FP64 passes (long).
    Bounds of test_step3_matches_oracle."""
    case = fallback(mixed_walls_case(), kind)
    d = case["desc"]
    g = O3.Grid3(d["nx"], d["ny"], d["nz"], d["lx"] / d["nx"], d["ly"] / d["ny"], d["lz"] / d["nz"],
                 tuple(d["bc"]), d["c"], d["a_r"], d["c_v"], None)
    ref, ost, ohist = O3.implicit_step(g, case["dt"], case["sa"], case["ss"], case["state"],
                                       O3.SolveParams3(lmax=3, tol=1e-10, max_cycles=8))
    grid = m1.grid3_from_case(case, lmax=3)
    st = grid.implicit_step(case["dt"], m1.m1_default_params(tol=1e-10, max_cycles=8),
                            allow_not_converged=True)
    out = grid.get_state()
    hist, _ = grid.step_history(st.cycles + 1)
    grid.close()
    assert (st.cycles, st.damped, st.newton_fail) == (ost["cycles"], ost["damped"], 0)
    np.testing.assert_allclose(hist, ohist, rtol=1e-8, atol=1e-12 * ohist[0])
    assert rel(out, ref, d["c"]) <= 1e-10
