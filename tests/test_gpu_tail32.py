"""The coarse end of a mixed cycle in one launch against the same levels in launches of
their own.  How much of an instance's hierarchy the one launch takes depends on the
number of instances beside it (fewer blocks each): alone, all the levels below the
finest; beside 79 others, the last or the last two.  The two evaluate the same
expressions with the same roundings, so states, cycles and residuals are equal bit for
bit."""
import numpy as np
import pytest

from paper_2208_14703_gb300 import inputs

pytestmark = pytest.mark.gpu

m1 = pytest.importorskip("paper_2208_14703_gb300.m1")


def case(kind):
    if kind == "hot":
        return inputs.hot_square_2d(256, lmax=4)
    if kind == "beam":
        return inputs.beam_channel_2d(256, lmax=4)
    if kind == "random":
        return inputs.random_admissible_2d(208, 176, seed=5, fmax=0.9, cfl=30,
                                           bc=("reflect",) * 4, lmax=4)
    if kind == "periodic":
        return inputs.random_admissible_2d(96, 256, seed=6, fmax=0.9, cfl=30,
                                           bc=("periodic",) * 4, lmax=4)
    return inputs.gaussian_1d(4096, lmax=4)


@pytest.mark.parametrize("kind", ["hot", "beam", "random", "periodic", "1d"])
@pytest.mark.parametrize("cycle", [0, 1])
def test_one_launch_equals_levels(kind, cycle):
    c = case(kind)
    params = m1.m1_default_params(tol=1e-8, cycle=cycle, max_cycles=8)
    g = m1.grid_from_case(c, precision=1)
    st = g.implicit_step(c["dt"], params, allow_not_converged=True)
    alone = np.stack(g.get_state())
    g.close()
    assert np.isfinite(alone).all()
    filler = inputs.hot_square_2d(16, lmax=4)
    cases = [c] + [filler] * 79
    b = m1.batch_from_cases(cases, precision=1)
    stats = b.implicit_step([x["dt"] for x in cases], params, allow_not_converged=True)
    beside = np.stack(b.get_state(0))
    b.close()
    assert (st.cycles, st.res) == (stats[0].cycles, stats[0].res)
    np.testing.assert_array_equal(alone, beside)


@pytest.fixture
def staging(request):
    """Both row stagings of the strips, for every size of level."""
    m1.set_tuning([{"kind": 1, "n": 1 << c, "strip_rows": 4, "staging": request.param}
                   for c in range(16)])
    yield request.param
    m1.set_tuning([{"kind": 1, "n": 1 << c, "strip_rows": 0, "staging": 0} for c in range(16)])


def general_case(dim):
    """No constant equal to one, unequal cell sides, walls of every kind, fluxes at the
    cone: a product, fusion or association that differs shows."""
    bc = ("reflect", "neumann", "inflow", "inflow") if dim == 2 else ("inflow", "neumann", "periodic",
                                                                      "periodic")
    c = inputs.random_admissible_2d(208 if dim == 2 else 4096, 176, seed=8, fmax=0.99, cfl=20, bc=bc,
                                    lmax=4, dim=dim)
    d = c["desc"] = dict(c["desc"])
    d.update(c=3.7, a_r=0.83, c_v=1.9)
    if dim == 2:
        d["ly"] *= 1.7
    c["state"] = c["state"].copy()
    c["state"][1:3] *= d["c"]
    c["inflow"][:, 1:] *= d["c"]
    c["inflow"][:, 2] = 0.3 * d["c"] if dim == 2 else 0.0
    return c


@pytest.mark.parametrize("staging", [0, 1], indirect=True)
@pytest.mark.parametrize("dim", [2, 1])
@pytest.mark.parametrize("cycle,dtau0", [(0, 1e-3), (2, 1.0)])
def test_one_launch_equals_levels_with_general_constants(staging, dim, cycle, dtau0):
    c = general_case(dim)
    params = m1.m1_default_params(tol=1e-8, cycle=cycle, max_cycles=8, dtau0=dtau0)
    g = m1.grid_from_case(c, precision=1)
    st = g.implicit_step(c["dt"], params, allow_not_converged=True)
    alone = np.stack(g.get_state())
    g.close()
    assert np.isfinite(alone).all()
    # beside 79 others whose rows are staged alike (1D rows are not staged by cp.async but
    # beside larger 2D instances that are, where they agree to rounding: test_tuning.py)
    filler = inputs.hot_square_2d(16, lmax=4) if dim == 2 else inputs.gaussian_1d(64, lmax=4)
    cases = [c] + [filler] * 79
    b = m1.batch_from_cases(cases, precision=1)
    stats = b.implicit_step([x["dt"] for x in cases], params, allow_not_converged=True)
    beside = np.stack(b.get_state(0))
    b.close()
    assert (st.cycles, st.res) == (stats[0].cycles, stats[0].res)
    np.testing.assert_array_equal(alone, beside)
