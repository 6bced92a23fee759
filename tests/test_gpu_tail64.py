"""The coarse end of an FP64 cycle in one launch per cluster size (csrc/m1_tail.cu).  The
cluster an instance gets shrinks with the number of instances beside it, as far as it holds
the instance's levels; those of several sizes run side by side.  No result depends on it:
states, cycles and residuals equal those of the instance alone bit for bit."""
import numpy as np
import pytest

from paper_2208_14703_gb300 import inputs

pytestmark = pytest.mark.gpu

m1 = pytest.importorskip("paper_2208_14703_gb300.m1")


def cases():
    """Tails that need 16, 16, 8, 4, 2, 1 and 1 blocks (first levels of 8192, which fill the
    shared memory, 4160, 4096, 2288, 1024, 2048 and 64)."""
    return [inputs.random_admissible_2d(512, 256, seed=7, fmax=0.9, cfl=30, bc=("neumann",) * 4, lmax=5),
            inputs.random_admissible_2d(320, 208, seed=4, fmax=0.9, cfl=30, bc=("periodic",) * 4, lmax=5),
            inputs.hot_square_2d(256, lmax=5),
            inputs.random_admissible_2d(208, 176, seed=5, fmax=0.9, cfl=30, bc=("reflect",) * 4, lmax=5),
            inputs.beam_channel_2d(64, lmax=5),
            inputs.gaussian_1d(4096, lmax=5),
            inputs.hot_square_2d(16, lmax=5)]


@pytest.mark.parametrize("count", [9, 12, 24, 48, 90])
@pytest.mark.parametrize("cycle", [0, 1, 2])
def test_results_do_not_depend_on_the_cluster(count, cycle):
    some = cases()
    params = m1.m1_default_params(tol=1e-8, cycle=cycle, max_cycles=4)
    batch = some + [some[-1]] * (count - len(some))
    b = m1.batch_from_cases(batch)
    stats = b.implicit_step([x["dt"] for x in batch], params, allow_not_converged=True)
    for k, c in enumerate(some):
        g = m1.grid_from_case(c)
        st = g.implicit_step(c["dt"], params, allow_not_converged=True)
        alone = np.stack(g.get_state())
        g.close()
        assert np.isfinite(alone).all()
        assert (st.cycles, st.res, st.damped) == (stats[k].cycles, stats[k].res, stats[k].damped), k
        np.testing.assert_array_equal(alone, np.stack(b.get_state(k)), err_msg=str(k))
    b.close()
