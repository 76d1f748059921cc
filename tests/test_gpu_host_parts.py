"""rhd_step_host on grids whose stage launches march 16 planes a block while a
part holds an odd number of 8-plane rows: the same bits and the same step info
(the solves counted once) as set + step + get."""
import numpy as np
import pytest

from test_gpu_host_step import R, check_same, problem  # noqa: F401

pytestmark = pytest.mark.gpu

# Grids with 16 planes a block and parts of an odd number of 8-plane rows: FP64
# 64 x 48 x 355 (stage 1: planes [16, 88); last stage 2: [112, 200), [200, 288)),
# mixed 64 x 64 x 288 (stage 1: [16, 72); last stage 2: [16, 88), [88, 160), ..)
N64, N32 = (64, 48, 355), (64, 64, 288)
CASES = {"periodic_tau": (N64, {}, 1, "fp64"), "two_steps": (N64, {}, 2, "fp64"),
         "reflect": (N64, {"bc": "reflect"}, 1, "fp64"),
         "no_tau": (N64, {"hll_mode": "none"}, 1, "fp64"), "mixed": (N32, {}, 1, "mixed"),
         "ppm": (N64, {"reconstruction": "ppm", "cfl": 0.3}, 1, "fp64")}


@pytest.mark.parametrize("name", sorted(CASES))
def test_tall_host_steps_equal_set_step_get(R, name):  # noqa: F811
    n, kw, nsteps, prec = CASES[name]
    prob, U = problem(3, n, 930, **kw)
    _, info = check_same(R, prob, U, nsteps, prec)
    assert info["status"] == R.RHD_OK
    assert info["n_solves"] == 2 * nsteps * U[0].size


def test_the_first_call_of_a_context_with_other_factors_before(R):  # noqa: F811
    """A context that has stepped another material: its optical-depth factors
    are rewritten part by part, and no part reads the old ones."""
    prob, U = problem(3, N64, 931)
    V = U.copy()
    V[9] *= 1e3
    with R.RHDContext(prob) as a, R.RHDContext(prob) as b:
        a.step_host(V, None, 1)
        out = a.step_host(U.copy(), None, 1)["out"]
        b.set_state(U)
        b.step(1)
        assert np.array_equal(out, b.get_state())
