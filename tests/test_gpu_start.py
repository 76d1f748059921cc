"""The local solve's warm start (csrc/rhd_start.cuh, pairs of floats) over the
range of units, optical depths and options in which it runs or gives up: the
step agrees with the oracle (same iterates, Sec. 3.3) everywhere."""
import numpy as np
import pytest

from paper_2404_08247_gb300 import inputs as I
from parity import assert_parity

pytestmark = pytest.mark.gpu

TOL = 1e-11  # the FP64 parity bound of every other field comparison


@pytest.fixture(scope="module")
def R():
    from paper_2404_08247_gb300 import rhd
    rhd.load()
    return rhd


@pytest.fixture(scope="module")
def oracle_mod():
    from oracle import oracle
    oracle.build()
    return oracle


# energy and velocity units: inside the float range, at its edge (some cells
# give up) and far outside (every cell starts from the explicit state)
@pytest.mark.parametrize("energy,speed", [(1.0, 1.0), (1e-30, 1e9), (1e36, 1.0), (1e150, 1e-3)])
@pytest.mark.parametrize("tau", [(1e-3, 1e3), (1e-10, 1e-6)])
@pytest.mark.parametrize("closure,order", [("m1", 2), ("eddington", 1)])
def test_step_in_any_units_matches_oracle(R, oracle_mod, energy, speed, tau, closure, order):
    """One 35-cell row (a ragged warp) and one 9 x 5 x 3 box, two steps: the
    state of the unit system scaled by (energy, speed) against the oracle on
    the same bytes."""
    for n in ((35,), (9, 5, 3)):
        nd = len(n)
        kw = dict(c=1e3 * speed, chat=1e2 * speed, hll_mode="none", closure=closure,
                  vc_order=order, a_rad=energy, kB_over_mu=speed ** 2)
        prob = I.base_problem(nd, n, (1.0 / n[0],) * nd, **kw)
        rho_unit = energy / speed ** 2
        base = I.base_problem(nd, n, (1.0 / n[0],) * nd, c=1e3, chat=1e2, closure=closure,
                              vc_order=order)
        U = I.random_state(base, seed=41, tau_range=tau, T_range=(1.0, 2.0))
        U[I.F_RHO] *= rho_unit
        U[I.F_KAPPA] /= rho_unit
        U[I.F_MX:I.F_MZ + 1] *= rho_unit * speed
        U[I.F_EGAS:I.F_ERAD + 1] *= energy
        U[I.F_FX:I.F_FZ + 1] *= energy * speed
        with R.RHDContext(prob, "fp64") as ctx:
            ctx.set_state(U)
            info = ctx.step(2)
            Ug = ctx.get_state()
        Uo = U.copy()
        oracle_mod.step(prob, Uo, 2)
        assert info["n_solves"] == 4 * U[0].size
        assert_parity(Ug, Uo, TOL, "units %g %g, %d-D" % (energy, speed, nd))
