"""Radiation energies whose square is below the double range (E < 1e-162): the M1
closure cannot be formed from E^2 and |F|^2, and the step is refused as
nonphysical, the state left as it was, rather than taken with a pressure of
-E/3."""
import numpy as np
import pytest

from paper_2404_08247_gb300 import inputs as I

pytestmark = pytest.mark.gpu


def row(energy, speed=1e3):
    prob = I.base_problem(1, (35,), (1 / 35,), c=1e3 * speed, chat=1e2 * speed, hll_mode="none",
                          a_rad=energy, kB_over_mu=speed ** 2)
    base = I.base_problem(1, (35,), (1 / 35,), c=1e3, chat=1e2)
    U = I.random_state(base, 41, tau_range=(1e-3, 1e3), T_range=(1.0, 2.0))
    rho = energy / speed ** 2
    U[I.F_RHO] *= rho
    U[I.F_KAPPA] /= rho
    U[I.F_MX:I.F_MZ + 1] *= rho * speed
    U[I.F_EGAS:I.F_ERAD + 1] *= energy
    U[I.F_FX:I.F_FZ + 1] *= energy * speed
    return prob, U


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("energy", [1e-165, 1e-200, 1e-250])
def test_steps_whose_energy_squares_vanish_are_refused(energy, prec):
    from paper_2404_08247_gb300 import rhd
    prob, U = row(energy)
    with rhd.RHDContext(prob, prec) as ctx:
        ctx.set_state(U)
        info = ctx.step(2, raise_on_error=False)
        assert info["status"] == rhd.RHD_ERR_NONPHYSICAL
        assert info["steps_done"] == 0
        assert np.array_equal(ctx.get_state(), U)
