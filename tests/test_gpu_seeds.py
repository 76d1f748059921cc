"""Reciprocals and roots from integer-built seeds (csrc/rhd_internal.cuh): they
take the squares of E through the double range, so the step is compared with the
oracle where those squares, or those of F = c E, are near an end of the range
(2^-1019 to 2^1017) and far outside single precision's."""
import pytest

from paper_2404_08247_gb300 import inputs as I
from parity import assert_parity

TOL = 1e-11  # the FP64 parity bound of every other field comparison


def row(energy, n=35):
    prob = I.base_problem(1, (n,), (1.0 / n,), c=1e3, chat=1e2, hll_mode="none", a_rad=energy)
    base = I.base_problem(1, (n,), (1.0 / n,), c=1e3, chat=1e2)
    U = I.random_state(base, seed=43, tau_range=(1e-3, 1e2), T_range=(1.0, 2.0))
    U[I.F_RHO] *= energy
    U[I.F_KAPPA] /= energy
    U[I.F_MX:I.F_FZ + 1] *= energy
    return prob, U


@pytest.mark.gpu
@pytest.mark.parametrize("energy", [5e-154, 1e-152, 1e-60, 1e60, 1e148, 1e149])
def test_squares_near_the_ends_of_the_double_range(energy):
    from oracle import oracle
    from paper_2404_08247_gb300 import rhd
    oracle.build()
    prob, U = row(energy)
    with rhd.RHDContext(prob, "fp64") as ctx:
        ctx.set_state(U)
        ctx.step(2)
        Ug = ctx.get_state()
    Uo = U.copy()
    oracle.step(prob, Uo, 2)
    assert_parity(Ug, Uo, TOL, "energy unit %g" % energy)
