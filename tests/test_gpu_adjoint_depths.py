"""The adjoint of the local solve at optical depths far beyond any in use: past
1e60 a cell keeps nothing but its totals, the derivative no longer depends on
the depth, and it does not overflow (k = chat chi dt enters a determinant as
k^2)."""
import numpy as np
import pytest

from paper_2404_08247_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def gradient(depth, closure):
    from paper_2404_08247_gb300 import rhd
    n = 64
    prob = I.base_problem(1, (n,), (1 / n,), c=1e3, chat=1e2, hll_mode="none", closure=closure)
    U = I.random_state(prob, 3)
    U[I.F_KAPPA] *= depth
    with rhd.RHDContext(prob) as ctx:
        ctx.set_stream(torch.cuda.current_stream())
        ctx.set_state(U)
        tape = torch.zeros(3 * 8 * n, dtype=torch.float64, device="cuda")
        ybar = torch.ones(8 * n, dtype=torch.float64, device="cuda")
        kbar = torch.zeros(n, dtype=torch.float64, device="cuda")
        ctx.step_record(1, 0.0, tape)
        ctx.adjoint(tape, 1, 0.0, ybar, kbar)
        assert torch.isfinite(kbar).all()
        return ybar.cpu().numpy().reshape(8, n)


@pytest.mark.parametrize("closure", ["m1", "eddington"])
@pytest.mark.parametrize("depth", [1e140, 1e152, 1e160, 1e200, 1e280])
def test_gradient_past_any_depth_is_that_of_a_deep_cell(depth, closure):
    want, got = gradient(1e100, closure), gradient(depth, closure)
    for q in range(8):
        assert np.max(np.abs(got[q] - want[q])) <= 1e-10 * np.max(np.abs(want[q])), q
