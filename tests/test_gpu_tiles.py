"""Grids at the edges of the tiles the stage launches choose among (256- and
32-cell rows, 32 x 8 and 16 x 4 planes, 1 to 16 planes a block): partial
tiles, single rows and planes, one cell more and less than whole tiles."""
import numpy as np
import pytest

from paper_2404_08247_gb300 import inputs as I
from parity import assert_parity

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-11, "mixed": 1e-5}  # the parity bounds of the two precisions


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


SHAPES = [(31,), (33,), (257,), (16, 4), (17, 5), (33, 9), (300, 3), (16, 4, 3), (17, 5, 4),
          (15, 3, 17), (33, 9, 5), (64, 33, 19)]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("recon", ["plm", "ppm"])
@pytest.mark.parametrize("n", SHAPES, ids=lambda n: "x".join(map(str, n)))
def test_tile_edges_match_oracle(R, oracle_mod, n, recon, prec):
    nd = len(n)
    prob = I.base_problem(nd, n, (1.0 / n[0],) * nd, c=1e3, chat=1e2, reconstruction=recon,
                          cfl=0.3, bc="reflect" if nd == 2 else "periodic")
    U = I.random_state(prob, seed=5, T_range=(1.0, 2.0))
    with R.RHDContext(prob, prec) as ctx:
        ctx.set_state(U)
        ctx.step(1)
        Ug = ctx.get_state()
    Uo = U.copy()
    oracle_mod.step(prob, Uo, 1)
    assert_parity(Ug, Uo, TOL[prec], "%s %s %s" % (n, recon, prec))


@pytest.mark.parametrize("recon", ["plm", "ppm"])
def test_rows_stepped_by_parts_equal_the_whole(R, recon):
    """rhd_step_host launches ranges of rows; the tiles are the whole grid's,
    so that the bits are those of rhd_step (3-D, ragged in every axis)."""
    n = (35, 18, 41)
    prob = I.base_problem(3, n, (1.0 / 35,) * 3, c=1e3, chat=1e2, reconstruction=recon, cfl=0.3)
    U = I.random_state(prob, seed=6, T_range=(1.0, 2.0))
    with R.RHDContext(prob) as a, R.RHDContext(prob) as b:
        a.set_state(U)
        a.step(2)
        out = b.step_host(U.copy(), nsteps=2)["out"]
        assert np.array_equal(a.get_state(), out)
