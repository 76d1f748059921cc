"""Halves and quarters formed on the integer pipe (csrc/rhd_internal.cuh) are the
products' bits over the whole double range, subnormal results rounded to even:
the CPU compiles the same functions, the GPU steps fields that small."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2404_08247_gb300 import build as B
from paper_2404_08247_gb300 import inputs as I

SRC = r"""
#include "rhd_internal.cuh"
extern "C" void mags(const long long* a, int n, long long* half, long long* quarter) {
  for (int i = 0; i < n; ++i) {
    half[i] = rhd::half_mag(a[i]);
    quarter[i] = rhd::quarter_mag(a[i]);
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("mags")
    src, so = d / "mags.cu", d / "mags.so"
    src.write_text(SRC)
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", str(src), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(so))


def test_halves_and_quarters_are_the_products_bits(lib):
    rng = np.random.default_rng(0)
    edges = [b + d for e in (0, 1, 2, 3, 4, 2046) for b in (e << 52,) for d in range(-9, 10)]
    a = np.concatenate([np.arange(64), rng.integers(0, 6 << 52, 200000),
                        rng.integers(0, 0x7ff << 52, 200000), [0x7ff << 52], edges])
    a = a[(a >= 0) & (a <= 0x7ff << 52)].astype(np.int64)
    half, quarter = np.empty_like(a), np.empty_like(a)
    p = [x.ctypes.data_as(ctypes.c_void_p) for x in (a, half, quarter)]
    lib.mags(p[0], ctypes.c_int(a.size), p[1], p[2])
    x = a.view(np.float64)
    assert np.array_equal(half, (0.5 * x).view(np.int64))
    assert np.array_equal(quarter, (0.25 * x).view(np.int64))


@pytest.mark.gpu
@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("size", [1e-300, 1e-307, 3e-308, 1e-310, 5e-324])
def test_tiny_momenta_without_opacity_are_kept(size, prec):
    """Without opacity a step leaves the gas alone: (y + y)/2 is y."""
    from paper_2404_08247_gb300 import rhd
    prob = I.base_problem(1, (35,), (1 / 35,), c=1e3, chat=1e2)
    U = I.random_state(prob, seed=3)
    U[I.F_KAPPA] = 0.0
    u = np.random.default_rng(0).uniform(-1.0, 1.0, U[I.F_MX:I.F_MZ + 1].shape)
    U[I.F_MX:I.F_MZ + 1] = size * u if size > 1e-320 else np.sign(u) * size
    with rhd.RHDContext(prob, prec) as ctx:
        ctx.set_state(U)
        ctx.step(2)
        V = ctx.get_state()
    assert np.array_equal(V[I.F_MX:I.F_EGAS + 1], U[I.F_MX:I.F_EGAS + 1])


@pytest.mark.gpu
@pytest.mark.parametrize("recon", ["plm", "ppm"])
@pytest.mark.parametrize("n", [(35,), (17, 9, 7)], ids=["1d", "3d"])
def test_fluxes_below_the_normal_range_are_reconstructed(n, recon):
    """F/c near 1e-310, whose half slopes and interface values are subnormal
    (units of 5e-324, 5e-14 of the field).  Beside a uniform E = 1 the transport
    of so small a flux is linear in it, so the step is that of the flux times
    2^690, scaled back.  (The oracle's PPM limiter multiplies differences, which
    underflow here.)"""
    from paper_2404_08247_gb300 import rhd
    nd = len(n)
    prob = I.base_problem(nd, n, (1.0 / n[0],) * nd, c=1e3, chat=1e2, hll_mode="none",
                          reconstruction=recon, cfl=0.3)
    U = I.random_state(prob, seed=4)
    U[I.F_KAPPA] = 0.0
    U[I.F_ERAD] = 1.0
    F = slice(I.F_FX, I.F_FZ + 1)
    flux = 1e-307 * np.random.default_rng(1).uniform(-1.0, 1.0, U[F].shape)
    out = []
    for scale in (1.0, 2.0 ** 690):
        U[F] = flux * scale
        with rhd.RHDContext(prob) as ctx:
            ctx.set_state(U)
            ctx.step(1)
            out.append(ctx.get_state()[F] / scale)
    err = np.max(np.abs(out[0] - out[1])) / np.max(np.abs(out[1]))
    assert err <= 1e-11, err
