"""The FP64 kernels' reciprocals, roots (one Newton step from a seed of 2^-44) and
whole powers of the temperature (csrc/rhd_internal.cuh) against exact rational
arithmetic: within 1 ulp for mantissas at random and beside powers of two,
exponents odd and even, and at the ends of the seeds' range, beyond which IEEE
operations run."""
import ctypes
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_2404_08247_gb300 import build as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = r"""
#include "rhd_internal.cuh"
__global__ void arith_kernel(const double* x, int n, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = rhd::rcp_pos(x[i]);
  out[n + i] = rhd::rsqrt_pos(x[i]);
  out[2 * n + i] = rhd::sqrt_pos(x[i]);
}
__global__ void power_kernel(const double* x, int n, int p, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  rhd::Physics ph = {};
  ph.kappa_T_int = p;
  ph.kappa_T_exp = p;
  out[i] = rhd::opacity_power(ph, x[i]);
}
extern "C" int arith(const double* x, int n, double* out) {
  arith_kernel<<<(n + 255) / 256, 256>>>(x, n, out);
  return (int)cudaDeviceSynchronize();
}
extern "C" int power(const double* x, int n, int p, double* out) {
  power_kernel<<<(n + 255) / 256, 256>>>(x, n, p, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("arith")
    src, so = d / "arith.cu", d / "arith.so"
    src.write_text(SRC)
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", str(src), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(so))


def mantissas(rng, n):
    """In [1, 2): at random, and the 64 values above 1 and below 2."""
    k = np.arange(64) * 2.0 ** -52
    return np.concatenate([1.0 + rng.random(n), 1.0 + k, 2.0 - 2.0 ** -52 - k])


@pytest.mark.parametrize("lo,hi", [(-1022, -1010), (-1010, -900), (-130, 130), (900, 1010),
                                   (1010, 1021)])
def test_reciprocals_and_roots_within_one_ulp(lib, lo, hi):
    rng = np.random.default_rng(lo + 2000)
    m = mantissas(rng, 3000)
    e = rng.integers(lo, hi + 1, m.size)
    e[-128:] = np.tile([lo, lo + 1], 64)  # odd and even beside the powers of two
    x = np.ldexp(m, e)
    xd = torch.from_numpy(x).cuda()
    out = torch.empty(3 * x.size, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    p = [ctypes.c_void_p(v.data_ptr()) for v in (xd, out)]
    assert lib.arith(p[0], ctypes.c_int(x.size), p[1]) == 0
    r, q, s = out.cpu().numpy().reshape(3, -1)
    # the exact value lies within one ulp (of the IEEE result) of each result
    for v, got, ulp in zip(x, r, np.spacing(1.0 / x)):
        v, got, ulp = Fraction(v), Fraction(got), Fraction(ulp)
        assert (got - ulp) * v <= 1 <= (got + ulp) * v, ("1/x", float(v))
    for v, got, ulp in zip(x, s, np.spacing(np.sqrt(x))):
        v, got, ulp = Fraction(v), Fraction(got), Fraction(ulp)
        assert (got - ulp) ** 2 <= v <= (got + ulp) ** 2, ("sqrt", float(v))
    # (outside the seeds' range 1/sqrt is two IEEE operations, each within 2^-53 of
    # its result: 2^-52 together, two ulps)
    seeded = (x >= 2.0 ** -1018) & (x < 2.0 ** 1017)
    for v, got, ulp in zip(x, q, np.spacing(1.0 / np.sqrt(x)) * np.where(seeded, 1.0, 2.0)):
        v, got, ulp = Fraction(v), Fraction(got), Fraction(ulp)
        assert (got - ulp) ** 2 * v <= 1 <= (got + ulp) ** 2 * v, ("1/sqrt", float(v))


@pytest.mark.parametrize("p", [-8, -7, -3, -2, -1, 1, 2, 3, 5, 8])
def test_whole_powers_within_one_ulp(lib, p):
    """Against exact rational arithmetic, over 1e-4 to 1e4."""
    rng = np.random.default_rng(p + 50)
    x = np.concatenate([10.0 ** rng.uniform(-4, 4, 1500), mantissas(rng, 200)])
    xd = torch.from_numpy(x).cuda()
    out = torch.empty_like(xd)
    torch.cuda.synchronize()
    assert lib.power(ctypes.c_void_p(xd.data_ptr()), ctypes.c_int(x.size), ctypes.c_int(p),
                     ctypes.c_void_p(out.data_ptr())) == 0
    got = out.cpu().numpy()
    worst = 0.0
    for v, g in zip(x, got):
        want = Fraction(float(v)) ** p
        ulp = Fraction(float(np.spacing(float(want))))
        worst = max(worst, float(abs(Fraction(float(g)) - want) / ulp))
    assert worst <= 1.0, worst
