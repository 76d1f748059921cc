"""Half slopes, interface values and halves formed the short way on the integer pipe
(csrc/rhd_internal.cuh), with the exact way where a result is rare, are the bits
of the plain products over the double range: fields of every size, subnormal and
near overflow, zeros, equal neighbours and infinite sums."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2404_08247_gb300 import build as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = r"""
#include "rhd_internal.cuh"
using namespace rhd;
__device__ double plain_slope(double um, double u0, double up) {
  const double dm = u0 - um, dp = up - u0;
  const double m = fmin(fmin(fabs(dm), fabs(dp)), __dmul_rn(0.25, fabs(dm + dp)));
  return (dm > 0.0 && dp > 0.0) ? m : (dm < 0.0 && dp < 0.0) ? -m : 0.0;
}
// u: 4 cells of 4 fields each thread; out: 4 slopes, 4 interface values, 4 halves,
// then the same by plain products
__global__ void limiter_kernel(const double* u, int n, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  double c[4][4], h[4], a[4];
  for (int o = 0; o < 4; ++o)
    for (int q = 0; q < 4; ++q) c[o][q] = u[(o * 4 + q) * n + i];
  half_slopes(c[0], c[1], c[2], h);
  ppm_interfaces<true>(c[0], c[1], c[2], c[3], a);
  for (int q = 0; q < 4; ++q) {
    const double s = __dadd_rn(c[1][q], c[2][q]), half = __dmul_rn(0.5, s);
    bool rare = false;
    const double f = half_fast(s, rare);
    out[q * n + i] = h[q];
    out[(4 + q) * n + i] = a[q];
    out[(8 + q) * n + i] = rare ? half_of(s) : f;
    const double h0 = plain_slope(c[0][q], c[1][q], c[2][q]);
    const double h1 = plain_slope(c[1][q], c[2][q], c[3][q]);
    out[(12 + q) * n + i] = h0;
    out[(16 + q) * n + i] = fma(__dadd_rn(h0, -h1), 1.0 / 3.0, half);
    out[(20 + q) * n + i] = half;
  }
}
extern "C" int limiter(const double* u, int n, double* out) {
  limiter_kernel<<<(n + 127) / 128, 128>>>(u, n, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("limiter")
    src, so = d / "limiter.cu", d / "limiter.so"
    src.write_text(SRC)
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", str(src), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("lo,hi", [(-1074, -1060), (-1040, -1000), (-1030, -1010), (-60, 60),
                                   (-1074, 1023), (1015, 1023), (1021, 1023)])
def test_bits_of_the_plain_products(lib, lo, hi):
    rng = np.random.default_rng(lo + 4000 + hi)
    n = 20000
    u = np.ldexp(rng.uniform(-1.0, 1.0, (4, 4, n)), rng.integers(lo, hi + 1, (4, 4, n)))
    u[:, 0] = np.sort(u[:, 0], axis=0)  # a monotone field
    u[:, 1, ::3] = 0.0
    u[1:, 2, ::5] = u[:1, 2, ::5]  # equal neighbours
    u[:, 3, ::2] = np.ldexp(rng.integers(-5, 6, (4, n // 2)).astype(float), max(lo, -1074))
    ud = torch.from_numpy(u).cuda()
    out = torch.empty(24 * n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.limiter(ctypes.c_void_p(ud.data_ptr()), ctypes.c_int(n),
                       ctypes.c_void_p(out.data_ptr())) == 0
    got, want = out.cpu().numpy().reshape(2, 12 * n)
    same = (got.view(np.int64) == want.view(np.int64)) | (np.isnan(got) & np.isnan(want))
    zero = (got == 0.0) & (want == 0.0)  # a zero's sign is free
    assert np.all(same | zero), (got[~(same | zero)][:4], want[~(same | zero)][:4])
