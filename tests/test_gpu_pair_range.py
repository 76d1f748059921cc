"""The warm start of the local solve (csrc/rhd_start.cuh) towards the ends of its
range of units.  A change of units by powers of two (energies by 2^4j) changes
every pair by an exact factor, so where the start does not give up, its R and F
are those of the base units, scaled, to the bit, and a component that is zero
stays zero."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2404_08247_gb300 import build as B

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = r"""
#include <vector>
#include "rhd_internal.cuh"
using namespace rhd;

struct Cell {
  double rho, k0, etot, y[8], v[3];
  StartConsts K;
};

__global__ void start_kernel(const Cell* cells, int n, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const Cell& C = cells[i];
  WarmStart W;
  int nn = 0, no = 0;
  if (C.K.ok && pair_start(C.K, true, true, C.rho, C.k0, C.etot, C.y, C.v, 64, 32, W, nn, no)) {
    out[5 * i] = 1.0;
    out[5 * i + 1] = W.R;
    for (int q = 0; q < 3; ++q) out[5 * i + 2 + q] = W.F[q];
  }
}

// one cell in n unit systems: energies times 2^e[i], velocities times 2^v[i]; c
// over chat is 2^ratio; out: started, R, F of each (device, zero on entry)
extern "C" int starts(const int* e, const int* v, int n, int ratio, double* out) {
  std::vector<Cell> h(n);
  for (int i = 0; i < n; ++i) {
    const double en = ldexp(1.0, e[i]), sp = ldexp(1.0, v[i]);
    const double c = 1e3 * sp, chat = ldexp(c, -ratio), E = ldexp(3.0 * en, -ratio);
    Cell& C = h[i];
    C.rho = 1.3 * (en / sp) / sp;
    C.k0 = 0.7;
    for (double& q : C.y) q = 0.0;
    C.y[0] = 2.5 * en;
    C.y[1] = C.rho * 0.4 * sp;
    C.y[4] = E;
    C.y[5] = 0.1 * c * E;
    C.v[0] = 0.4 * sp;
    C.v[1] = C.v[2] = 0.0;
    C.etot = C.y[0] + ldexp(E, ratio);
    fill_start(C.K, c, chat, ldexp(2.0 * en, -ratio), 1.5 * sp * sp, 1e-13, 1e-13);
  }
  Cell* d = nullptr;
  if (cudaMalloc(&d, sizeof(Cell) * n) != cudaSuccess) return 1;
  cudaMemcpy(d, h.data(), sizeof(Cell) * n, cudaMemcpyHostToDevice);
  start_kernel<<<(n + 63) / 64, 64>>>(d, n, out);
  const cudaError_t err = cudaDeviceSynchronize();
  cudaFree(d);
  return (int)err;
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("start")
    src, so = d / "start.cu", d / "start.so"
    src.write_text(SRC)
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", str(src), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("ratio", [3, 100, 180, 201])
def test_a_start_is_the_base_units_start_scaled_or_none(lib, ratio):
    units = [(0, 0)] + [(e, v) for v in range(-198, 198, 6) for e in range(-640, 644, 4)
                        if abs(e - 2 * v) <= 196]
    e, v = (np.array(x, dtype=np.int32) for x in zip(*units))
    out = torch.zeros(len(units), 5, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    p = [x.ctypes.data_as(ctypes.c_void_p) for x in (e, v)]
    assert lib.starts(p[0], p[1], len(units), ratio, ctypes.c_void_p(out.data_ptr())) == 0
    out = out.cpu().numpy()
    started = out[:, 0] == 1.0
    if ratio > 200:  # c/chat beyond the range in which it runs at all
        assert not started.any()
        return
    assert started[0] and started.mean() > 0.05
    assert np.all(out[started, 3:] == 0.0)
    # (ldexp of the base: R with the energies, F with energies times velocities)
    want = np.ldexp(out[0, 1], e)
    assert np.array_equal(out[started, 1], want[started])
    want = np.ldexp(out[0, 2], e + v)
    assert np.array_equal(out[started, 2], want[started])
