"""The planes that the blocks of a 3-D stage launch march through, from the
launch code itself (csrc/rhd_stage.cuh compiled into a small host library; no
kernel runs): every launch over part of a grid, as rhd_step_host cuts it,
covers exactly its own planes, once each.  A block that ran on into the next
part would read optical-depth factors this launch has not waited for and write
cells that another stream's launch owns."""
import ctypes
import subprocess

import pytest

from paper_2404_08247_gb300 import build as B
from paper_2404_08247_gb300 import inputs as I

SRC = r"""
#include "rhd_stage.cuh"
// planes of the blocks over [lo, hi) as pairs in out; returns their number
extern "C" int blocks(const int* n, int mixed, int ppm, int rates, int lo, int hi, int* out,
                      int* lz) {
  rhd::Geometry g = {};
  g.ndim = 3;
  for (int d = 0; d < 3; ++d) g.n[d] = n[d];
  const rhd::TilePlan P = rhd::plan_tiles(g, mixed != 0, ppm != 0, rates == 0);
  *lz = P.lz;
  const int nb = (hi - lo + P.lz - 1) / P.lz;
  for (int b = 0; b < nb; ++b) rhd::block_planes(b, lo, hi, P.lz, out[2 * b], out[2 * b + 1]);
  return nb;
}
"""

SHAPES = [(9, 7, 5), (40, 24, 70), (35, 18, 41), (256, 256, 256), (64, 48, 355), (64, 64, 288),
          (160, 128, 384), (128, 128, 300), (288, 288, 288), (384, 384, 384), (400, 400, 400),
          (64, 64, 1000)]


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("parts")
    src, so = d / "parts.cu", d / "parts.so"
    src.write_text(SRC)
    r = subprocess.run([B.nvcc(), *B.ARCH, *B.FLAGS, "-shared", str(src), "-o", str(so)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("recon", ["plm", "ppm"])
@pytest.mark.parametrize("n", SHAPES, ids=lambda n: "x".join(map(str, n)))
def test_blocks_of_each_part_cover_exactly_its_planes(lib, n, recon, prec):
    B.build()
    from paper_2404_08247_gb300 import rhd
    plan = rhd.host_step_plan(I.base_problem(3, n, [1.0 / v for v in n], reconstruction=recon))
    cuts = [min(n[2], 8 * r) for r in plan["rows"]]
    parts = [(0, n[2])] + [(cuts[a], cuts[b]) for a, b in plan["stage1"] + plan["stage2"]]
    out, lz = (ctypes.c_int * (2 * n[2]))(), ctypes.c_int()
    size = (ctypes.c_int * 3)(*n)
    for lo, hi in parts:
        nb = lib.blocks(size, prec == "mixed", recon == "ppm", 0, lo, hi, out, ctypes.byref(lz))
        planes = [k for b in range(nb) for k in range(out[2 * b], out[2 * b + 1])]
        assert planes == list(range(lo, hi)), (lo, hi, lz.value)


def test_some_parts_hold_an_odd_number_of_rows_for_16_planes_a_block(lib):
    """The shapes above reach the case: 16 planes a block, a part of an odd
    number of 8-plane rows."""
    from paper_2404_08247_gb300 import rhd
    lz, out = ctypes.c_int(), (ctypes.c_int * 2000)()
    odd = set()
    for n in SHAPES:
        plan = rhd.host_step_plan(I.base_problem(3, n, [1.0 / v for v in n]))
        lib.blocks((ctypes.c_int * 3)(*n), 0, 0, 0, 0, n[2], out, ctypes.byref(lz))
        for k, groups in ((1, plan["stage1"]), (2, plan["stage2"])):
            if lz.value == 16 and any((plan["rows"][b] - plan["rows"][a]) % 2 and
                                      8 * plan["rows"][b] < n[2] for a, b in groups):
                odd.add((n, k))
    assert {k for _, k in odd} == {1, 2}, odd
    assert ((64, 48, 355), 1) in odd, odd
