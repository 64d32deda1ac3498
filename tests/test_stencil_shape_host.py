"""The launch-shape rule of the level-0 stencil passes (host arithmetic, compiled here with the host
compiler): a shape that a caller sets is launched as it stands at every size; only the default is
fitted to a small operator, and the launch always covers every chunk."""
import ctypes as C
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SMS = 152
UNITS = [1, 2, 7, 63, 64, 65, 151, 304, 607, 608, 609, 1215, 1216, 1217, 5000,
         8 * 64 * SMS - 1, 8 * 64 * SMS, 8 * 64 * SMS + 1, 220_000, 60_000_000]

SHIM = """
#include "stencil_shape.cuh"
extern "C" void shape(int k, int packed, int block, int per_sm, int fit, long long units, int sms,
                      int* out) {
  const saamg::StencilLaunch l =
      saamg::stencil_launch(saamg::StencilCfg{k, packed, block, per_sm, fit != 0}, units, sms);
  out[0] = l.k;
  out[1] = l.block;
  out[2] = l.blocks;
}
"""


@pytest.fixture(scope="module")
def launch(tmp_path_factory):
    d = tmp_path_factory.mktemp("shape")
    (d / "shim.cpp").write_text(SHIM)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_0907_4863_gb300", "csrc"), str(d / "shim.cpp"), "-o",
                    str(d / "shim.so")], check=True)
    f = C.CDLL(str(d / "shim.so")).shape

    def call(k, packed, block, per_sm, fit, units):
        out = (C.c_int * 3)()
        f(k, packed, block, per_sm, fit, C.c_longlong(units), SMS, out)
        return tuple(out)
    return call


@pytest.mark.parametrize("units", UNITS)
def test_a_set_shape_is_launched_as_it_stands(launch, units):
    for k in (1, 2, 4):
        for packed in (0, 1):
            for block in (128, 256):
                for per_sm in (8, 16, 32):
                    need = -(-units // (block // 32 * k))
                    assert launch(k, packed, block, per_sm, 0, units) == \
                        (k, block, min(need, SMS * per_sm))


@pytest.mark.parametrize("units", UNITS)
def test_the_default_is_fitted_to_a_small_operator(launch, units):
    k, block, blocks = launch(2, 1, 256, 32, 1, units)
    assert k == (1 if units < 8 * 64 * SMS else 2)
    assert block in (64, 128, 256) and (block == 64 or units * 32 >= SMS * block)
    assert block == 256 or units * 32 < SMS * 2 * block
    assert blocks == min(-(-units // (block // 32 * k)), SMS * 32)
