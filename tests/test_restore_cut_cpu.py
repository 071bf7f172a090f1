"""The rule that cuts a restore (csrc/crac_grids.h), run on the host: coded parts of
long chunks are looked up together only where allocations are much shorter than a part."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
MIB = 1 << 20


@pytest.fixture(scope="module")
def cut(tmp_path_factory):
    d = tmp_path_factory.mktemp("cut")
    (d / "wrap.cpp").write_text("""
#include "crac_grids.h"
extern "C" uint32_t cut(uint64_t n, uint64_t b, uint32_t l, uint32_t *out) {
    const crac::RestoreCut c = crac::restore_cut(n, b, l, true, 152, ~0ull);
    out[0] = c.log2_part;
    out[1] = c.lanes;
    return c.ctas;
}
""")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2008_10596_gb300", "csrc"), str(d / "wrap.cpp"), "-o", str(d / "w.so")],
                   check=True)
    so = ctypes.CDLL(str(d / "w.so"))
    so.cut.argtypes = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_uint32, ctypes.POINTER(ctypes.c_uint32)]
    return so.cut


@pytest.mark.parametrize("n,nbytes", [(1208, 96 * MIB), (300, 20 * MIB), (20000, 400 * MIB)])
@pytest.mark.parametrize("log2S", [20, 22, 24])
def test_a_warp_a_part_of_ragged_allocations(cut, n, nbytes, log2S):
    out = (ctypes.c_uint32 * 2)()
    ctas = cut(n, nbytes, log2S, out)
    assert not out[1] and ctas == ((n << (log2S - out[0])) + 7) // 8


@pytest.mark.parametrize("n,each", [(1200, 64), (20000, 2000)])
@pytest.mark.parametrize("log2S", [20, 22, 24])
def test_short_allocations_together(cut, n, each, log2S):
    out = (ctypes.c_uint32 * 2)()
    assert cut(n, n * each, log2S, out) < (n << (log2S - out[0])) // 8 and out[1]
