"""The rules that cut a pass into segments, grids and work per warp
(csrc/crac_grids.h), compiled and run on the host: every byte is some warp's, and
the chip is not left idle by allocations much shorter than a chunk."""
import ctypes
import os
import random
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SM = 152

WRAP = """
#include "crac_grids.h"
using namespace crac;
extern "C" {
uint32_t hash_seg(uint64_t n, uint64_t b, uint32_t l, int copy) { return split_hash_seg(n, b, l, copy); }
uint32_t hash_grid(uint64_t n, uint64_t b, uint32_t l, uint32_t s, int copy, int sm, uint32_t *per) {
    return split_hash_grid(n, b, l, s, copy, sm, per);
}
int dense(float f, uint32_t l) { return dense_by_cta(f, l); }
uint32_t restore_plan(uint64_t n, uint64_t b, uint32_t l, int coded, int sm, uint64_t most, uint32_t *out) {
    const RestoreCut c = restore_cut(n, b, l, coded, sm, most);
    out[0] = c.log2_part;
    out[1] = c.lanes;
    return c.ctas;
}
}
"""


@pytest.fixture(scope="module")
def rules(tmp_path_factory):
    d = tmp_path_factory.mktemp("grids")
    (d / "wrap.cpp").write_text(WRAP)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2008_10596_gb300", "csrc"), str(d / "wrap.cpp"), "-o", str(d / "w.so")],
                   check=True)
    so = ctypes.CDLL(str(d / "w.so"))
    u64, u32 = ctypes.c_uint64, ctypes.c_uint32
    so.hash_seg.argtypes = [u64, u64, u32, ctypes.c_int]
    so.hash_grid.argtypes = [u64, u64, u32, u32, ctypes.c_int, ctypes.c_int, ctypes.POINTER(u32)]
    so.dense.argtypes = [ctypes.c_float, u32]
    so.restore_plan.argtypes = [u64, u64, u32, ctypes.c_int, ctypes.c_int, u64, ctypes.POINTER(u32)]
    return so


def hash_plan(so, n, nbytes, log2S, copy, sm=SM):
    seg = so.hash_seg(n, nbytes, log2S, copy)
    per = ctypes.c_uint32()
    return seg, so.hash_grid(n, nbytes, log2S, seg, copy, sm, ctypes.byref(per)), per.value


@pytest.mark.parametrize("copy", [0, 1])
@pytest.mark.parametrize("log2S", range(13, 25))
def test_full_chunks_one_segment_a_warp(rules, log2S, copy):
    """4 GiB of full chunks: a warp a segment of 8 KiB, or of 16 where the pass reads or
    few chunks take all sums, whatever the chunk."""
    n = (4 << 30) >> log2S
    seg, grid, per = hash_plan(rules, n, 4 << 30, log2S, copy)
    assert seg == min(log2S, 13 if copy and log2S < 21 else 14) and per == 1 and grid == ((n << (log2S - seg)) + 7) // 8


@pytest.mark.parametrize("copy", [0, 1])
@pytest.mark.parametrize("log2S", [4, 6, 8, 13, 14, 16, 18, 20, 24])
@pytest.mark.parametrize("n,each", [(1200, 5), (1200, 64), (1200, 4096), (20000, 2000), (50000, 200), (1 << 20, 16)])
def test_short_allocations_keep_the_chip_busy(rules, n, each, log2S, copy):
    """n allocations of `each` bytes, one chunk each: work for every SM, if there
    are chunks for it."""
    each = min(each, 1 << log2S)
    seg, grid, per = hash_plan(rules, n, n * each, log2S, copy)
    assert grid >= min(4 * SM, (n + 7) // 8)
    assert per <= max(1, (n << (log2S - seg)) // (8 * 4 * SM))


def visit(n_chunks, lens, log2S, seg, grid, per):
    """The hash kernel's walk over its rows of segments: {(chunk, offset): visits}."""
    spc = log2S - seg
    rsh, seen = max(spc - 3, 0), {}
    for block in range(grid):
        for warp in range(8):
            r = 0
            while r < per:
                row = block * per + r
                q = row * 8 + ((warp + (row >> rsh)) & 7)
                c, off = q >> spc, (q & ((1 << spc) - 1)) << seg
                if c >= n_chunks:
                    break
                if off >= lens[c]:
                    r += (1 << rsh) - 1 - (row & ((1 << rsh) - 1))
                else:
                    seen[c, off] = seen.get((c, off), 0) + 1
                r += 1
    return seen


@pytest.mark.parametrize("seed", range(40))
def test_the_hash_walk_takes_every_segment_once(rules, seed):
    rng = random.Random(seed)
    log2S = rng.choice([4, 8, 13, 14, 15, 16, 17, 18, 20])
    allocs = [rng.choice([1, 16, 300, 5000, 70000, 1 << log2S, rng.randrange(1, 4 << log2S)])
              for _ in range(rng.randrange(1, 120))]
    lens = [min(1 << log2S, a - o) for a in allocs for o in range(0, a, 1 << log2S)]
    for copy in (0, 1):
        for sm in (1, 3):   # few SMs, so that warps take several rows
            seg, grid, per = hash_plan(rules, len(lens), sum(lens), log2S, copy, sm)
            seen = visit(len(lens), lens, log2S, seg, grid, per)
            assert set(seen.values()) <= {1}
            assert set(seen) == {(c, o) for c, ln in enumerate(lens) for o in range(0, ln, 1 << seg)}


def restore_plan(so, n, nbytes, log2S, coded, sm=SM, most=(1 << 64) - 1):
    out = (ctypes.c_uint32 * 2)()
    return so.restore_plan(n, nbytes, log2S, coded, sm, most, out), out[0], bool(out[1])


@pytest.mark.parametrize("log2S", range(13, 25))
def test_restore_of_full_chunks_a_warp_a_part(rules, log2S):
    n = (4 << 30) >> log2S
    ctas, part, _ = restore_plan(rules, n, 4 << 30, log2S, 0)
    assert part == 13 and ctas == (n << (log2S - 13)) // 8
    ctas, part, lanes = restore_plan(rules, n, 4 << 30, log2S, 1)
    assert part == max(min(15, log2S), log2S - 4) and ctas == ((n << (log2S - part)) + 7) // 8 and not lanes


@pytest.mark.parametrize("coded", [0, 1])
@pytest.mark.parametrize("log2S", [6, 9, 12, 13, 16, 18, 20, 24])
@pytest.mark.parametrize("n,each", [(1200, 5), (1200, 64), (1200, 4096), (20000, 2000), (50000, 200)])
def test_restore_of_short_allocations(rules, n, each, log2S, coded):
    """Work for every SM, and no more than a look-up of 32 parts at a time per warp."""
    each = min(each, 1 << log2S)
    ctas, part, lanes = restore_plan(rules, n, n * each, log2S, coded)
    items = n << (log2S - part)
    assert ctas >= min(4 * SM, items // 8) - 1
    assert ctas <= max(4 * SM, (n * each >> 13) + n // 8 + 1)
    assert not coded or lanes or items <= 2 * ((n * each >> part) + 1)


@pytest.mark.parametrize("seed", range(60))
def test_the_restore_walk_takes_every_part_once(rules, seed):
    rng = random.Random(seed)
    log2S, sm = rng.choice([4, 9, 13, 16, 18, 20, 24]), rng.choice([1, 3, 16])
    n, coded = rng.randrange(1, 400), rng.randrange(2)
    nbytes = rng.randrange(n, (n << log2S) + 1)
    ctas, part, lanes = restore_plan(rules, n, nbytes, log2S, coded, sm, rng.choice([1, 2, 5, 1 << 40]))
    items, nw = n << (log2S - part), 8 * ctas
    seen = [0] * items
    for j in range((items + nw - 1) // nw):
        for w in range(nw):
            it = j * nw + w // 8 * 8 + ((w % 8 + j) & 7)
            if it < items:
                seen[it] += 1
    assert set(seen) == {1}


def test_dense_placement_by_cta_where_the_counter_would_set_the_pace(rules):
    """Once per CTA from about three in ten 4 KiB with a dirty chunk, on 4 KiB chunks from 22%."""
    for log2S in (9, 10, 11, 12):
        n, least = 4096 >> log2S, 0.3 if log2S < 12 else 0.22
        for f in np.linspace(0, 0.25, 251):
            p = 1 - (1 - f) ** n
            if abs(p - least) > 1e-3:
                assert bool(rules.dense(f, log2S)) == (p > least), (f, log2S)
