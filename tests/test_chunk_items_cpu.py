"""The rule that gives chunks their work items (csrc/crac_grids.h), compiled and run on
the host: every part is some item's, full chunks keep an item per part, and empty items
stay few."""
import ctypes
import os
import random
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
LANES = 32 * 152 * 64


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("items")
    (d / "wrap.cpp").write_text('#include "crac_grids.h"\nextern "C" uint32_t items(uint64_t n, uint64_t b, uint32_t p, '
                                'uint32_t q, uint64_t l) { return crac::chunk_items(n, b, p, q, l); }\n')
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2008_10596_gb300", "csrc"), str(d / "wrap.cpp"), "-o", str(d / "w.so")],
                   check=True)
    so = ctypes.CDLL(str(d / "w.so"))
    so.items.argtypes = [ctypes.c_uint64, ctypes.c_uint64, ctypes.c_uint32, ctypes.c_uint32, ctypes.c_uint64]
    return so.items


@pytest.mark.parametrize("log2S", range(13, 25))
@pytest.mark.parametrize("n", [1, 3, 1000, 1 << 20])
def test_full_chunks_an_item_a_part(rule, n, log2S):
    assert rule(n, n << log2S, 13, log2S - 13, LANES) == log2S - 13
    assert rule(n, (n << log2S) // 2, 13, log2S - 13, LANES) == log2S - 13


@pytest.mark.parametrize("log2S", range(13, 25))
@pytest.mark.parametrize("n,each", [(1200, 5), (20000, 2000), (50000, 200), (1 << 20, 16)])
def test_short_chunks_few_items(rule, n, each, log2S):
    parts = log2S - 13
    items = rule(n, n * each, 13, parts, LANES)
    assert min(3, max(parts - 2, 0)) <= items <= parts
    assert items <= 3 or (n << items) <= LANES


@pytest.mark.parametrize("seed", range(40))
def test_every_part_once(rule, seed):
    rng = random.Random(seed)
    log2S, lanes = rng.choice([13, 16, 17, 20, 24]), rng.choice([64, 1000, LANES])
    lens = [rng.choice([1, 100, 8192, 8193, 1 << log2S, rng.randrange(1, (1 << log2S) + 1)]) if rng.random() < 0.1
            else rng.randrange(1, 4096) for _ in range(rng.randrange(1, 300))]
    lens = [min(x, 1 << log2S) for x in lens]
    items = rule(len(lens), sum(lens), 13, log2S - 13, lanes)
    stride = 1 << (13 + items)
    for n in set(lens):
        seen = []
        for s in range(1 << items):
            po, rest = s << 13, n - (s << 13)
            while rest > 0:   # the gather's loop
                seen.append((po, min(8192, rest)))
                if rest <= stride:
                    break
                rest -= stride
                po += stride
        assert sorted(seen) == [(o, min(8192, n - o)) for o in range(0, n, 8192)]
