"""Chunks below 512 bytes (GPU), which the hash kernel takes a warp each: images against
the oracle at lengths and payload offsets of every residue, and the allocation-free
pass, whose time follows what a chunk holds."""
import numpy as np
import pytest
import torch

import paper_2008_10596_gb300 as C
from tests.gpu_harness import Harness, pattern_mutations

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

GIB = 1 << 30


@pytest.mark.parametrize("S", [16, 32, 128, 256])
@pytest.mark.parametrize("ragged", [False, True])
@pytest.mark.parametrize("residency", [C.CRAC_RESIDENCY_DEVICE, C.CRAC_RESIDENCY_HOST])
def test_tiny_chunks(S, ragged, residency):
    rng = np.random.default_rng(S)
    sizes = [int(x) for x in rng.integers(1, 40 * S, 60)] + [S, 1, 16, S + 1, 3 * S - 1]
    if not ragged:
        sizes = [(n + 15) // 16 * 16 for n in sizes]
    h = Harness(S, lineage=2800 + S, image_residency=residency, pass_kernel=C.CRAC_PASS_SPLIT)
    try:
        for i, n in enumerate(sizes):
            h.add(n, seed=900 + i)
        img, lib, ora = h.checkpoint()
        assert lib == ora
        for pattern in ("alternating", "alternating", "random10", "all"):   # repeated: the predicted chunks too
            h.mutate(pattern_mutations(h.first(), sizes, S, pattern, seed=7))
            img, lib, ora = h.checkpoint()
            assert lib == ora
        want = h.host()
        for b in h.bufs:
            b.zero()
        h.restart(img)
        for b, w in zip(h.bufs, want):
            assert np.array_equal(b.read(), w)
    finally:
        h.close()


def test_time_follows_the_chunk():
    """The allocation-free pass over 512 MiB in chunks of 256 B against 512 B, nothing
    dirty: twice the chunks (7 times as long with the work of a 4 KiB segment for
    each)."""
    mem = torch.zeros(GIB // 16, dtype=torch.int64, device="cuda")
    total = mem.numel() * 8
    times = []
    for S in (512, 256):
        n = total // S
        reg = torch.tensor([[mem.data_ptr(), total, 0, 0]], dtype=torch.int64, device="cuda")
        fp = [torch.zeros(n, dtype=torch.int64, device="cuda") for _ in range(2)]
        idx, off = torch.zeros(n, dtype=torch.int64, device="cuda"), torch.zeros(n + 1, dtype=torch.int64, device="cuda")
        out = torch.empty(total, dtype=torch.uint8, device="cuda")
        t = torch.zeros(3, dtype=torch.int64, device="cuda")
        C.crac_pass_noalloc(reg, 1, n, S, None, fp[0], idx, off, n, out, total, t, None)
        assert int(t[1]) == n and int(t[2]) == total
        ms = []
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda.synchronize()
            e0.record()
            C.crac_pass_noalloc(reg, 1, n, S, fp[0], fp[1], idx, off, n, out, total, t, None)
            e1.record()
            torch.cuda.synchronize()
            assert int(t[1]) == 0 and torch.equal(fp[0], fp[1])
            ms.append(e0.elapsed_time(e1))
        times.append(min(ms))
    assert times[1] < 6 * times[0], times
