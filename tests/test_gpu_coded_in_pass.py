"""Coded device images of one segment (GPU), coded in the pass's own graph from
the allocations or gathered into staging first (here: while an injected sizing
fault is armed that too few entries meet, or with allocations in host memory):
the same images, byte for byte against the oracle, around the sizing kernel's
64 entries a tile, with nothing dirty, and with more than the coder's grid."""
import numpy as np
import pytest

import paper_2008_10596_gb300 as C
import workloads as W
from tests.gpu_harness import Harness, pattern_mutations

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

KIB = 1024


def _launches(h):
    return C.crac_ctx_last_pass(h.ctx)["kernel_launches"]


def _check(h, img):
    want = h.host()
    for b in h.bufs:
        b.zero()
    h.restart(img)
    for b, w in zip(h.bufs, want):
        assert np.array_equal(b.read(), w)


@pytest.mark.parametrize("staged", [False, True])
@pytest.mark.parametrize("S", [8 * KIB, 64 * KIB, 512 * KIB])
@pytest.mark.parametrize("entries", [1, 63, 64, 65, 129])
def test_coded_in_pass(S, entries, staged):
    if staged and entries > 64:
        pytest.skip("the armed fault would be met")
    h = Harness(S, lineage=2100 + entries, image_residency=C.CRAC_RESIDENCY_DEVICE, flags=C.CRAC_FLAG_COMPRESS)
    try:
        ends = [1, 511, 512, 1024, 16 * KIB + 16, S - 1]   # of each allocation's last chunk
        left, i = entries, 0
        while left:
            n = min(left, 1 + 7 * i)
            size = (n - 1) * S + min(ends[i % len(ends)], S)
            h.add(size, data=W.host_contents(["f32_normal", "u8", "bf16"][i % 3], size, 30 + i))
            left -= n
            i += 1
        sizes = [b.nbytes for b in h.bufs]
        if staged:
            C.crac_debug_inject_fault(C.CRAC_FAULT_ENCODE_WAIT, 1)
        for step in range(4):   # FULL, a delta, a like one (predicted), nothing dirty
            if step in (1, 2):
                h.mutate(pattern_mutations(h.first(), sizes, S, "alternating", seed=5))
            img, lib, ora = h.checkpoint()
            assert lib == ora
            assert _launches(h) == (7 if not staged else 8 if step < 3 else 5)   # (no entries: nothing to code)
        _check(h, img)
    finally:
        C.crac_debug_inject_fault(C.CRAC_FAULT_NONE, 0)
        h.close()


@pytest.mark.parametrize("kind", [C.CRAC_KIND_DEVICE, C.CRAC_KIND_HOST, C.CRAC_KIND_MANAGED])
def test_coded_in_pass_strides(kind):
    """A delta of 24000 entries, more than the coder's grid has warps."""
    S = 8 * KIB
    h = Harness(S, lineage=2200, image_residency=C.CRAC_RESIDENCY_DEVICE, flags=C.CRAC_FLAG_COMPRESS)
    try:
        n = 24000 * S if kind == C.CRAC_KIND_DEVICE else 300 * S
        h.add(n, kind=kind, data=W.host_contents("bf16", n, 3))
        img, lib, ora = h.checkpoint()
        assert lib == ora
        h.mutate(pattern_mutations(h.first(), [n], S, "all", seed=4))
        img, lib, ora = h.checkpoint()
        assert lib == ora
        assert _launches(h) == (8 if kind == C.CRAC_KIND_HOST else 7)
        _check(h, img)
    finally:
        h.close()
