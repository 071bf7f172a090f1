"""Coded images of chunks that the coder and the decoder share out among warps
(GPU): lengths around the 16 KiB coding segments and the 32 KiB decoding parts,
odd block counts, tails, raw chunks among coded ones, and planes that use the
whole byte range, byte for byte against the oracle."""
import numpy as np
import pytest

import paper_2008_10596_gb300 as C
import workloads as W
from tests.gpu_harness import Harness, pattern_mutations

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

KIB = 1024


def _contents(kind, n, seed):
    if kind == "zeros":
        return np.zeros(n, np.uint8)
    if kind == "wide":   # planes whose largest offset reaches 255 on a minimum above 0, next to narrow ones
        rng = np.random.default_rng(seed)
        w = rng.integers(0, 128, size=(-(-n // 4), 4), dtype=np.uint8) * 2 + 1
        w[:, 1] = rng.integers(200, 203, size=w.shape[0])
        w[:, 2] = 0
        return w.reshape(-1)[:n].copy()
    if kind == "half":   # windows of constant blocks before and between others
        h = W.host_contents("f32_normal", n, seed)
        h[: n // 2] = 0x7F
        h[3 * n // 4: 3 * n // 4 + 20 * KIB] = 0
        return h
    return W.host_contents(kind, n, seed)


@pytest.mark.parametrize("S", [8 * KIB, 16 * KIB, 32 * KIB, 64 * KIB, 1024 * KIB])
@pytest.mark.parametrize("residency,flags", [(C.CRAC_RESIDENCY_DEVICE, 0), (C.CRAC_RESIDENCY_HOST, 0),
                                             (C.CRAC_RESIDENCY_HOST, C.CRAC_FLAG_DIRECT_DRAIN)])
def test_coded_parts(S, residency, flags):
    edges = [512, 513, 16 * KIB - 512, 16 * KIB, 16 * KIB + 512 + 4, 32 * KIB - 16, 32 * KIB + 511, 48 * KIB + 1024,
             64 * KIB - 1, 2 * S, S + 16 * KIB + 3]
    kinds = ["f32_normal", "zeros", "bf16", "half", "wide", "u8"]
    h = Harness(S, lineage=1900 + S % 97 + flags, image_residency=residency, flags=C.CRAC_FLAG_COMPRESS | flags)
    try:
        sizes = []
        for i, n in enumerate(edges):
            h.add(n, data=_contents(kinds[i % len(kinds)], n, 40 + i))
            h.add(16 * (n // 16) + 16, data=_contents(kinds[(i + 2) % len(kinds)], 16 * (n // 16) + 16, 60 + i))
            sizes += [n, 16 * (n // 16) + 16]
        img, lib, ora = h.checkpoint()
        assert lib == ora
        h.mutate(pattern_mutations(h.first(), sizes, S, "alternating", seed=5))
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
