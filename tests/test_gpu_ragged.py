"""Payloads off the 16-byte grid (GPU): allocations of any byte size shift every
later chunk's payload offset, so the copies into the payload and back out of it
run between differently aligned addresses.  Byte for byte against the oracle."""
import numpy as np
import pytest

import paper_2008_10596_gb300 as C
from tests.gpu_harness import Harness, pattern_mutations

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

KIB = 1024

# Every residue of the payload offset mod 16, and lengths around one vector, one
# warp's 512-byte row and its 2 KiB strip; then chunks cut into 8 KiB parts.
SHORT = [1, 15, 16, 17, 31, 33, 47, 62, 63, 64, 511, 512, 513, 527, 2047, 2048, 2049, 2063, 2064, 4095, 4111]
LONG = [64 * KIB + 1, 3, 64 * KIB - 1, 8 * KIB + 7, 16 * KIB - 5, 200001, 64 * KIB * 3, 24 * KIB + 2, 131072 + 13]


@pytest.mark.parametrize("S,sizes", [(4 * KIB, SHORT), (64 * KIB, LONG + SHORT), (256 * KIB, LONG + [700001, 5, 262144])])
@pytest.mark.parametrize("kern", [C.CRAC_PASS_SPLIT, C.CRAC_PASS_LDG, C.CRAC_PASS_AUTO])
@pytest.mark.parametrize("residency", [C.CRAC_RESIDENCY_DEVICE, C.CRAC_RESIDENCY_HOST])
def test_ragged_sizes(S, sizes, kern, residency):
    flags = C.CRAC_FLAG_STAGED_RESTORE if residency == C.CRAC_RESIDENCY_HOST and kern == C.CRAC_PASS_LDG else 0
    h = Harness(S, lineage=1500 + S % 97 + kern, pass_kernel=kern, image_residency=residency, flags=flags)
    try:
        for i, n in enumerate(sizes):
            h.add(n, seed=400 + i)
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


@pytest.mark.parametrize("S", [64, 256, 512, 1 * KIB, 2 * KIB, 4 * KIB, 8 * KIB, 16 * KIB, 64 * KIB])
@pytest.mark.parametrize("flags", [0, C.CRAC_FLAG_DIRECT_DRAIN, C.CRAC_FLAG_COMPRESS])
def test_ragged_write_through(S, flags):
    """The hash kernels write FULL and predicted chunks to payload offsets of any
    alignment: chunks of every length mod 16, each at every offset mod 16 across
    the list, in every lane layout of the hash kernels."""
    rng = np.random.default_rng(S + flags)
    sizes = [S + 1, 1, 15, 16, 17, S - 1, 3 * S + 7] + [int(x) for x in rng.integers(1, 3 * S, 40)] + [2 * S, 5]
    h = Harness(S, lineage=1700 + S % 97 + flags, flags=flags)
    try:
        for i, n in enumerate(sizes):
            h.add(n, seed=800 + i)
        img, lib, ora = h.checkpoint()
        assert lib == ora
        muts = pattern_mutations(h.first(), sizes, S, "random10", seed=11)
        for _ in range(3):   # the same chunks: found in place from the second pass on
            h.mutate(muts)
            img, lib, ora = h.checkpoint()
            assert lib == ora
        if not flags:
            assert C.crac_ctx_last_pass(h.ctx)["in_place"] == len(muts)
        want = h.host()
        for b in h.bufs:
            b.zero()
        h.restart(img)
        for b, w in zip(h.bufs, want):
            assert np.array_equal(b.read(), w)
    finally:
        h.close()
