"""Allocations much shorter than a chunk, alone and beside long ones (GPU): images
and restores byte for byte against the oracle, over every way a chunk is cut into
segments, and the pass's work spread over the chip."""
import numpy as np
import pytest
import torch

import paper_2008_10596_gb300 as C
import workloads as W
from tests.gpu_harness import Harness, pattern_mutations

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

KIB, MIB = 1024, 1 << 20
FORMS = {
    "device": dict(image_residency=C.CRAC_RESIDENCY_DEVICE),
    "coded": dict(image_residency=C.CRAC_RESIDENCY_DEVICE, flags=C.CRAC_FLAG_COMPRESS),
    "incremental": dict(image_residency=C.CRAC_RESIDENCY_DEVICE, flags=C.CRAC_FLAG_INCREMENTAL_RESTORE),
    "host": dict(image_residency=C.CRAC_RESIDENCY_HOST),
}


def _sizes(layout, S):
    short = [64, 5, 300, 17, 511, 16]
    if layout == "short":
        return [min(S, short[i % 6]) for i in range(900)]
    if layout == "aligned":
        return [min(S, 16 * (1 + i % 5)) for i in range(900)]
    return [2 * S + 100] + [min(S, short[i % 6]) for i in range(300)] + [S - 1, S, S + 1]


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("layout", ["short", "aligned", "mixed"])
@pytest.mark.parametrize("S", [64, 512, 8 * KIB, 64 * KIB, 256 * KIB, MIB, 16 * MIB])
def test_short_allocations(S, layout, form):
    if (S, layout, form) == (16 * MIB, "mixed", "coded"):
        pytest.skip("80 MB through the oracle's coder")
    h = Harness(S, lineage=2400, **FORMS[form])
    try:
        sizes = _sizes(layout, S)
        for i, n in enumerate(sizes):
            h.add(n, data=W.host_contents(["u8", "f32_normal", "bf16"][i % 3], n, 30 + i))
        for step in range(3):   # FULL, a delta, nothing dirty
            if step == 1:
                h.mutate(pattern_mutations(h.first(), sizes, S, "alternating", seed=8))
            img, lib, ora = h.checkpoint()
            assert lib == ora
            if layout != "mixed" and not 512 <= S < 8 * KIB:
                sms = torch.cuda.get_device_properties(0).multi_processor_count
                n = C.crac_ctx_last_pass(h.ctx)["n_chunks"]
                assert C.crac_ctx_last_pass(h.ctx)["grid"] >= min(4 * sms, n // 8)
        want = h.host()
        h.mutate(pattern_mutations(h.first(), sizes, S, "random10", seed=9))
        h.restart(img)
        for b, w in zip(h.bufs, want):
            assert np.array_equal(b.read(), w)
    finally:
        h.close()
