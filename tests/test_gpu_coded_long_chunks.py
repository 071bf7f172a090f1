"""Coded images in long chunks (GPU), whose streams many warps code: every segment's
units start where the sizing kernel says, also past 65535 units, with segments of
one block, and in images coded in the pass's graph, staged and drained directly.
And the coder's time does not grow with the chunk."""
import numpy as np
import pytest
import torch

import paper_2008_10596_gb300 as C
import workloads as W
from tests.gpu_harness import Harness, pattern_mutations

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

KIB, MIB = 1024, 1 << 20
FORMS = {"device": dict(image_residency=C.CRAC_RESIDENCY_DEVICE, flags=C.CRAC_FLAG_COMPRESS),
         "host": dict(image_residency=C.CRAC_RESIDENCY_HOST, flags=C.CRAC_FLAG_COMPRESS),
         "direct": dict(image_residency=C.CRAC_RESIDENCY_HOST, flags=C.CRAC_FLAG_COMPRESS | C.CRAC_FLAG_DIRECT_DRAIN)}


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("S,blocks", [(16 * KIB, 32), (32 * KIB, 33), (64 * KIB, 97), (MIB, 2 * 2048 - 31),
                                      (4 * MIB, 8192 + 4097), (16 * MIB, 9000)])
def test_units_of_every_segment(S, blocks, form):
    h = Harness(S, lineage=2600, **FORMS[form])
    try:
        sizes = [512 * blocks + 37, 512 * min(blocks, 300), S]
        for i, n in enumerate(sizes):
            data = W.host_contents("f32_normal", n, 50 + i)
            data[n // 3:n // 2] = 7   # constant blocks: no units
            h.add(n, data=data)
        for step in range(4):   # FULL, a delta, the same chunks again (predicted), nothing dirty
            if step in (1, 2):
                h.mutate(pattern_mutations(h.first(), sizes, S, "alternating", seed=8))
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


def test_coding_time_in_long_chunks():
    """256 MiB of fp32: the coder in chunks of 4 MiB against 64 KiB (8 times as long
    where every warp summed up its entry's widths so far)."""
    mem = torch.empty(64 * MIB, dtype=torch.float32, device="cuda").normal_()
    st = torch.cuda.Stream()
    times = []
    for S in (64 * KIB, 4 * MIB):
        ctx = C.crac_ctx_create(C.crac_config_default(chunk_bytes=S, reserve_device_bytes=1 << 30, **FORMS["device"]))
        try:
            C.crac_ctx_register_alloc(ctx, mem.data_ptr(), 256 * MIB)
            ms = []
            for _ in range(5):
                C.crac_ctx_invalidate(ctx)
                img = C.crac_ctx_checkpoint(ctx, st)
                C.crac_ctx_drop_history(ctx)
                C.crac_image_release(img)
                ms.append(C.crac_ctx_last_pass(ctx)["codec_ms"])
            times.append(min(ms))
        finally:
            torch.cuda.synchronize()
            C.crac_ctx_destroy(ctx)
    assert times[1] < 2.5 * times[0], times
