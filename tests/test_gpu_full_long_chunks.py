"""FULL passes over chunks of several MiB (GPU): the warps of the whole chip add to a
few chunks' sums, which must not set the pass's pace."""
import pytest
import torch

import paper_2008_10596_gb300 as C

pytestmark = pytest.mark.gpu

KIB, MIB, GIB = 1024, 1 << 20, 1 << 30


@pytest.mark.parametrize("S", [4 * MIB, 16 * MIB])
def test_full_pass_in_long_chunks(S):
    """2 GiB, device time of the hash kernel against chunks of 64 KiB (1.25 times with
    an addition per 8 KiB into sums of 16 MiB)."""
    mem = torch.zeros(2 * GIB // 8, dtype=torch.int64, device="cuda")
    st = torch.cuda.Stream()
    times = []
    for chunk in (64 * KIB, S):
        ctx = C.crac_ctx_create(C.crac_config_default(chunk_bytes=chunk, image_residency=C.CRAC_RESIDENCY_DEVICE,
                                                      reserve_device_bytes=5 * GIB))
        try:
            C.crac_ctx_register_alloc(ctx, mem.data_ptr(), 2 * GIB)
            ms = []
            for _ in range(12):
                C.crac_ctx_invalidate(ctx)
                img = C.crac_ctx_checkpoint(ctx, st)
                C.crac_image_wait(img)
                C.crac_ctx_drop_history(ctx)
                C.crac_image_release(img)
                ms.append(C.crac_ctx_last_pass(ctx)["hash_ms"])
            times.append(min(ms))
        finally:
            torch.cuda.synchronize()
            C.crac_ctx_destroy(ctx)
    assert times[1] < 1.06 * times[0], times
