"""Deltas and coded images over allocations much shorter than a chunk (GPU), beside a
few long ones: the gather and the coder take several parts of an entry per item, byte
for byte against the oracle, and empty parts do not set their pace."""
import random

import numpy as np
import pytest
import torch

import paper_2008_10596_gb300 as C
import workloads as W
from paper_2008_10596_gb300 import testkit
from tests.gpu_harness import Harness, pattern_mutations

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

KIB, MIB = 1024, 1 << 20
FORMS = {"device": dict(image_residency=C.CRAC_RESIDENCY_DEVICE),
         "host": dict(image_residency=C.CRAC_RESIDENCY_HOST),
         "segments": dict(image_residency=C.CRAC_RESIDENCY_DEVICE, staging_bytes=18 * MIB),   # one long chunk in each
         "coded": dict(image_residency=C.CRAC_RESIDENCY_DEVICE, flags=C.CRAC_FLAG_COMPRESS),
         "coded host": dict(image_residency=C.CRAC_RESIDENCY_HOST, flags=C.CRAC_FLAG_COMPRESS),
         "coded direct": dict(image_residency=C.CRAC_RESIDENCY_HOST,
                              flags=C.CRAC_FLAG_COMPRESS | C.CRAC_FLAG_DIRECT_DRAIN)}


@pytest.mark.parametrize("form", sorted(FORMS))
@pytest.mark.parametrize("S,n", [(4 * MIB, 700), (16 * MIB, 700)])
def test_entries_of_several_parts(S, n, form):
    """A full chunk and one of an odd length between short ones, all dirty."""
    h = Harness(S, lineage=2700, **FORMS[form])
    try:
        sizes = [16 + 13 * (i % 90) for i in range(n)] + [S, S // 2 + 8191] + [48] * 40
        for i, b in enumerate(sizes):
            data = W.host_contents(["u8", "f32_normal", "bf16"][i % 3], b, 30 + i)
            data[b // 3:b // 2] = 7   # constant blocks: no units
            h.add(b, data=data)
        for step in range(3):   # FULL, two deltas: the same chunks again (predicted)
            if step:
                h.mutate(pattern_mutations(h.first(), sizes, S, "all", seed=8))
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


@pytest.mark.parametrize("form", ["device", "coded"])
def test_empty_parts_do_not_set_the_pace(form):
    """20000 allocations below 4 KiB, all dirty, in chunks of 4 MiB against 16 KiB: the
    gather and the coder (eight times as long and more where every part of a chunk was
    looked up)."""
    r = random.Random(5)
    sizes = [r.randrange(1, 4096) for _ in range(20000)]
    mem = torch.zeros(20000 * 4096 // 4, dtype=torch.float32, device="cuda").normal_()
    st = torch.cuda.Stream()
    rows = torch.tensor([[mem.data_ptr() + 4096 * i, n, 1] for i, n in enumerate(sizes)], dtype=torch.int64, device="cuda")
    times = []
    for S in (16 * KIB, 4 * MIB):
        ctx = C.crac_ctx_create(C.crac_config_default(chunk_bytes=S, pass_kernel=C.CRAC_PASS_SPLIT,
                                                      reserve_device_bytes=1 << 30, **FORMS[form]))
        try:
            for i, n in enumerate(sizes):
                C.crac_ctx_register_alloc(ctx, mem.data_ptr() + 4096 * i, n)
            img = C.crac_ctx_checkpoint(ctx, st)
            ms = []
            for _ in range(5):
                C.crac_image_wait(img)
                torch.cuda.synchronize()
                testkit.mutate_xor(rows.data_ptr(), len(sizes))
                torch.cuda.synchronize()
                new = C.crac_ctx_checkpoint(ctx, st)
                C.crac_image_wait(new)
                C.crac_ctx_drop_history(ctx)
                C.crac_image_release(img)
                img = new
                info = C.crac_ctx_last_pass(ctx)
                assert info["k"] == len(sizes)
                ms.append(info["gather_ms"] + info["codec_ms"])
            C.crac_image_release(img)
            times.append(min(ms))
        finally:
            torch.cuda.synchronize()
            C.crac_ctx_destroy(ctx)
    assert times[1] < 4 * times[0], times
