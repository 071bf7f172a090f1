"""The fused LDG pass over sizes off the 16-byte grid (GPU): short chunks are copied
without vectors, longer ones by shifted vectors, against the oracle, and the former do
not take much longer than aligned ones."""
import numpy as np
import pytest
import torch

import paper_2008_10596_gb300 as C
from tests.gpu_harness import Harness, pattern_mutations

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

KIB, MIB = 1024, 1 << 20


@pytest.mark.parametrize("step", [1, 4, 16])   # sizes off the grid, on the 4-byte grid, on the 16-byte grid
@pytest.mark.parametrize("S", [16, 64, 256, 512, 8 * KIB, 16 * KIB])
def test_ragged_chunks(S, step):
    rng = np.random.default_rng(S + step)
    top = max(2, 5 * S // step)
    sizes = [int(x) * step for x in rng.integers(1, top, 50)] + [step, S, 3 * S + step]
    h = Harness(S, lineage=2900 + S % 97, pass_kernel=C.CRAC_PASS_LDG, image_residency=C.CRAC_RESIDENCY_DEVICE)
    try:
        for i, n in enumerate(sizes):
            h.add(n, seed=700 + i)
        img, lib, ora = h.checkpoint()
        assert lib == ora
        for pattern in ("alternating", "all"):
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


def test_short_ragged_chunks_against_aligned_ones():
    """256 MiB in 64 allocations, 256 B chunks, all dirty: off the 4-byte grid against on
    the 16-byte grid (1.7 times as long by the shifted copy's call)."""
    mem = torch.zeros(256 * MIB, dtype=torch.uint8, device="cuda")
    st = torch.cuda.Stream()
    times = []
    for less in (0, 1):
        ctx = C.crac_ctx_create(C.crac_config_default(chunk_bytes=256, pass_kernel=C.CRAC_PASS_LDG,
                                                      image_residency=C.CRAC_RESIDENCY_DEVICE,
                                                      reserve_device_bytes=2 << 30))
        try:
            for i in range(64):
                C.crac_ctx_register_alloc(ctx, mem.data_ptr() + 4 * MIB * i, 4 * MIB - less)
            img = C.crac_ctx_checkpoint(ctx, st)
            ms = []
            for _ in range(6):
                C.crac_image_wait(img)
                torch.cuda.synchronize()
                mem.bitwise_xor_(1)
                torch.cuda.synchronize()
                new = C.crac_ctx_checkpoint(ctx, st)
                C.crac_image_wait(new)
                C.crac_ctx_drop_history(ctx)
                C.crac_image_release(img)
                img = new
                info = C.crac_ctx_last_pass(ctx)
                assert info["k"] == info["n_chunks"] and info["pass_kernel"] == C.CRAC_PASS_LDG
                ms.append(info["device_ms"])
            C.crac_image_release(img)
            times.append(min(ms))
        finally:
            torch.cuda.synchronize()
            C.crac_ctx_destroy(ctx)
    assert times[1] < 1.45 * times[0], times
