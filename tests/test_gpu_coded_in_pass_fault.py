"""A coded device image coded in the pass's own graph whose sizing wait runs out
(GPU): a tile of the sizing kernel is skipped, so the later tiles' bounded look-backs
expire.  The checkpoint reports CRAC_ERR_TIMEOUT, the coder's kernels having run
as nodes of the graph; no block stays taken, and the context goes on from its
last good image.  Nothing traps, faults or hangs."""
import numpy as np
import pytest

import paper_2008_10596_gb300 as C
import workloads as W
from tests.gpu_harness import Harness, pattern_mutations

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

KIB = 1024


@pytest.mark.parametrize("S", [8 * KIB, 64 * KIB])
@pytest.mark.parametrize("entries", [65, 300])   # two tiles of the sizing kernel, five
@pytest.mark.parametrize("first", [True, False], ids=["first", "later"])
def test_sizing_wait_runs_out_in_the_graph(S, entries, first):
    h = Harness(S, lineage=2300 + entries, image_residency=C.CRAC_RESIDENCY_DEVICE, flags=C.CRAC_FLAG_COMPRESS,
                timeout_ns=20_000_000, reserve_device_bytes=4 * entries * S + (16 << 20))
    try:
        sizes = [(entries - 10) * S, 9 * S + 100]
        for i, n in enumerate(sizes):
            h.add(n, data=W.host_contents(["f32_normal", "bf16"][i], n, 70 + i))
        if not first:   # a good chain, then a FULL pass again
            _, lib, ora = h.checkpoint()
            assert lib == ora
            C.crac_ctx_invalidate(h.ctx)
            h.oracle.invalidate()
        used = C.crac_memory_stats()["device_used_bytes"]
        C.crac_debug_inject_fault(C.CRAC_FAULT_ENCODE_WAIT, 1)
        with pytest.raises(C.CracError) as e:
            C.crac_ctx_checkpoint(h.ctx, h.stream)
        assert e.value.code == C.CRAC_ERR_TIMEOUT
        assert C.crac_ctx_last_pass(h.ctx)["kernel_launches"] == 7   # the coder's two among them
        assert C.crac_memory_stats()["device_used_bytes"] == used
        for step in range(3):   # FULL (the fault is spent), a delta, nothing dirty
            if step == 1:
                h.mutate(pattern_mutations(h.first(), sizes, S, "alternating", seed=6))
            img, lib, ora = h.checkpoint()
            assert lib == ora
            assert C.crac_ctx_last_pass(h.ctx)["kernel_launches"] == 7
        want = h.host()
        for b in h.bufs:
            b.zero()
        h.restart(img)
        for b, w in zip(h.bufs, want):
            assert np.array_equal(b.read(), w)
    finally:
        C.crac_debug_inject_fault(C.CRAC_FAULT_NONE, 0)
        h.close()
