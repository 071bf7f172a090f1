"""The allocation-free pass over many regions (GPU): payload offsets of a pass
without a baseline, which one CTA sums up, around its 32 warps of 32 regions and
past the scratch's room for them; and that summing up does not outweigh the pass."""
import numpy as np
import pytest
import torch

import paper_2008_10596_gb300 as C
import workloads as W
from tests.test_gpu_noalloc_forms import _call, _expect

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]


@pytest.mark.parametrize("n", [1, 31, 32, 33, 1023, 1024, 1025, 2049, 20000, 64000, 70000])
def test_payload_offsets_of_many_regions(n):
    rng = np.random.default_rng(n)
    sizes = rng.integers(1, 65, n)
    sizes[n // 2] = 4096 * 5 + 3
    at = np.concatenate([[0], np.cumsum(-(-sizes // 16) * 16)])
    data = torch.from_numpy(rng.integers(0, 256, int(at[-1]), dtype=np.uint8)).cuda()
    host = data.cpu().numpy()
    bufs = [data[a:a + s] for a, s in zip(at.tolist(), sizes.tolist())]
    parts = [host[a:a + s] for a, s in zip(at.tolist(), sizes.tolist())]
    S = 4096
    err, k, d, fp, idx, off, staged = _call(bufs, parts, S, [False] * n, None)
    fps, ids, offs, pay = _expect(parts, S, np.ones(int(W.chunk_layout(sizes.tolist(), S)[-1]), bool))
    assert (err, k, d) == (0, len(ids), pay.size)
    assert np.array_equal(fp.cpu().numpy().view(np.uint64), fps)
    assert np.array_equal(idx[:k], ids) and np.array_equal(off[:k + 1], offs)
    assert np.array_equal(staged[:d], pay)


def test_summing_up_the_regions_is_a_small_part():
    """50000 regions of 200 bytes: the pass that sums them up against the one with a
    baseline and nothing dirty, which does not (2.0 times its time where each thread
    walked its own run of regions)."""
    n, S = 50000, 256
    mem = torch.zeros(n * 256, dtype=torch.uint8, device="cuda")
    rows = np.stack([mem.data_ptr() + 256 * np.arange(n), np.full(n, 200), np.arange(n), np.arange(n)], 1)
    reg = torch.from_numpy(rows.astype(np.int64)).cuda()
    fp, fp2, idx, off = (torch.zeros(n + 1, dtype=torch.int64, device="cuda") for _ in range(4))
    room, totals = torch.zeros(n * 200, dtype=torch.uint8, device="cuda"), torch.zeros(3, dtype=torch.int64, device="cuda")
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]

    def least(fp_old, fp_new):
        best = 1e9
        for _ in range(20):
            torch.cuda.synchronize()
            ev[0].record()
            for _ in range(10):   # so that the calls' host time does not count
                C.crac_pass_noalloc(reg, n, n, S, fp_old, fp_new, idx, off, n, room, n * 200, totals,
                                    torch.cuda.current_stream())
            ev[1].record()
            torch.cuda.synchronize()
            best = min(best, ev[0].elapsed_time(ev[1]) / 10)
        return best

    full, clean = least(None, fp), least(fp, fp2)
    assert full < 1.6 * clean, (full, clean)
