"""Lists of several hundred thousand chunks (GPU), which the compaction takes in
larger tiles: chunk counts around its threshold, every chunk listed, few, and
dense placement, against the oracle's images and fingerprints."""
import numpy as np
import pytest
import torch

import paper_2008_10596_gb300 as C
import workloads as W
from oracle import oracle as O
from tests.gpu_harness import Harness

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]


@pytest.mark.parametrize("S,total,residency", [(64, 20 << 20, C.CRAC_RESIDENCY_HOST), (64, 40 << 20, C.CRAC_RESIDENCY_HOST),
                                               (512, 170 << 20, C.CRAC_RESIDENCY_DEVICE),
                                               (2048, 420 << 20, C.CRAC_RESIDENCY_HOST)])   # three iterations a warp
def test_many_chunks(S, total, residency):
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    at = 2 * n_sm * 1024 * S if S == 64 and total < 30 << 20 else total   # just past the threshold, or well past it
    sizes = [at // 2 // 16 * 16, 16 * 1001, at // 2 // 16 * 16]
    h = Harness(S, lineage=2100 + S % 97, image_residency=residency)
    try:
        for i, n in enumerate(sizes):
            h.add(n, data=np.random.default_rng(i).integers(0, 256, n, dtype=np.uint8))
        img, lib, ora = h.checkpoint()
        assert lib == ora
        n = int(h.first()[-1])
        rng = np.random.default_rng(9)
        for _ in range(2):   # the second of them with dense placement on 512 B - 4 KiB chunks of device images
            ids = np.unique(rng.integers(0, n, n // 50))
            h.mutate([W.ChunkMutation(int(c), 0x5A5A5A5B) for c in ids])
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


def test_many_chunks_without_allocation():
    S, n_bytes = 64, (40 << 20) + 5
    host = np.random.default_rng(3).integers(0, 256, n_bytes, dtype=np.uint8)
    buf = torch.from_numpy(host).to("cuda")
    n = -(-n_bytes // S)
    regions = torch.tensor([[buf.data_ptr(), n_bytes, 0, 0]], dtype=torch.int64, device="cuda")
    out = [torch.zeros(n + 1, dtype=torch.int64, device="cuda") for _ in range(4)]
    staging = torch.zeros(n_bytes, dtype=torch.uint8, device="cuda")
    totals = torch.zeros(3, dtype=torch.int64, device="cuda")
    C.crac_pass_noalloc(regions, 1, n, S, None, out[0], out[2], out[3], n, staging, n_bytes, totals)
    torch.cuda.synchronize()
    assert np.array_equal(out[0].cpu().numpy().view(np.uint64)[:n], O.fp_chunks(host, S))
    assert totals.tolist()[1:] == [n, n_bytes] and np.array_equal(staging.cpu().numpy(), host)
    ids = np.unique(np.random.default_rng(4).integers(0, n, 5000))
    host[ids * S] ^= 1
    buf.copy_(torch.from_numpy(host))
    C.crac_pass_noalloc(regions, 1, n, S, out[0], out[1], out[2], out[3], n, staging, n_bytes, totals)
    torch.cuda.synchronize()
    assert np.array_equal(out[1].cpu().numpy().view(np.uint64)[:n], O.fp_chunks(host, S))
    assert totals.tolist()[1] == len(ids) and np.array_equal(out[2].cpu().numpy()[:len(ids)], ids)
    off = out[3].cpu().numpy()
    lens = np.minimum(S, n_bytes - ids * S)
    assert np.array_equal(off[:len(ids) + 1], np.concatenate([[0], np.cumsum(lens)]))
    st = staging.cpu().numpy()
    assert all(np.array_equal(st[o:o + ln], host[c * S:c * S + ln]) for c, o, ln in zip(ids[:500], off, lens))
