"""The allocation-free pass over the forms it accepts (GPU): chunk sizes of every
hash kernel, sizes on and off the 16-byte grid (with and without the write-through
of a pass without a baseline), a staging buffer off the grid, no staging, and
buffers that are too small.  Bit for bit against the oracle's fingerprints."""
import numpy as np
import pytest
import torch

import paper_2008_10596_gb300 as C
import workloads as W
from oracle import oracle as O

pytestmark = [pytest.mark.gpu, pytest.mark.usefixtures("oracle_lib")]

NO_BASE = -1


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.uint64).view(np.int64)).to("cuda")


def _call(bufs, host, S, base, fp_old, shift=0, staging=True, idx_cap=None, cap=None):
    """One call; returns (err, k, bytes, fp, idx, off, staged bytes)."""
    sizes = [b.size for b in host]
    first = W.chunk_layout(sizes, S)
    n, total = int(first[-1]), sum(sizes)
    rows = np.array([[b.data_ptr(), s, f, (f if has else NO_BASE) % (1 << 64)]
                     for b, s, f, has in zip(bufs, sizes, first[:-1].tolist(), base)], dtype=np.uint64)
    idx_cap = n if idx_cap is None else idx_cap
    cap = total if cap is None else cap
    fp = torch.full((n,), 7, dtype=torch.int64, device="cuda")
    idx = torch.zeros(idx_cap + 1, dtype=torch.int64, device="cuda")
    off = torch.zeros(idx_cap + 2, dtype=torch.int64, device="cuda")
    room = torch.zeros(cap + 64, dtype=torch.uint8, device="cuda")
    totals = torch.zeros(3, dtype=torch.int64, device="cuda")
    C.crac_pass_noalloc(_dev(rows), len(sizes), n, S, fp_old, fp, idx, off, idx_cap,
                        room[shift:] if staging else None, cap, totals, torch.cuda.Stream())
    torch.cuda.synchronize()
    t = totals.cpu().numpy().view(np.uint64)
    assert not room[:shift].any() and not room[shift + cap:].any()
    return (int(t[0]) >> 32, int(t[1]), int(t[2]), fp, idx.cpu().numpy(), off.cpu().numpy(),
            room[shift:shift + cap].cpu().numpy())


def _expect(host, S, dirty):
    fps = np.concatenate([O.fp_chunks(h, S) for h in host])
    chunks = [h[i:i + S] for h in host for i in range(0, h.size, S)]
    ids = np.nonzero(dirty)[0]
    lens = np.array([chunks[i].size for i in ids], dtype=np.int64)
    pay = np.concatenate([chunks[i] for i in ids]) if len(ids) else np.zeros(0, np.uint8)
    return fps, ids, np.concatenate([[0], np.cumsum(lens)]), pay


ALIGNED = [65536 * 3 + 48, 16, 4096, 8192 + 512, 131072, 262144 + 16]
RAGGED = [65536 * 3 + 5, 3, 4097, 8191, 131072, 262144 + 1, 16]
FEW = [4096 * 3 + 5, 3, 4097, 100, 70001]   # one short list with 4-16 KiB chunks


@pytest.mark.parametrize("S", [64, 512, 4096, 8192, 16384, 65536, 262144])
@pytest.mark.parametrize("sizes", [ALIGNED, RAGGED, FEW], ids=["aligned", "ragged", "few"])
@pytest.mark.parametrize("shift", [0, 8])
def test_forms(S, sizes, shift):
    host = [W.host_contents("u32_xorshift", n, 70 + i) for i, n in enumerate(sizes)]
    bufs = [torch.from_numpy(h).to("cuda") for h in host]
    n = int(W.chunk_layout(sizes, S)[-1])
    every = [True] * len(sizes)

    def check(got, dirty):
        err, k, d, fp, idx, off, room = got
        fps, ids, offs, pay = _expect(host, S, dirty)
        assert err == 0 and k == len(ids) and d == pay.size
        assert np.array_equal(fp.cpu().numpy().view(np.uint64), fps)
        assert np.array_equal(idx[:k], ids) and np.array_equal(off[:k + 1], offs)
        assert np.array_equal(room[:d], pay)
        return fp

    base = check(_call(bufs, host, S, every, None, shift), np.ones(n, bool))
    check(_call(bufs, host, S, every, base, shift), np.zeros(n, bool))
    # two regions rewritten at one byte each, one region without a baseline
    first = W.chunk_layout(sizes, S)
    dirty = np.zeros(n, bool)
    for a, at in ((0, sizes[0] - 1), (4, 70000)):
        host[a][at] ^= 0x40
        dirty[int(first[a]) + at // S] = True
    dirty[int(first[2]):int(first[3])] = True
    bufs = [torch.from_numpy(h).to("cuda") for h in host]
    check(_call(bufs, host, S, [i != 2 for i in range(len(sizes))], base, shift), dirty)


@pytest.mark.parametrize("sizes", [ALIGNED, RAGGED, FEW], ids=["aligned", "ragged", "few"])
def test_too_small_buffers_are_reported(sizes):
    S = 4096
    host = [W.host_contents("u32_xorshift", n, 90 + i) for i, n in enumerate(sizes)]
    bufs = [torch.from_numpy(h).to("cuda") for h in host]
    n, total = int(W.chunk_layout(sizes, S)[-1]), sum(sizes)
    every = [True] * len(sizes)
    for kw in ({"idx_cap": n - 1}, {"cap": total - 1}, {"cap": 100}, {"staging": False, "cap": 0}):
        err, k, d, fp, *_ = _call(bufs, host, S, every, None, **kw)
        assert err == 2 and k == n and d == total, kw
        assert np.array_equal(fp.cpu().numpy().view(np.uint64), _expect(host, S, np.ones(n, bool))[0])
    # nothing dirty needs no room
    assert _call(bufs, host, S, every, fp, staging=False, cap=0, idx_cap=0)[:3] == (0, 0, 0)
