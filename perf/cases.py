"""Performance cases of the checkpoint/restart data pass, through the package's
public entry points.

A case is one pass of what a program does with this library:

  cycle     FULL checkpoint of every allocation, then `deltas` times: the
            application rewrites part of its memory and takes an incremental
            checkpoint; then the newest image (its whole chain) is restored
            into a second context, the restarted process's own allocations.
  rollback  the application rewrites part of its memory and goes back to a
            saved image in place.
  noalloc   the allocation-free pass over caller-owned buffers: once with no
            baseline (every chunk), once against a baseline.
  serve     many process contexts through the request server: FULL and
            incremental checkpoints of each, restarts of some.

Sizes, chunk sizes, contents and dirty fractions follow the benchmark's five
configurations, scaled so that three sets of inputs fit the card.  Outputs are
whole bytes and counts (restored memory, tables, payload), so two versions of
the library have to agree on every one; there is nothing to compare in 64 bits.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2008_10596_gb300 as C
from paper_2008_10596_gb300 import testkit

KIB, MIB, GIB = 1 << 10, 1 << 20, 1 << 30
PLACE = 512   # allocations start on 512-byte boundaries, as a caching allocator places them


def _cycle(name, total, n, lo, hi, chunk, content, **kw):
    c = {"name": name, "op": "cycle", "total": total, "n": n, "lo": lo, "hi": hi, "align": 256, "chunk": chunk,
         "content": content, "page": chunk, "dirty": 0.10, "hot": True, "deltas": 1, "host": False, "coded": False,
         "managed": 0.0, "persist": False, "layout": "loguniform", "sizes_seed": 2008105960}
    c.update(kw)
    return c


def listed():
    return [
        # Configuration 1: one 16 MiB buffer of random words in 4 KiB chunks, 1% of them
        # rewritten, images in pinned host memory (the default), the delta written out.
        # The smallest call: its time is launches and round trips.
        _cycle("c1_16MiB_host", 16 * MIB, 1, 16 * MIB, 16 * MIB, 4 * KIB, "u32", dirty=0.01, host=True, persist=True),
        # The tensors of a small bf16 model, registered with their exact byte sizes (any even
        # number): many short allocations, ragged ends, chunks longer than most of them.
        _cycle("tensors_96MiB", 96 * MIB, 1200, 258, 1 * MIB, 64 * KIB, "bf16", align=2, dirty=0.25, deltas=3),
        # Configuration 2 at a quarter of its size with host images: the everyday
        # checkpoint that drains over the host link and restarts from there.
        _cycle("c2_1GiB_host", 1 * GIB, 256, 4 * KIB, 16 * MIB, 64 * KIB, "f32", host=True, deltas=2),
        # Configuration 2 as it stands: 256 allocations, 4 GiB, 10% of the chunks rewritten,
        # images kept in device memory; every fourth checkpoint FULL, as the serving loop does.
        _cycle("c2_4GiB", 4 * GIB, 256, 4 * KIB, 64 * MIB, 64 * KIB, "f32", deltas=3),
        # Configuration 3: device and managed allocations, bf16 contents, 25% of 64 KiB
        # pages rewritten at random places, three successive checkpoints and a restart.
        _cycle("c3_2GiB_managed", 2 * GIB, 40, 64 * KIB, 256 * MIB, 64 * KIB, "bf16", align=64 * KIB, dirty=0.25,
               deltas=2, hot=False, managed=0.25),
        # Configuration 4's memory (Zipf sizes, mixed contents) in 4 KiB chunks, 10% of the
        # pages rewritten at random places: large tables, many short dirty runs.
        _cycle("c4_8GiB_4KiB", 8 * GIB, 512, 4 * KIB, 2 * GIB, 4 * KIB, "mixed", layout="zipf", align=4 * KIB,
               deltas=2, hot=False),
        # The same memory in 256 KiB chunks with half of the 4 KiB pages rewritten, so that
        # nearly every chunk is dirty: the largest pass, payloads as large as the memory.
        _cycle("c4_16GiB_256KiB", 16 * GIB, 1024, 4 * KIB, 4 * GIB, 256 * KIB, "mixed", layout="zipf", align=4 * KIB,
               page=4 * KIB, dirty=0.5, deltas=2, hot=False),
        # Allocations of any byte size (odd ones among them): payload offsets off the
        # 16-byte grid, no straight write-through, unaligned copies both ways.
        _cycle("ragged_1GiB", 1 * GIB, 200, 1 * KIB, 32 * MIB, 64 * KIB, "mixed", align=1),
        # Compressed images of fp32 state in device memory: encode and decode.
        _cycle("coded_f32_2GiB", 2 * GIB, 256, 4 * KIB, 32 * MIB, 64 * KIB, "f32", coded=True),
        # Speculative execution: run ahead, then go back to the saved image in place,
        # rewriting only what differs.
        _cycle("rollback_2GiB", 2 * GIB, 256, 4 * KIB, 32 * MIB, 64 * KIB, "f32", op="rollback", incremental=True),
        # The allocation-free pass, as an allocator hook runs it.
        _cycle("noalloc_1GiB", 1 * GIB, 128, 4 * KIB, 32 * MIB, 64 * KIB, "f32", op="noalloc"),
        # Configuration 5: process contexts of log-uniform sizes through the request server.
        _cycle("serve_16x512MiB", 512 * MIB, 16, 8 * MIB, 128 * MIB, 64 * KIB, "f32", op="serve", host=True, slots=8),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    op = rng.choice(["cycle"] * 6 + ["rollback", "noalloc", "serve"])
    host = rng.random() < 0.35 if op != "noalloc" else False
    coded = op in ("cycle", "rollback") and rng.random() < 0.3
    most = 1 * GIB if host or op in ("noalloc", "serve") else 2 * GIB if coded else 8 * GIB
    total = int(_log(rng, 16 * MIB, most))
    chunk = rng.choice([4 * KIB, 64 * KIB, 64 * KIB, 256 * KIB])
    if op == "serve":
        n, lo, hi = rng.randrange(4, 17), total // 64, total // 2
    else:
        n = int(_log(rng, 1, min(2048, total // (8 * KIB))))
        lo = rng.choice([258, 4 * KIB])
        hi = max(2 * total // n, min(total, 64 * MIB))
    return {"op": op, "total": total, "n": n, "lo": lo, "hi": hi, "align": rng.choice([1, 2, 16, 256, 256, 4096]),
            "chunk": chunk, "content": rng.choice(["u32", "f32", "bf16", "mixed"]),
            "page": min(chunk, rng.choice([4 * KIB, 64 * KIB])), "dirty": rng.choice([0.0, 0.01, 0.1, 0.25, 0.5, 1.0]),
            "hot": rng.random() < 0.5, "deltas": rng.randrange(1, 4), "host": host, "coded": coded,
            "managed": 0.25 if op == "cycle" and rng.random() < 0.15 else 0.0,
            "persist": op == "cycle" and total <= 64 * MIB and rng.random() < 0.5,
            "layout": rng.choice(["loguniform", "zipf"]), "sizes_seed": rng.randrange(1 << 30),
            "incremental": rng.random() < 0.5, "slots": rng.choice([4, 8])}


# ---- inputs -----------------------------------------------------------------

def _sizes(case):
    """Allocation sizes in bytes: raw draws scaled by one factor, clamped to
    [lo, hi], so that they sum to about the total."""
    n, lo, hi, total, align = case["n"], case["lo"], case["hi"], case["total"], case["align"]
    if n == 1:
        return [max(align, total // align * align)]
    rng = np.random.default_rng(case["sizes_seed"])
    if case["layout"] == "zipf":
        ranks = np.arange(1, (1 << 20) + 1, dtype=np.float64)
        cdf = np.cumsum(ranks ** -1.1)
        raw = 1.0 + np.searchsorted(cdf / cdf[-1], rng.uniform(0.0, 1.0, n))
    else:
        raw = np.exp(rng.uniform(math.log(4 * KIB), math.log(64 * MIB), n))
    f_lo, f_hi = 0.0, 1.0
    while np.clip(raw * f_hi, lo, hi).sum() < total and f_hi < 1e12:
        f_hi *= 2
    for _ in range(100):
        mid = (f_lo + f_hi) / 2
        f_lo, f_hi = (mid, f_hi) if np.clip(raw * mid, lo, hi).sum() < total else (f_lo, mid)
    return [max(align, int(s) // align * align) for s in np.clip(raw * f_hi, lo, hi)]


class _Managed:
    """A managed block for torch to wrap (torch does not allocate managed memory itself).
    The tensor made of it holds a reference, so the block lives as long as any view of it."""

    def __init__(self, nbytes):
        self.ptr = C.crac_alloc_managed(nbytes)
        self.__cuda_array_interface__ = {"shape": (nbytes // 8,), "typestr": "<i8", "data": (self.ptr, False),
                                         "version": 3, "strides": None}

    def __del__(self):
        try:
            torch.cuda.synchronize()
            C.crac_free_managed(self.ptr)
        except Exception:   # at interpreter exit the driver may be gone
            pass


class _Memory:
    """One process's allocations: ranges of one device block and, for the last
    part of them, of one managed block."""

    def __init__(self, sizes, n_managed):
        n_dev = len(sizes) - n_managed
        self.sizes, self.kinds, at, end = sizes, [], [], [0, 0]
        for i, s in enumerate(sizes):
            m = int(i >= n_dev)
            self.kinds.append(C.CRAC_KIND_MANAGED if m else C.CRAC_KIND_DEVICE)
            at.append((m, end[m]))
            end[m] += -(-s // PLACE) * PLACE
        self.blocks = [torch.zeros(max(end[0], PLACE) // 8, dtype=torch.int64, device="cuda")]
        if n_managed:
            self.blocks.append(torch.as_tensor(_Managed(end[1]), device="cuda").zero_())
        self.at = at
        self.ptrs = [self.blocks[m].data_ptr() + o for m, o in at]

    def fill(self, content, gen):
        for b in self.blocks:
            if content == "f32":
                b.view(torch.float32).normal_(generator=gen)
            elif content == "bf16":
                b.view(torch.bfloat16).normal_(generator=gen)
            else:
                b.random_(-(1 << 62), 1 << 62, generator=gen)
        if content == "mixed":   # random bytes, fp32 values, 64-bit counters, allocation by allocation
            for i, (m, o) in enumerate(self.at):
                words = self.blocks[m][o // 8:(o + self.sizes[i] + 7) // 8]
                if i % 3 == 1:
                    words.view(torch.float32).normal_(generator=gen)
                elif i % 3 == 2:
                    words.random_(0, 1 << 40, generator=gen)

    def register(self, ctx, which=None):
        for i in range(len(self.sizes)) if which is None else which:
            C.crac_ctx_register_alloc(ctx, self.ptrs[i], self.sizes[i], self.kinds[i])

    def rewrites(self, case, count, gen, which=None):
        """`count` lists of page rewrites for the application's steps (device rows of
        pointer, length, XOR mask; masks keep floats' signs and exponents)."""
        which = range(len(self.sizes)) if which is None else which
        size = torch.tensor([self.sizes[i] for i in which], device="cuda")
        base = torch.tensor([self.ptrs[i] for i in which], device="cuda")
        pages = (size + case["page"] - 1) // case["page"]
        first = torch.cumsum(pages, 0) - pages
        n_pages = int(pages.sum())
        k = int(round(case["dirty"] * n_pages))
        if case["dirty"] > 0:
            k = max(k, 1)
        keep = {"f32": 0x007FFFFF, "bf16": 0x007F007F}.get(case["content"], 0xFFFFFFFF)
        out = []
        for _ in range(1 if case["hot"] else count):
            pick = torch.randperm(n_pages, generator=gen, device="cuda")[:k]
            a = torch.searchsorted(first, pick, right=True) - 1
            o = (pick - first[a]) * case["page"]
            mask = torch.randint(0, 1 << 32, (k,), generator=gen, device="cuda") & keep | 1
            out.append(torch.stack([base[a] + o, torch.clamp(size[a] - o, max=case["page"]), mask], 1).contiguous())
        return out * count if case["hot"] else out


def _config(case, total, **kw):
    keep = int((case["deltas"] + 2) * 1.25 * total) + 64 * MIB   # images of one pass, as a program reserves them
    return C.crac_config_default(
        chunk_bytes=case["chunk"], image_residency=C.CRAC_RESIDENCY_HOST if case["host"] else C.CRAC_RESIDENCY_DEVICE,
        flags=(C.CRAC_FLAG_COMPRESS if case["coded"] else 0) |
              (C.CRAC_FLAG_INCREMENTAL_RESTORE if case.get("incremental") else 0),
        reserve_host_bytes=keep if case["host"] else 0, reserve_device_bytes=0 if case["host"] else keep, **kw)


class _State:
    def __init__(self, case):
        self.case, self.ctxs, self.images, self.memory, self.server = case, [], [], [], None

    def __del__(self):
        try:
            torch.cuda.synchronize()
            if self.server:
                C.crac_server_destroy(self.server)
            for i in self.images:
                C.crac_image_release(i)
            for c in self.ctxs:
                C.crac_ctx_destroy(c)
        except Exception:   # at interpreter exit the driver may be gone
            pass


def _step(rows, stream):
    """One step of the application: it rewrites some of its pages."""
    if rows.shape[0]:
        testkit.mutate_xor(rows.data_ptr(), rows.shape[0], stream)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    s = _State(case)
    sizes = _sizes(case)
    total = sum(sizes)
    if case["op"] == "serve":   # each of the n contexts holds four allocations
        sizes = [x for t in sizes for x in (t // 2, t // 4, t // 8, t // 8)]
        sizes = [max(16, x // case["align"] * case["align"]) for x in sizes]
    mem = _Memory(sizes, int(round(case["managed"] * len(sizes))) if case["op"] == "cycle" else 0)
    mem.fill(case["content"], gen)
    s.memory.append(mem)
    s.stream = torch.cuda.Stream()
    if case["op"] == "noalloc":
        _prepare_noalloc(s, case, mem, gen)
    elif case["op"] == "serve":
        s.server = C.crac_server_create(workers=case["slots"], staging_budget=2 * GIB)
        s.streams, s.steps = [], []
        for i in range(case["n"]):
            which = range(4 * i, 4 * i + 4)
            ctx = C.crac_ctx_create(_config(case, total if i == 0 else 1))
            mem.register(ctx, which)
            s.ctxs.append(ctx)
            s.streams.append(torch.cuda.Stream())
            s.steps.append(mem.rewrites(dict(case, hot=False), 2, gen, which))
    else:
        s.ctxs.append(C.crac_ctx_create(_config(case, total)))
        mem.register(s.ctxs[0])
        s.steps = mem.rewrites(case, case["deltas"], gen)
        torch.cuda.synchronize()
        if case["op"] == "rollback":   # the saved image and its fingerprints
            s.images.append(C.crac_ctx_checkpoint(s.ctxs[0], s.stream))
            C.crac_image_wait(s.images[0])
        else:                          # the restarted process: its own allocations, nothing in them yet
            again = _Memory(sizes, mem.kinds.count(C.CRAC_KIND_MANAGED))
            s.memory.append(again)
            s.ctxs.append(C.crac_ctx_create(_config(case, 1)))
            again.register(s.ctxs[1])
            if case["persist"]:
                s.file = np.zeros(total + total // 8 + MIB, dtype=np.uint8)
    torch.cuda.synchronize()
    return s


def _prepare_noalloc(s, case, mem, gen):
    S = case["chunk"]
    counts = [-(-b // S) for b in mem.sizes]
    first = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    n, total = int(first[-1]), sum(mem.sizes)
    rows = np.stack([np.array(mem.ptrs), np.array(mem.sizes), first[:-1], first[:-1]], 1).astype(np.int64)
    s.regions, s.n, s.total = torch.from_numpy(rows).cuda(), n, total

    def outputs(cap):
        return {"fp": torch.zeros(n, dtype=torch.int64, device="cuda"),
                "idx": torch.zeros(n, dtype=torch.int64, device="cuda"),
                "off": torch.zeros(n + 1, dtype=torch.int64, device="cuda"),
                "staging": torch.zeros((cap + 7) // 8, dtype=torch.int64, device="cuda"),
                "totals": torch.zeros(3, dtype=torch.int64, device="cuda")}

    s.full, s.delta = outputs(total), outputs(total)
    before = outputs(total)   # the baseline: fingerprints taken before the application's last step
    _noalloc(s, None, before)
    torch.cuda.synchronize()
    s.baseline = before["fp"]
    _step(mem.rewrites(case, 1, gen)[0], None)


def _noalloc(s, fp_old, o):
    # On the default stream: calls share one scratch area and must not overlap.
    C.crac_pass_noalloc(s.regions, s.regions.shape[0], s.n, s.case["chunk"], fp_old, o["fp"], o["idx"], o["off"], s.n,
                        o["staging"], s.total, o["totals"], None)


# ---- one pass -----------------------------------------------------------------

def run(s):
    return {"cycle": _run_cycle, "rollback": _run_rollback, "noalloc": _run_noalloc, "serve": _run_serve}[s.case["op"]](s)


def _run_cycle(s):
    a, b = s.ctxs
    C.crac_ctx_invalidate(a)
    images = [C.crac_ctx_checkpoint(a, s.stream)]
    for rows in s.steps:
        _step(rows, s.stream)
        images.append(C.crac_ctx_checkpoint(a, s.stream))
    out = {}
    if s.case["persist"]:   # fingerprints, chunk list and payload of the delta (its header holds addresses)
        at = 80 + 40 * len(s.memory[0].sizes)
        n = C.crac_image_info(images[-1])["serialized_bytes"] - at
        out["file"] = C.crac_image_read(images[-1], at, n, s.file[:n])
    C.crac_ctx_restart(b, images[-1], s.stream)
    for key in ("k", "payload_bytes", "raw_bytes", "n_chunks"):
        out[key] = [C.crac_image_info(i)[key] for i in images]
    for ctx in s.ctxs:
        C.crac_ctx_drop_history(ctx)
    for i in images:
        C.crac_image_release(i)
    return dict(out, memory=s.memory[1].blocks)


def _run_rollback(s):
    _step(s.steps[0], s.stream)
    C.crac_ctx_restart(s.ctxs[0], s.images[0], s.stream)
    return {"memory": s.memory[0].blocks, "rewritten": C.crac_ctx_last_restart(s.ctxs[0])["chunks_rewritten"]}


def _run_noalloc(s):
    _noalloc(s, None, s.full)
    _noalloc(s, s.baseline, s.delta)
    return {"full": s.full, "delta": s.delta}


def _run_serve(s):
    def collect(tickets):
        got = [C.crac_server_wait(s.server, t) for t in tickets]
        if any(r["status"] for r in got):
            raise RuntimeError("request failed: " + C.crac_status_str(next(r["status"] for r in got if r["status"])))
        return got

    def checkpoints():
        return collect([C.crac_server_submit(s.server, c, C.CRAC_REQ_CHECKPOINT, stream=st)
                        for c, st in zip(s.ctxs, s.streams)])

    for c in s.ctxs:
        C.crac_ctx_invalidate(c)
    got = checkpoints()
    images = [r["image"] for r in got]
    for steps, st in zip(s.steps, s.streams):
        _step(steps[0], st)
    new = checkpoints()
    images += [r["image"] for r in new]
    back = range(0, len(s.ctxs), 3)
    for i in back:   # these processes are rolled back to their newest image after running on
        _step(s.steps[i][1], s.streams[i])
    collect([C.crac_server_submit(s.server, s.ctxs[i], C.CRAC_REQ_RESTART, new[i]["image"], s.streams[i]) for i in back])
    for c in s.ctxs:
        C.crac_ctx_drop_history(c)
    for i in images:
        C.crac_image_release(i)
    return {"memory": s.memory[0].blocks, "payload": [r["payload_bytes"] for r in got + new]}


# ---- what a pass cannot do without --------------------------------------------

def work(case):
    sizes, S, page = _sizes(case), case["chunk"], case["page"]
    B = sum(sizes)
    n = sum(-(-b // S) for b in sizes)
    pages = case["dirty"] * B                                    # bytes the application rewrites in a step
    D = B * (1 - (1 - case["dirty"]) ** (max(1, S // page)))     # bytes of the chunks those lie in
    step, full, delta, restart = 2 * pages, 2 * B + 8 * n, B + D + 16 * n, 2 * B
    if case["op"] == "cycle":
        return {"bytes": full + case["deltas"] * (step + delta) + restart + (D + 8 * n if case["persist"] else 0),
                "flops": 0}
    if case["op"] == "rollback":
        return {"bytes": step + (B + 2 * D + 16 * n if case.get("incremental") else restart), "flops": 0}
    if case["op"] == "noalloc":
        return {"bytes": full + delta, "flops": 0}
    return {"bytes": full + step + delta + (step + restart) / 3, "flops": 0}
