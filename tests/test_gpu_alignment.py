"""GPU parity of the wide paths for buffers off a 16-byte boundary, at the
sizes where they can go wrong: lengths around a vector, a unit and a tile, and
every kind of offset of either side."""
import numpy as np
import pytest
import torch

import oracle
from paper_2607_21686_gb300 import pcs
from helpers import np_view, u64

pytestmark = pytest.mark.gpu

OFFSETS = [0, 1, 2, 3, 4, 7, 8, 11, 12, 15]


def _arena(n, seed, dev):
    h = torch.randint(0, 256, (n,), generator=torch.Generator().manual_seed(seed), dtype=torch.uint8)
    return h, h.to(dev)


@pytest.mark.parametrize("oa", OFFSETS)
def test_mismatch_of_offset_pairs(ctx, dev, oa):
    # Differences at the first and the last byte of a pair and in between.
    sizes = [0, 1, 5, 15, 16, 17, 31, 32, 33, 47, 48, 63, 2047, 2048, 2049, 2064, 2079, 4096 + 15,
             6 * 2048 + 16, 70001]
    ha, da = _arena(70100, 1, dev)
    a, b, want = [], [], []
    for ob in OFFSETS:
        for n in sizes:
            hb = ha[oa:oa + n].clone()
            for at in {0, n - 1, n // 2, n // 3, n - 16, n - 17, 16}:
                if 0 <= at < n:
                    hb[at] ^= 1 + (at + ob) % 255
            full = torch.zeros(ob + n + 3, dtype=torch.uint8)
            full[ob:ob + n] = hb
            a.append(da[oa:oa + n])
            b.append(full.to(dev)[ob:ob + n])
            want.append(int((hb != ha[oa:oa + n]).sum()))
            assert want[-1] == oracle.mismatch(ha[oa:oa + n].numpy(), hb.numpy())
    assert ctx.mismatch(a, b).cpu().tolist() == want
    assert ctx.mismatch(a, b).cpu().tolist() == want  # the scratch sums start over


# Calls of few pairs have their plan with the launch, in two sizes; more pairs
# have it in the workspace.
@pytest.mark.parametrize("n", [1, 64, 65, 512, 513, 1500])
def test_mismatch_of_many_pairs(ctx, dev, n):
    rnd = np.random.default_rng(n)
    ha, da = _arena(200000, 11, dev)
    hb = ha.clone()
    hb[torch.from_numpy(rnd.integers(0, 200000, 20000))] ^= 0x40
    db = hb.to(dev)
    for _ in range(2):  # the scratch sums start over
        a, b, want = [], [], []
        for i in range(n):
            m = 0 if i % 7 == 3 else int(np.exp(rnd.uniform(0, 9.5)))
            o, extra = int(rnd.integers(0, 150000)), (i % 3) * 5
            a.append(da[o:o + m])
            b.append(db[o:o + m + extra])
            want.append(int((ha[o:o + m] != hb[o:o + m]).sum()) + extra)
        assert ctx.mismatch(a, b).cpu().tolist() == want
        shift = [int(x) for x in rnd.integers(0, 16, n)]  # and other offsets of b
        b = [db[s:s + len(x)] for s, x in zip(shift, a)]
        want = [int((ha[x.storage_offset():x.storage_offset() + len(x)] != hb[s:s + len(x)]).sum())
                for s, x in zip(shift, a)]
        assert ctx.mismatch(a, b).cpu().tolist() == want


def _read_flags(spans, ro, rn):
    """1 for each (start, bytes) some read [ro, ro + rn) of at least one byte overlaps."""
    ro, rn = ro[rn > 0], rn[rn > 0]
    return [int(n > 0 and bool(((ro < o + n) & (ro + rn > o)).any())) for o, n in spans]


# Buffers: one; few and many staged in shared memory; the most staged and one
# more; more flags than one round of the block that writes them.  Reads: below and above the line where the address table is used.
@pytest.mark.parametrize("n,m", [(1, 40), (33, 3_000_001), (600, 2_600_000), (4096, 2_500_000),
                                 (4096, 5000), (4097, 5000), (8192, 900), (8193, 5000), (20011, 3000)])
def test_classify_reads_paths(ctx, dev, n, m):
    rnd = np.random.default_rng(n + m)
    size = 1 << 26
    space = torch.empty(size, dtype=torch.uint8, device=dev)
    start = rnd.integers(0, size // 2, n)
    length = np.minimum(np.exp(rnd.uniform(0, 16, n)).astype(np.int64), size - start)
    length[rnd.random(n) < 0.1] = 0          # empty buffers
    length[0] = max(length[0], 1)
    # Reads around a few places, before the first buffer and after the last.
    at = rnd.integers(0, size // 2, 12)
    ro = (at[rnd.integers(0, 12, m)] + rnd.integers(-2000, 2000, m)).clip(0, size - 1)
    ro[:: 5] = size - 1 - rnd.integers(0, 1000, len(ro[:: 5]))
    rn = rnd.integers(0, 200, m)
    rn[:: 1001] = 0
    base = space.data_ptr()
    addr = torch.from_numpy(base + ro).to(dev)
    flags = torch.full((n,), 7, dtype=torch.uint8, device=dev)
    bufs = [space[o:o + k] for o, k in zip(start.tolist(), length.tolist())]
    ctx.classify_reads(bufs, addr, torch.from_numpy(rn).to(dev), flags)
    pick = rnd.permutation(n)[:150].tolist() if m > 100000 else range(n)
    got = flags.cpu().tolist()
    spans = list(zip(start.tolist(), length.tolist()))
    assert set(got) <= {0, 1}
    assert [got[i] for i in pick] == _read_flags([spans[i] for i in pick], ro, rn)


# Sections off a 16-byte boundary, pairs of chunks per task (more than 40 MB in
# the register kernel) and single ones: lengths around chunks and tiles, restored
# to another offset with guard bytes around every target.
@pytest.mark.parametrize("big", [0, 24])
def test_offset_sections_round_trip(ctx, dev, big):
    sizes = [1, 15, 16, 17, 4095, 4096, 4097, 8191, 8192, 8193, 8192 + 4096, 3 * 8192 - 5,
             3 * 8192 + 15, 5 * 8192, 100003]
    sizes = [n for n in sizes for _ in OFFSETS] + [2 * 1024 * 1024 + 11 * i for i in range(big)]
    need = sum(sizes) + 64 * len(sizes)
    host, src = _arena(need, 5, dev)
    dst = torch.full((need,), 0xA5, dtype=torch.uint8, device=dev)
    at, to, secs_a, secs_b, aligned, used = 0, 0, [], [], [], torch.zeros(need, dtype=torch.bool)
    views = []
    for i, n in enumerate(sizes):
        oa, ob = OFFSETS[i % len(OFFSETS)], OFFSETS[(7 * i + 3) % len(OFFSETS)]
        at, to = (at + 15) // 16 * 16 + 16 + oa, (to + 15) // 16 * 16 + 16 + ob
        views.append((at, to, n))
        used[to:to + n] = True
        secs_a.append(pcs.contig_section(9, src[at:at + n]))
        secs_b.append(pcs.contig_section(9, dst[to:to + n]))
        aligned.append(src[at:at + n].clone())
        at, to = at + n, to + n
    snap = ctx.checkpoint([pcs.Session(1, 9, secs_a, keep=[src])])[0]
    want = u64(ctx.fingerprint(aligned))
    assert [ctx.section(snap, i).fp for i in range(len(sizes))] == want
    assert want[:20] == [oracle.fingerprint(host[a:a + n].numpy()) for a, _, n in views[:20]]
    assert u64(ctx.fingerprint([src[a:a + n] for a, _, n in views])) == want
    for verify in (False, True):
        dst.fill_(0xA5)
        ctx.restore([snap], [pcs.Session(1, 9, secs_b, keep=[dst])], verify=verify)
        got = dst.cpu()
        for a, t, n in views:
            assert torch.equal(got[t:t + n], host[a:a + n]), (a, t, n)
        assert bool((got[~used] == 0xA5).all())
    ctx.delete(snap)
    ctx.sync()


# Small calls, finalised by the warps that complete their items: one and many
# sessions, one section and 32 (and 33, finalised by the last block), sections
# of no task beyond their first chunk; the counters start over at every call.
@pytest.mark.parametrize("n,secs", [(1, 1), (1, 32), (1, 33), (64, 2), (63, 5), (7, 40), (64, 32)])
def test_small_calls_of_many_items(ctx, dev, n, secs):
    rnd = np.random.default_rng(100 * n + secs)
    size = rnd.integers(0, 2 * (1 << 20) // (3 * n * secs) + 2, (n, secs))
    size[0, 0] = 0
    host, src = _arena(int(size.sum()) + 16 * size.size, 9, dev)
    dst = torch.zeros_like(src)
    at, spans = 0, []
    for b in size.reshape(-1).tolist():
        at = (at + 3) // 4 * 4 if b % 3 else at
        spans.append((at, b))
        at += b
    mk = lambda t: [pcs.Session(s, 9, [pcs.contig_section(1 + i, t[o:o + b]) for i, (o, b) in
                                       enumerate(spans[s * secs:(s + 1) * secs])], keep=[t])
                    for s in range(n)]
    want = [oracle.fingerprint(host[o:o + b].numpy()) for o, b in spans]
    for _ in range(2):
        snaps = ctx.checkpoint(mk(src))
        got = [ctx.section(s, i).fp for s in snaps for i in range(secs)]
        assert got == want
        dst.zero_()
        ctx.restore(snaps, mk(dst), verify=True)
        for o, b in spans:
            assert torch.equal(dst[o:o + b].cpu(), host[o:o + b])
        for s in snaps:
            ctx.delete(s)
        if n * secs <= 64:
            views = [src[o:o + b] for o, b in spans]
            assert u64(ctx.fingerprint(views)) == want
    # A wrong byte in one record is found.
    snap = ctx.checkpoint(mk(src))
    victim = int(np.argmax(size.sum(1)))
    sec = int(np.argmax(size[victim]))
    if size[victim, sec]:
        path = "/tmp/pcs_small_%d_%d.bin" % (n, secs)
        ctx.write_file(snap[victim], path)
        raw = bytearray(open(path, "rb").read())
        raw[ctx.section(snap[victim], sec).offset] ^= 1
        open(path, "wb").write(raw)
        bad = ctx.read_file(path)
        ctx.delete(snap[victim])
        snap[victim] = bad
        assert ctx.restore_status(snap, mk(dst)) == pcs.PCS_E_CORRUPT
    for s in snap:
        ctx.delete(s)


# Rings of rows below 512 bytes, walked by whole pages: pages of one row to many
# (below and above 512 bytes, powers of two and not), first rows at and inside a
# page, in a call large enough for the bulk-copy kernel.
@pytest.mark.parametrize("row,page_rows", [(16, 8), (16, 100), (48, 16), (128, 3), (128, 16),
                                           (256, 1), (256, 16), (496, 2), (496, 33)])
def test_rings_of_short_rows(ctx, dev, row, page_rows):
    pages = max(2, (1 << 18) // (row * page_rows))
    window = pages * page_rows
    starts = [0, 1, page_rows - 1, page_rows, window // 2 + 1, window - 1]
    host, pool = _arena(len(starts) * pages * page_rows * row, 3, dev)
    shape = (len(starts) * pages, page_rows, row)
    pool, host = pool.view(shape), host.view(shape)
    g = torch.Generator().manual_seed(row + page_rows)
    tab = torch.randperm(shape[0], generator=g).to(torch.int32).view(len(starts), pages)
    tab2 = torch.randperm(shape[0], generator=g).to(torch.int32).view(len(starts), pages)
    dt, dt2 = tab.to(dev), tab2.to(dev)
    out = torch.zeros_like(pool)

    def sessions(p, t, from_snapshot):
        return [pcs.Session(i, pcs.PCS_KIND_KV, [pcs.ring_section(
            pcs.PCS_SEC_K, p, t[i], pcs.PCS_RING_START_FROM_SNAPSHOT if from_snapshot else s,
            window)], keep=[p, t]) for i, s in enumerate(starts)]

    snaps = ctx.checkpoint(sessions(pool, dt, False))
    ctx.restore(snaps, sessions(out, dt2, True), verify=True)
    for i, s in enumerate(starts):
        slot = (s + torch.arange(window)) % window
        rows = host[tab[i].long()[slot // page_rows], slot % page_rows]
        assert ctx.section(snaps[i], 0).fp == oracle.fingerprint(rows.contiguous().view(-1).numpy())
        assert torch.equal(out.cpu()[tab2[i].long()[slot // page_rows], slot % page_rows], rows)
        ctx.delete(snaps[i])
    ctx.sync()


# The score kernel's shapes at their edges: keys that fill an entry's lanes and
# that leave some idle, banks shorter and longer than a round of entries and not
# multiples of one, narrower banks beside wider ones in a call.
@pytest.mark.parametrize("dims", [(8,), (56,), (64,), (72,), (120, 128), (136,), (248, 256), (264,),
                                  (504, 512), (520,), (760, 768, 8), (776,), (1016, 1024, 64)])
@pytest.mark.parametrize("dtype", [torch.float16, torch.bfloat16])
def test_scores_of_every_shape(ctx, dev, dims, dtype):
    g = torch.Generator().manual_seed(sum(dims))
    sizes = [1, 2, 3, 7, 8, 9, 15, 16, 17, 31, 32, 33, 0, 65, 127, 700]
    keys, queries = [], []
    for i, n in enumerate(sizes):
        d = dims[i % len(dims)]
        k = torch.randn(n, d, generator=g).to(dtype)
        if n > 2:
            k[1] = 0                     # a zero norm scores 0
            k[2] = torch.finfo(dtype).max  # sums past the largest float
        keys.append(k)
        queries.append(torch.randn(d, generator=g).to(dtype))
    dk, dq = [k.to(dev) for k in keys], [q.to(dev) for q in queries]
    banks = ctx.banks_array(dk, dq, [100 + 16 * (i % 3) for i in range(len(sizes))])
    want = np.concatenate([oracle.scores(np_view(q), np_view(k)) for q, k in zip(queries, keys)
                           if len(k)])
    total = sum(sizes)
    kept, off = (torch.zeros(n, dtype=torch.int32, device=dev) for n in (total, len(sizes) + 1))
    for budget in (None, 60 * total):
        scores = torch.full((total,), 7.0, device=dev)
        if budget is None:
            ctx.prune(banks, len(sizes), ctx.params(pcs.PCS_K_FIXED, k_max=1 << 20), kept, off, scores)
        else:
            ctx.prune_global(banks, len(sizes), budget, kept, off, scores)
        got = scores.cpu().numpy()
        nan = np.isnan(want)  # which NaN is not defined
        assert np.array_equal(np.isnan(got), nan)
        assert np.array_equal(got[~nan].view(np.uint32), want[~nan].view(np.uint32))


# The one-block global threshold at its limits (16,384 entries, 1,024 banks) and
# just past them: runs of ties across threads and banks, banks of one entry and
# empty ones, entry bytes of no byte, of few and past 32 bits.
@pytest.mark.parametrize("entries,n_banks", [(1, 1), (15, 3), (16, 16), (16384, 1), (16385, 1),
                                             (16384, 1024), (16380, 1025), (5000, 700)])
@pytest.mark.parametrize("kind", ["uniform", "mixed", "wide"])
def test_global_threshold_of_small_populations(ctx, dev, entries, n_banks, kind):
    rnd = np.random.default_rng(entries + n_banks)
    cuts = np.sort(rnd.integers(0, entries + 1, n_banks - 1))
    sizes = np.diff(np.concatenate([[0], cuts, [entries]])).tolist()
    pick = torch.randn(40, 16, generator=torch.Generator().manual_seed(entries)).half()
    keys = [pick[torch.from_numpy(rnd.integers(0, 40, s))] for s in sizes]
    q = pick[3] + pick[5]
    eb = {"uniform": [48] * n_banks, "mixed": rnd.integers(0, 5000, n_banks).tolist(),
          "wide": ((1 << 32) + rnd.integers(-2, 1 << 20, n_banks)).tolist()}[kind]
    s32 = np.concatenate([oracle.scores(np_view(q), np_view(k)) for k in keys if len(k)])
    dk, dq = [k.to(dev) for k in keys], q.to(dev)
    banks = ctx.banks_array(dk, [dq] * n_banks, eb)
    total = sum(a * b for a, b in zip(sizes, eb))
    for budget in sorted({0, min(eb), total // 3, total * 2 // 3 + 1, max(total - 1, 0), total}):
        kept = torch.full((entries,), -7, dtype=torch.int32, device=dev)
        off = torch.full((n_banks + 1,), -7, dtype=torch.int32, device=dev)
        ctx.prune_global(banks, n_banks, budget, kept, off)
        want, woff = oracle.prune_global(s32, sizes, eb, budget)
        assert off.cpu().tolist() == woff.tolist(), budget
        assert kept.cpu().tolist()[:woff[-1]] == want.tolist(), budget
    ctx.sync()


# The cooperative global threshold at the sizes where its launch shape changes on
# 152 SMs: 456 and 608 tiles of 4,096 entries fill three and four blocks per SM
# (one tile more: two tiles a block), 912 and 1,216 their second rounds.
@pytest.mark.parametrize("entries", [456 * 4096, 456 * 4096 + 1, 608 * 4096, 608 * 4096 + 1,
                                     912 * 4096 + 1, 1216 * 4096 + 5])
@pytest.mark.parametrize("kind", ["uniform", "mixed"])
def test_global_threshold_at_launch_shape_edges(ctx, dev, entries, kind):
    rnd = np.random.default_rng(entries)
    sizes = np.diff(np.concatenate([[0], np.sort(rnd.integers(0, entries, 8)), [entries]])).tolist()
    eb = [48] * 9 if kind == "uniform" else rnd.integers(1, 5000, 9).tolist()
    gen = torch.Generator(device=dev).manual_seed(entries)
    keys = torch.randn(entries, 8, generator=gen, device=dev).half()
    q = torch.randn(8, generator=gen, device=dev).half()
    cuts = np.cumsum([0] + sizes)
    banks = ctx.banks_array([keys[a:b] for a, b in zip(cuts[:-1], cuts[1:])], [q] * 9, eb)
    scores = torch.empty(entries, dtype=torch.float32, device=dev)
    total = sum(a * b for a, b in zip(sizes, eb))
    for budget in (total * 2 // 3 + 1, total // 50):
        kept = torch.full((entries,), -7, dtype=torch.int32, device=dev)
        off = torch.full((10,), -7, dtype=torch.int32, device=dev)
        ctx.prune_global(banks, 9, budget, kept, off, scores)
        want, woff = oracle.prune_global(scores.cpu().numpy(), sizes, eb, budget)
        assert off.cpu().tolist() == woff.tolist(), budget
        assert np.array_equal(kept.cpu().numpy()[:woff[-1]], want), budget
    ctx.sync()


# Top-k with and without the lists' offsets, by banks that travel with the launch
# and banks in the workspace: empty banks, nothing kept, all kept, ties.
@pytest.mark.parametrize("n_banks", [1, 60, 61, 300])
def test_topk_with_and_without_offsets(ctx, dev, n_banks):
    rnd = np.random.default_rng(n_banks)
    n = [int(x) for x in rnd.integers(0, 70, n_banks)]
    n[0] = 5000  # past what a block keeps in registers
    k = [int(rnd.integers(0, x + 2)) if i % 4 else (0, x)[i % 8 == 0] for i, x in enumerate(n)]
    k[0] = 1777
    keys = (rnd.integers(0, 40, sum(n)) / 8).astype(np.float32)
    dk = torch.from_numpy(keys).to(dev)
    cuts, want = np.cumsum([0] + n), []
    kept = [min(a, b) for a, b in zip(n, k)]
    for a, b, x in zip(cuts[:-1], cuts[1:], kept):
        want += oracle.topk(keys[a:b], x).tolist()
    for with_off in (True, False):
        out = torch.full((sum(kept) + 1,), -7, dtype=torch.int32, device=dev)
        off = torch.full((n_banks + 1,), -7, dtype=torch.int32, device=dev) if with_off else None
        ctx.topk(dk, n, k, out, off)
        assert out.cpu().tolist() == want + [-7]
        if with_off:
            assert off.cpu().tolist() == np.cumsum([0] + kept).tolist()
