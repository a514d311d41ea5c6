"""The calls whose time is measured: what a program that keeps sessions with
this library has it do, through the public binding, over the sizes it meets.

A case is a dict of plain values.  `kind` names the path:

  markov    checkpoint, verified restore and delete of uint8 observations with
            their 16-byte generator state, planned once or call by call
  bank      prune memory banks by relevance, checkpoint the kept entries to
            HBM or to pinned host memory, restore them into compacted banks,
            delete
  kv        checkpoint paged ring windows of a KV context, restore them into
            other pages, delete; with `fork`, the restore reads a fork
  classify  fingerprint buffers after a recompute and compare with before
  mismatch  the discovery distance: differing bytes of buffer pairs
  prune     relevance scores and per-bank top-k of a mass suspend
  global    one relevance threshold across all banks
  reads     which buffers a log of reads touched (state versus witness)

Sizes inside a population (entries per bank, bytes per buffer) come from the
case alone, so every seed of a case has the same shapes; contents come from
the seed.
"""
import math
import random

import torch

from paper_2607_21686_gb300 import pcs

_DEV = "cuda:0"
_MIB = 1 << 20
_ctx = None

# A bank's key types and the element types of a runtime's buffers.
_KEY_DTYPES = {"fp16": torch.float16, "bf16": torch.bfloat16}
_ELEMENT_BYTES = (1, 8, 2, 2, 4)  # u8, i64, f16, bf16, f32


def _context():
    """The one context a program keeps for its lifetime."""
    global _ctx
    if _ctx is None:
        _ctx = pcs.Context(0)
    return _ctx


# ---------------------------------------------------------------------------
# The cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # One Markovian session suspended and resumed between two requests:
        # latency of the smallest calls.
        dict(name="markov_one", kind="markov", sessions=1, height=256, width=256, planned=False),
        # The periodic checkpoint of every Markovian session a server holds.
        dict(name="markov_4096", kind="markov", sessions=4096, height=256, width=256, planned=True),
        # Memory banks of a world model with 32 KiB latents, cut to 128 entries.
        dict(name="bank_64", kind="bank", sessions=64, n_lo=1, n_hi=512, key_dim=256,
             key_dtype="fp16", value_bytes=32768, keep=0.0, k_max=128, kept_align=4,
             planned=False, host=False, sizes=2),
        # Sixteen banks of about 26 frames of 37 KB with short keys, halved
        # under a host budget and suspended to pinned host memory; kept lists
        # back to back (the default).
        dict(name="bank_16", kind="bank", sessions=16, n_lo=21, n_hi=26, key_dim=64,
             key_dtype="bf16", value_bytes=36928, keep=0.5, k_max=0, kept_align=1,
             planned=False, host=True, sizes=5),
        # Windowed KV contexts of 16 heads: the largest call.
        dict(name="kv_32", kind="kv", sessions=32, layers=24, heads=16, head_dim=64, window=1024,
             page_rows=16, fork=False),
        # A planner branches contexts of grouped-query attention (2 KV heads):
        # checkpoint, fork, resume the fork.
        dict(name="kv_fork_8", kind="kv", sessions=8, layers=24, heads=2, head_dim=64, window=1024,
             page_rows=16, fork=True),
        # The classification sweep: 200 separately allocated buffers.
        dict(name="classify_200", kind="classify", buffers=200, lo=64, hi=256 * _MIB, packed=False,
             sizes=4),
        # The same decision over buffers carved back to back out of one arena,
        # each only as aligned as its element type.
        dict(name="classify_packed", kind="classify", buffers=200, lo=64, hi=16 * _MIB,
             packed=True, sizes=7),
        # One probe of the discovery procedure over buffers of one arena.
        dict(name="mismatch_64", kind="mismatch", buffers=64, lo=64, hi=16 * _MIB, packed=True,
             sizes=9),
        # Relevance pruning of a mass suspend under a host budget.
        dict(name="prune_2048", kind="prune", banks=2048, n_lo=256, n_hi=4096, key_dim=512,
             key_dtype="bf16", value_bytes=2048, keep=0.6, sizes=5),
        # One threshold across banks whose entries cost different bytes.
        dict(name="global_256", kind="global", banks=256, n_lo=64, n_hi=2048, key_dim=128,
             key_dtype="fp16", value_bytes=4096, keep=0.4, mixed=True, sizes=6),
        # A read log of 16M ranges over 140 of 200 buffers.
        dict(name="reads_16m", kind="reads", reads=1 << 24, buffers=200, lo=64, hi=64 * _MIB,
             sizes=4),
    ]


def _log(rng, lo, hi):
    """A whole number in [lo, hi], spread evenly over its logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("markov", "bank", "kv", "classify", "mismatch", "prune", "global", "reads"))
    if kind == "markov":
        return dict(kind=kind, sessions=_log(rng, 1, 4096), height=rng.randint(33, 256),
                    width=rng.randint(33, 256), planned=rng.random() < 0.5)
    if kind == "bank":
        c = dict(kind=kind, n_lo=1, n_hi=_log(rng, 8, 1024),
                 key_dim=rng.choice((64, 96, 128, 256, 264, 512)),
                 key_dtype=rng.choice(("fp16", "bf16")), value_bytes=16 * _log(rng, 16, 2308),
                 keep=rng.choice((0.25, 0.5, 0.75)), k_max=0, kept_align=rng.choice((1, 4)),
                 planned=rng.random() < 0.3, host=rng.random() < 0.3,
                 sizes=rng.randint(0, 10 ** 6))
        entry = 2 * c["key_dim"] + c["value_bytes"]
        most = max(1, min(512, (128 if c["host"] else 1024) * _MIB // (entry * c["n_hi"])))
        c["sessions"] = _log(rng, 1, most)
        return c
    if kind == "kv":
        c = dict(kind=kind, layers=rng.randint(4, 30), heads=rng.choice((1, 2, 4, 8, 16)),
                 head_dim=rng.choice((64, 128)), page_rows=rng.choice((16, 32)),
                 fork=rng.random() < 0.4)
        c["window"] = c["page_rows"] * rng.randint(8, 48)
        session = 4 * c["layers"] * c["window"] * c["heads"] * c["head_dim"]
        c["sessions"] = _log(rng, 1, max(1, min(64, 2048 * _MIB // session)))
        return c
    if kind in ("classify", "mismatch"):
        packed = rng.random() < 0.5
        c = dict(kind=kind, buffers=_log(rng, 8, 512), lo=64, packed=packed,
                 hi=_log(rng, 64 << 10, (16 if packed else 64) * _MIB),
                 sizes=rng.randint(0, 10 ** 6))
        while _total(c) > (512 if packed else 2048) * _MIB:
            c["hi"] //= 2
        return c
    if kind in ("prune", "global"):
        c = dict(kind=kind, n_lo=16, n_hi=_log(rng, 32, 4096),
                 key_dim=rng.choice((64, 128, 256, 264, 512, 768, 1024)),
                 key_dtype=rng.choice(("fp16", "bf16")), value_bytes=16 * _log(rng, 16, 2308),
                 keep=rng.choice((0.25, 0.5, 0.75)), sizes=rng.randint(0, 10 ** 6))
        most = max(1, min(2048, 2048 * _MIB // (2 * c["key_dim"] * c["n_hi"])))
        c["banks"] = _log(rng, 1, most)
        if kind == "global":
            c["mixed"] = rng.random() < 0.5
        return c
    return dict(kind=kind, reads=_log(rng, 4096, 1 << 24), buffers=_log(rng, 8, 2048), lo=64,
                hi=_log(rng, 64 << 10, 64 * _MIB), sizes=rng.randint(0, 10 ** 6))


# ---------------------------------------------------------------------------
# Shapes of a case
# ---------------------------------------------------------------------------

def _entries(case):
    """Entries of each bank."""
    r = random.Random(case["sizes"])
    return [r.randint(case["n_lo"], case["n_hi"]) for _ in range(case.get("sessions") or case["banks"])]


def _kept(case):
    """Entries each bank keeps (the k-rules of the library, Sec. 7.5)."""
    n = _entries(case)
    if case.get("k_max"):
        return [min(x, case["k_max"]) for x in n]
    total, budget = sum(n), _budget(case) // _entry_bytes(case)[0]
    if total <= budget:
        return n
    eb = _entry_bytes(case)[0]
    return [x * _budget(case) // (total * eb) for x in n]


def _entry_bytes(case):
    """Bytes one kept entry of each bank costs."""
    eb = 2 * case["key_dim"] + case["value_bytes"]
    banks = case.get("sessions") or case["banks"]
    if case.get("mixed"):
        return [eb + 64 * (b % 7) for b in range(banks)]
    return [eb] * banks


def _budget(case):
    return int(case["keep"] * sum(n * b for n, b in zip(_entries(case), _entry_bytes(case))))


def _buffers(case):
    """(bytes, element bytes) of each buffer: bytes spread over their logarithm."""
    r = random.Random(case["sizes"])
    out = []
    for _ in range(case["buffers"]):
        b = _log(r, case["lo"], case["hi"])
        es = r.choice(_ELEMENT_BYTES)
        out.append((max(es, b - b % es), es))
    return out


def _total(case):
    return sum(b for b, _ in _buffers(case))


def _offsets(case):
    """(start of each buffer, bytes of the arena): back to back at the element
    type's alignment if packed, else at an allocator's 512 bytes."""
    at, out = 0, []
    for b, es in _buffers(case):
        a = es if case.get("packed") else 512
        at = (at + a - 1) // a * a
        out.append(at)
        at += b
    return out, at


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=_DEV).manual_seed(int(seed))


def _random_bytes(n, g):
    """n random bytes, on 16-byte boundaries."""
    return torch.randint(-2 ** 63, 2 ** 63 - 1, ((n + 7) // 8 + 1,), generator=g, device=_DEV,
                         dtype=torch.int64).view(torch.uint8)[:n]


def _normal(shape, dtype, g):
    """N(0, 1) values, drawn in pieces that bound the fp32 temporary."""
    out = torch.empty(shape, dtype=dtype, device=_DEV)
    flat = out.view(-1)
    step = 1 << 27
    for at in range(0, flat.numel(), step):
        part = flat[at:at + step]
        part.copy_(torch.randn(part.numel(), generator=g, device=_DEV))
    return out


class _State:
    """What a program keeps between calls; prepared calls end with it."""

    def __init__(self, case):
        self.case = case
        self.ctx = _context()
        self.plans, self.handles = [], None

    def __del__(self):
        for p in self.plans:
            self.ctx.plan_destroy(p)
        if self.handles is not None:
            self.ctx.delete_raw(*self.handles)


def _placement(case):
    return pcs.PCS_PLACE_PINNED_HOST if case.get("host") else pcs.PCS_PLACE_DEVICE


def _plan(s):
    """The checkpoint and restore of a state, planned once."""
    cplan, hs = s.ctx.plan_checkpoint(s.source, s.n, _placement(s.case))
    s.handles = (hs, s.n)
    s.plans = [cplan]
    s.plans.append(s.ctx.plan_restore(hs, s.n, s.target, verify=2))


def _prepare_markov(s, case, g):
    S, shape = case["sessions"], (3, case["height"], case["width"])
    nb = math.prod(shape)
    obs = _random_bytes(S * nb, g).view((S,) + shape)
    rng = _random_bytes(16 * S, g).view(torch.int64).view(S, 2)
    s.out = (torch.zeros_like(obs), torch.zeros_like(rng))
    s.n = S
    s.source = s.ctx.session_array([pcs.markov_session(i, obs[i], rng[i]) for i in range(S)])
    s.target = s.ctx.session_array([pcs.markov_session(i, s.out[0][i], s.out[1][i])
                                    for i in range(S)])


def _prepare_banks(s, case, g):
    """Banks of keys (and their queries) stored back to back."""
    n, D = _entries(case), case["key_dim"]
    off = [0]
    for x in n:
        off.append(off[-1] + x)
    s.keys = _normal((off[-1], D), _KEY_DTYPES[case["key_dtype"]], g)
    s.queries = _normal((len(n), D), _KEY_DTYPES[case["key_dtype"]], g)
    s.off = off
    s.bank_keys = [s.keys[off[b]:off[b + 1]] for b in range(len(n))]
    s.n = len(n)
    s.banks = s.ctx.banks_array(s.bank_keys, [s.queries[b] for b in range(len(n))],
                                _entry_bytes(case))


def _prepare_bank(s, case, g):
    _prepare_banks(s, case, g)
    a, V = case["kept_align"], case["value_bytes"]
    if case["k_max"]:
        s.params = s.ctx.params(pcs.PCS_K_FIXED, k_max=case["k_max"], kept_align=a)
    else:
        s.params = s.ctx.params(pcs.PCS_K_BUDGET, budget=_budget(case), kept_align=a)
    ks = s.ctx.prune_counts(s.banks, s.n, s.params)
    at = [0]
    for k in ks:
        at.append(at[-1] + (k + a - 1) // a * a)
    values = _random_bytes(s.off[-1] * V, g).view(s.off[-1], V)
    s.kept = torch.zeros(at[-1], dtype=torch.int32, device=_DEV)
    total = sum(ks)
    # The compacted banks a resume fills: kept lists, keys and values of all.
    s.out = (torch.zeros(at[-1], dtype=torch.int32, device=_DEV),
             torch.zeros((total, case["key_dim"]), dtype=s.keys.dtype, device=_DEV),
             torch.zeros((total, V), dtype=torch.uint8, device=_DEV))
    src, dst, r = [], [], 0
    for b, k in enumerate(ks):
        src.append(pcs.bank_session(b, s.bank_keys[b], values[s.off[b]:s.off[b + 1]],
                                    s.kept[at[b]:at[b] + k]))
        dst.append(pcs.bank_targets(b, s.out[0][at[b]:at[b] + k], s.out[1][r:r + k],
                                    s.out[2][r:r + k]))
        r += k
    s.source, s.target = s.ctx.session_array(src), s.ctx.session_array(dst)


def _prepare_kv(s, case, g):
    S, L, W, pr = case["sessions"], case["layers"], case["window"], case["page_rows"]
    per = W // pr
    pages = S * L * per
    shape = (pages, pr, case["heads"], case["head_dim"])
    pools = [_normal(shape, torch.bfloat16, g) for _ in range(2)]
    meta = _random_bytes(32 * S, g).view(torch.int64).view(S, 4)
    tables = [torch.randperm(pages, generator=g, device=_DEV).to(torch.int32).view(S, L, per)
              for _ in range(2)]
    starts = torch.randint(0, W, (S,), generator=g, device=_DEV).tolist()
    s.out = (torch.zeros_like(meta), torch.zeros_like(pools[0]), torch.zeros_like(pools[1]))
    s.n = S
    s.source = s.ctx.session_array([pcs.kv_session(i, meta[i], pools[0], pools[1], tables[0][i],
                                                   starts[i], W) for i in range(S)])
    s.target = s.ctx.session_array([pcs.kv_session(i, s.out[0][i], s.out[1], s.out[2],
                                                   tables[1][i], pcs.PCS_RING_START_FROM_SNAPSHOT,
                                                   W) for i in range(S)])


def _prepare_buffers(s, case, g):
    """Buffers as first computed, and after a recompute that changed one bit
    of some of them."""
    off, nb = _offsets(case)
    sizes = [b for b, _ in _buffers(case)]
    before = _random_bytes(nb, g)
    after = before.clone()
    flip = torch.rand(len(sizes), generator=g, device=_DEV) < 0.3
    where = (torch.rand(len(sizes), generator=g, device=_DEV, dtype=torch.float64)
             * torch.tensor(sizes, device=_DEV)).long() + torch.tensor(off, device=_DEV)
    after[where[flip]] ^= 4
    s.n = len(sizes)
    s.after = s.ctx.buf_array([after[o:o + b] for o, b in zip(off, sizes)])
    s.before = s.ctx.buf_array([before[o:o + b] for o, b in zip(off, sizes)])
    if case["kind"] == "classify":
        s.fp_before = s.ctx.fingerprint(s.before)
        s.fp_after = torch.zeros(s.n, dtype=torch.int64, device=_DEV)
        s.must = torch.zeros(s.n, dtype=torch.uint8, device=_DEV)
        s.before = None
    else:
        s.counts = torch.zeros(s.n, dtype=torch.int64, device=_DEV)


def _prepare_prune(s, case, g):
    _prepare_banks(s, case, g)
    entries = s.off[-1]
    s.scores = torch.zeros(entries, dtype=torch.float32, device=_DEV)
    s.kept_off = torch.zeros(s.n + 1, dtype=torch.int32, device=_DEV)
    if case["kind"] == "prune":
        s.params = s.ctx.params(pcs.PCS_K_BUDGET, budget=_budget(case))
        kept = sum(s.ctx.prune_counts(s.banks, s.n, s.params))
    else:
        s.budget, kept = _budget(case), entries
    s.kept = torch.zeros(kept, dtype=torch.int32, device=_DEV)


def _prepare_reads(s, case, g):
    off, nb = _offsets(case)
    sizes = [b for b, _ in _buffers(case)]
    arena = torch.empty(nb, dtype=torch.uint8, device=_DEV)
    s.n, m = len(sizes), case["reads"]
    s.bufs = s.ctx.buf_array([arena[o:o + b] for o, b in zip(off, sizes)])
    lens = torch.tensor(sizes, device=_DEV)
    base = torch.tensor(off, device=_DEV) + arena.data_ptr()
    # A resume reads 70 % of the buffers, each range inside its buffer.
    which = torch.randperm(s.n, generator=g, device=_DEV)[:max(1, s.n * 7 // 10)]
    which = which[torch.randint(0, which.numel(), (m,), generator=g, device=_DEV)]
    at = (torch.rand(m, generator=g, device=_DEV) * lens[which]).long().clamp(max=lens[which] - 1)
    s.addr = base[which] + at
    s.nbytes = torch.minimum(torch.randint(1, 4097, (m,), generator=g, device=_DEV),
                             lens[which] - at)
    s.flags = torch.zeros(s.n, dtype=torch.uint8, device=_DEV)


def prepare(case, seed):
    s, g = _State(case), _gen(seed)
    {"markov": _prepare_markov, "bank": _prepare_bank, "kv": _prepare_kv,
     "classify": _prepare_buffers, "mismatch": _prepare_buffers, "prune": _prepare_prune,
     "global": _prepare_prune, "reads": _prepare_reads}[case["kind"]](s, case, g)
    if case.get("planned"):
        if case["kind"] == "bank":  # the planned checkpoint runs once here: its lists first
            s.ctx.prune(s.banks, s.n, s.params, s.kept)
        _plan(s)
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def run(s):
    c, ctx = s.case, s.ctx
    kind = c["kind"]
    if kind == "classify":
        return ctx.classify(s.after, s.fp_before, s.fp_after, s.must)
    if kind == "mismatch":
        return ctx.mismatch(s.before, s.after, s.counts)
    if kind == "prune":
        ctx.prune(s.banks, s.n, s.params, s.kept, s.kept_off, s.scores)
        return {"scores": s.scores, "kept": s.kept, "offsets": s.kept_off}
    if kind == "global":
        ctx.prune_global(s.banks, s.n, s.budget, s.kept, s.kept_off, s.scores)
        return {"scores": s.scores, "kept": s.kept, "offsets": s.kept_off}
    if kind == "reads":
        return ctx.classify_reads(s.bufs, s.addr, s.nbytes, s.flags)
    if kind == "bank":
        ctx.prune(s.banks, s.n, s.params, s.kept)
    if s.plans:
        for p in s.plans:
            ctx.plan_run(p)
        return s.out
    hs = ctx.checkpoint_raw(s.source, s.n, _placement(c))
    if c.get("fork"):
        child = ctx.fork_raw(hs, s.n)
        ctx.delete_raw(hs, s.n)
        hs = child
    ctx.restore_raw(hs, s.n, s.target, verify=2)
    ctx.delete_raw(hs, s.n)
    return s.out


# ---------------------------------------------------------------------------
# What a pass cannot do without, and what it may be off by
# ---------------------------------------------------------------------------

def work(case):
    """Bytes read once and written once per pass (checkpoint, restore and fork
    each read and write the payload), and the multiply-adds of the scores."""
    kind = case["kind"]
    if kind == "markov":
        return {"bytes": 4 * case["sessions"] * (3 * case["height"] * case["width"] + 16)}
    if kind == "kv":
        payload = case["sessions"] * (32 + 4 * case["layers"] * case["window"] * case["heads"]
                                      * case["head_dim"])
        return {"bytes": (6 if case["fork"] else 4) * payload}
    if kind == "classify":
        return {"bytes": _total(case) + 17 * case["buffers"]}
    if kind == "mismatch":
        return {"bytes": 2 * _total(case) + 8 * case["buffers"]}
    if kind == "reads":
        return {"bytes": 16 * case["reads"] + 17 * case["buffers"]}
    entries = sum(_entries(case))
    score = 2 * case["key_dim"] * entries
    flops = 4 * case["key_dim"] * entries  # q.k and k.k
    if kind == "bank":
        k = sum(_kept(case))
        return {"bytes": score + 4 * k * (4 + 2 * case["key_dim"] + case["value_bytes"]),
                "flops": flops}
    kept = sum(_kept(case)) if kind == "prune" else int(case["keep"] * entries)
    return {"bytes": score + 4 * entries + 4 * kept, "flops": flops}


def tolerance(case):
    """Copies, fingerprints and counts are exact; the fp32 score is defined
    with a fixed order of separately rounded operations, which decides the
    kept entries, so it is exact as well."""
    return "exact"


def exact(case, seed):
    """The cosine scores in 64 bits; nothing else here is a computed number."""
    if case["kind"] not in ("prune", "global"):
        return None
    s, g = _State(case), _gen(seed)
    _prepare_banks(s, case, g)
    out = torch.empty(s.off[-1], dtype=torch.float64, device=_DEV)
    for b, keys in enumerate(s.bank_keys):
        k, q = keys.double(), s.queries[b].double()
        out[s.off[b]:s.off[b + 1]] = (k @ q) / (k.norm(dim=1) * q.norm())
    return {"scores": out, "kept": None, "offsets": None}
