"""The transfers that this library's users make, as measurable cases.

A case is one call, or one short run of calls, that a serving replica makes
between two scheduler steps: it stores the new tokens of a context into pinned
host chunks, restores a prefix into fresh pages, packs or unpacks pages on the
device, moves a hybrid model's KV together with its state snapshot, restores
through the shared tier, or stores without allocating.  Every case has its
shape spelled out, so that a drawn case is the same code at other sizes.

Payloads are bytes, moved unchanged: every output is compared exactly (as
64-bit words, which any byte that differs changes).
"""
import ctypes
import math

import torch

from paper_2609_15021_gb300 import hybrid
from paper_2609_15021_gb300 import kvxfer as k

_POISON = 0xA5
_ctx = None


def _context():
    """The one transfer context that a program makes at start-up and keeps."""
    global _ctx
    if _ctx is None:
        _ctx = k.KvTransfer(0)
    return _ctx.ctx


def _kv(name, op, layers, heads, head_dim, elem, block, layout, chunk, tokens, begin=0, per_block=1, stacked=False):
    """tokens: how many are moved, from token `begin`; per_block: pages per logical block; stacked: all layers
    in one allocation, as some engines keep them, rather than one allocation for each layer."""
    return {"name": name, "op": op, "layers": layers, "heads": heads, "head_dim": head_dim, "elem": elem,
            "block": block, "layout": layout, "chunk": chunk, "tokens": tokens, "begin": begin,
            "per_block": per_block, "stacked": stacked}


def listed():
    return [
        # The smallest context that the tests and the smoke run use: two layers, 512 tokens.  A short prompt of a
        # draft model: latency, launches and host work are all there is.
        _kv("store_tiny", "store", 2, 2, 64, 2, 16, "hnd", 256, 512),
        _kv("load_tiny", "load", 2, 2, 64, 2, 16, "hnd", 256, 512),
        # The 27B-class shape (62 x 8 x 128 bf16, 16-token pages): the one chunk that 256 decoded tokens fill,
        # stored when it is full, behind a context of eight chunks.
        _kv("store_27b_chunk", "store", 62, 8, 128, 2, 16, "hnd", 256, 256, begin=2048),
        # The same shape, a whole 32k-token prefix restored into another replica's pages: the largest.
        _kv("load_27b_32k", "load", 62, 8, 128, 2, 16, "hnd", 256, 32768, stacked=True),
        # The paper's FP8 attention KV: 1,568-token logical blocks of 49 pages of 32 tokens, and a prompt
        # whose end fills neither a chunk nor a page.
        _kv("store_fp8_ragged", "store", 16, 4, 256, 1, 32, "hnd", 1568, 12345, per_block=49),
        # Rows that are no power of two (head_dim 96), a ragged 1,237-token prompt: restore.
        _kv("load_dim96_ragged", "load", 32, 8, 96, 2, 16, "hnd", 256, 1237),
        # Device-side moves (a prefill replica's export buffer and the import on the decode side): the 27B
        # shape, and one KV head of it, as each GPU of an eight-way tensor-parallel replica holds.
        _kv("pack_27b_4k", "pack", 62, 8, 128, 2, 16, "hnd", 256, 4096, stacked=True),
        _kv("unpack_1head_ragged", "unpack", 62, 1, 128, 2, 16, "hnd", 256, 4093),
        # A turn of the six-turn hybrid session: 2,048 tokens of 16 attention layers and the 48-layer state
        # snapshot, stored at the end of the turn and restored on the other replica at the start of the next.
        {"name": "session_store", "op": "session_store", "attn_layers": 16, "state_layers": 48, "begin": 2048,
         "tokens": 2048},
        {"name": "session_load", "op": "session_load", "attn_layers": 16, "state_layers": 48, "begin": 2048,
         "tokens": 2048},
        # A prefix found in the shared tier and restored into an NHD pool: lookup, acquire, load, release.
        _kv("tier_load_nhd", "tier_load", 32, 4, 128, 2, 32, "nhd", 512, 3001),
        # The store for callers that cannot allocate: 2,048 tokens of the 27B shape.
        _kv("store_noalloc_2k", "store_noalloc", 62, 8, 128, 2, 16, "hnd", 256, 2048),
    ]


def _log_uniform(rng, low, high):
    return max(low, min(high, int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))))


def draw(rng):
    op = rng.choice(["store", "load", "store", "load", "pack", "unpack", "tier_load", "store_noalloc",
                     "session_store", "session_load"])
    if op.startswith("session"):
        return {"op": op, "attn_layers": rng.choice([4, 8, 12, 16]), "state_layers": rng.choice([12, 24, 36, 48]),
                "begin": 256 * rng.randint(0, 16), "tokens": 256 * _log_uniform(rng, 1, 32)}
    layers = _log_uniform(rng, 2, 64)
    heads = rng.choice([1, 2, 4, 8, 8, 12])
    head_dim, elem = rng.choice([(64, 2), (80, 2), (96, 2), (128, 2), (128, 2), (128, 2), (128, 1), (192, 2), (256, 1),
                                 (256, 2)])
    block = rng.choice([16, 16, 16, 32, 64])
    per_block, chunk = 1, rng.choice([128, 256, 256, 512, 1024])
    if block == 32 and rng.random() < 0.5:
        per_block, chunk = 49, 1568
    per_token = layers * 2 * heads * head_dim * elem
    most = max(64, min(32768, (2 << 30) // per_token))  # at most 2 GiB each way
    tokens = _log_uniform(rng, 17, most)
    c = _kv("", op, layers, heads, head_dim, elem, block, rng.choice(["hnd", "hnd", "nhd"]), chunk, tokens,
            begin=chunk * rng.randint(0, 2), per_block=per_block, stacked=rng.random() < 0.5)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs


def _fill(t, g, elem=2):
    """KV values ~ N(0, 1) in bf16 (uniform bytes for 1-byte KV, whose scales are the quantiser's)."""
    if elem == 2:
        t.view(torch.bfloat16).normal_(generator=g)
    else:
        t.view(torch.uint8).random_(0, 256, generator=g)
    return t


def _words(t):
    return t.reshape(-1).view(torch.int64)


def _shape(c, pages):
    mid = (c["heads"], c["block"]) if c["layout"] == "hnd" else (c["block"], c["heads"])
    return (pages, 2, *mid, c["head_dim"])


def _span(c):
    """(tokens of one table entry, table entries, pages of the pool): the context up to its last token, and
    a quarter as many pages again for other requests."""
    span = c["block"] * c["per_block"]
    used = -(-(c["begin"] + c["tokens"]) // span)
    return span, used, (used + used // 4 + 1) * c["per_block"]


def _pool(c, g, poison):
    _, _, pages = _span(c)
    dtype = torch.bfloat16 if c["elem"] == 2 else torch.uint8
    shape = _shape(c, pages)
    if c["stacked"]:
        whole = torch.empty((c["layers"], *shape), dtype=dtype, device="cuda")
        layers = list(whole.unbind(0))
        out = [whole]
    else:
        layers = out = [torch.empty(shape, dtype=dtype, device="cuda") for _ in range(c["layers"])]
    for t in out:
        if poison:
            t.view(torch.uint8).fill_(_POISON)
        else:
            _fill(t, g, c["elem"])
    layout = k.KVX_LAYOUT_HND if c["layout"] == "hnd" else k.KVX_LAYOUT_NHD
    if c["per_block"] > 1:  # the packed view: [logical blocks, pages per block, 2, ...]
        layers = [t.view(-1, c["per_block"], *t.shape[1:]) for t in layers]
    pool = k.KvPool.from_tensors(layers, c["heads"], c["block"], layout, c["per_block"])
    return pool, [_words(t) for t in out]


def _table(c, g):
    _, used, pages = _span(c)
    return torch.randperm(pages // c["per_block"], generator=g, device="cuda")[:used].to(torch.int32)


def _chunk_sizes(c):
    per_token = c["layers"] * 2 * c["heads"] * c["head_dim"] * c["elem"]
    sizes, left = [], c["tokens"]
    while left > 0:
        sizes.append(per_token * min(c["chunk"], left))
        left -= c["chunk"]
    return sizes


def _cut(t, sizes):
    """Views of consecutive chunks of `t`, which holds sum(sizes) bytes."""
    at, views = 0, []
    for n in sizes:
        views.append(t[at:at + n])
        at += n
    return views


def _session(case, seed):
    load = case["op"] == "session_load"
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    shape = hybrid.HybridShape(attn_layers=case["attn_layers"], state_layers=case["state_layers"])
    t0, t1 = case["begin"], case["begin"] + case["tokens"]
    pages = t1 // shape.block_tokens
    blocks = pages + pages // 4 + 1

    def replica():
        order = torch.randperm(blocks, generator=g, device="cuda").tolist()
        return hybrid.Replica(shape, blocks, 4, order)

    tier = hybrid.SharedTier(shape, t1, 2)
    tier.chunks.tensor.fill_(_POISON)
    tier.snaps.tensor.fill_(_POISON)
    a = replica()
    for t in a.attn_layers + a.state:
        _fill(t, g)
    a.grow(t1)
    s = {"op": case["op"], "tier": tier, "rep": a, "t0": t0, "t1": t1}
    if load:
        hybrid.store_prefix(_context(), a, tier, t0, t1, 1)
        torch.cuda.synchronize()
        s["rep"] = b = replica()
        for t in b.attn_layers + b.state:
            t.fill_(_POISON)
        s["out"] = [_words(t) for t in b.attn_layers + b.state]
    else:
        s["out"] = [_words(tier.chunks.tensor), _words(tier.snaps.tensor)]
    return s


def prepare(case, seed):
    _context()
    if case["op"].startswith("session"):
        return _session(case, seed)
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    op = case["op"]
    to_pool = op in ("load", "unpack", "tier_load")
    pool, pool_out = _pool(case, g, poison=to_pool)
    s = {"op": op, "pool": pool, "table": _table(case, g), "t0": case["begin"],
         "t1": case["begin"] + case["tokens"], "chunk": case["chunk"]}
    sizes = _chunk_sizes(case)
    total = sum(sizes)
    data = None
    if to_pool:
        data = torch.empty(total, dtype=torch.uint8, device="cuda")
        _fill(data, g, case["elem"])
    if op in ("pack", "unpack"):
        if data is None:
            data = torch.full((total,), _POISON, dtype=torch.uint8, device="cuda")
        s["chunks"] = k.ChunkList(_cut(data, sizes))
        s["out"] = pool_out if op == "unpack" else [_words(data)]
    elif op == "tier_load":
        # another request's prefill left the prefix in the tier: one slot for each chunk, committed
        n = len(sizes)
        s["tier"] = tier = k.KvTier(sizes[0], n)
        tokens = torch.randint(0, 1 << 17, (case["begin"] + case["tokens"],), generator=g, device="cuda")
        keys = k.kv_chunk_keys(tokens.cpu().numpy(), case["chunk"], salt=seed)
        s["keys"] = keys = keys[case["begin"] // case["chunk"]:]
        for key, part in zip(keys, _cut(data, sizes)):
            tier.reserve(key)[:part.numel()].copy_(part)
            tier.commit(key, k.KVX_NO_STREAM)
        s["out"] = pool_out
    else:
        s["host"] = host = k.HostBuffer(total).tensor
        if to_pool:
            host.copy_(data)
        else:
            ctypes.memset(host.data_ptr(), _POISON, total)
        views = _cut(host, sizes)
        s["chunks"] = views if op == "store_noalloc" else k.ChunkList(views)
        s["out"] = pool_out if to_pool else [_words(host)]
    torch.cuda.synchronize()
    return s


def run(s):
    op = s["op"]
    if op == "session_store":
        hybrid.store_prefix(_context(), s["rep"], s["tier"], s["t0"], s["t1"], 1)
    elif op == "session_load":
        hybrid.load_prefix(_context(), s["rep"], s["tier"], s["t0"], s["t1"], 1)
    elif op == "store":
        k.kv_store(_context(), s["pool"], s["table"], s["t0"], s["t1"], s["chunk"], s["chunks"])
    elif op == "load":
        k.kv_load(_context(), s["pool"], s["table"], s["t0"], s["t1"], s["chunk"], s["chunks"])
    elif op == "pack":
        k.kv_pack(_context(), s["pool"], s["table"], s["t0"], s["t1"], s["chunk"], s["chunks"])
    elif op == "unpack":
        k.kv_unpack(_context(), s["pool"], s["table"], s["t0"], s["t1"], s["chunk"], s["chunks"])
    elif op == "store_noalloc":
        k.kv_store_noalloc(s["pool"], s["table"], s["t0"], s["t1"], s["chunk"], s["chunks"])
    else:
        tier, keys = s["tier"], s["keys"]
        keys = keys[:tier.prefix_hits(keys)]
        chunks = tier.acquire_many(keys, as_chunk_list=True)
        k.kv_load(_context(), s["pool"], s["table"], s["t0"], s["t1"], s["chunk"], chunks)
        tier.release_many(keys)
    return s["out"]


def work(case):
    if case["op"].startswith("session"):
        shape = hybrid.HybridShape(attn_layers=case["attn_layers"], state_layers=case["state_layers"])
        payload = case["tokens"] * shape.chunk_bytes // shape.chunk_tokens + shape.snapshot_bytes
    else:
        payload = sum(_chunk_sizes(case))
    return {"bytes": 2 * payload, "flops": 0}


def tolerance(case):
    return "exact"


def exact(case, seed):
    return None  # nothing is computed: bytes are moved, and compared exactly
