"""The calls whose speed counts: what a decoder with visual revisits has the library do.

A decoding multimodal model keeps raw visual K/V per layer, lets attention choose the tokens to revisit, rebinds and
appends them to its cache and takes its next decode step over the grown cache. Each case is one such call (or the
whole chain) through the package's public entry points, on inputs of the shapes of ``workloads/configs.py`` or of
generic odd ones. ``draw`` gives more cases of the same ranges:

  op         what                                                   sizes
  revisit    Revisit.run: plan, rebind, inject (prcr_rebind_inject)  1..16 sequences, 1..4 revisits of 16..1024 tokens
  store      store_raw of every sequence's prefill rows              1..8 sequences, 64..16384 visual tokens
  capture    prefill_capture of every sequence's prefill rows        as store
  select     select_topk from the raw store                          1..32 sequences, 64..16384 visual tokens
  cached     select_topk_cached from the position-bound cache        as select
  decode     decode_attention over the active cache                  1..16 sequences of up to 8192 slots
  pipeline   select_topk, then rebind_inject, then decode_attention  1..4 sequences

with 1..36 layers, 1..8 KV heads, GQA groups of 1..8, head_dim 64, 128 (the usual one) and 256, contiguous caches and
paged ones of several block sizes, and both M-RoPE band layouts. K/V are bf16 N(0, 1), made on the GPU from the seed.
Everything that decides how much work a case is (token counts, lengths) follows from the case alone, not from the seed.
"""
import math

import numpy as np
import torch

import paper_2606_26631_gb300 as prcr

DEV = "cuda"
THETA = 1.0e6
LEFT = 2  # the method's default left extension


# ----------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------
def listed():
    b8 = dict(layers=36, kv_heads=8, group=4, head_dim=128, sec_t=24, layout="sectioned")  # Qwen3-VL-8B geometry
    b7 = dict(layers=28, kv_heads=4, group=7, head_dim=128, sec_t=16, layout="sectioned")  # Qwen2.5-VL-7B geometry
    paged = dict(cache="paged", block=16)
    flat = dict(cache="contiguous", block=1)
    small = dict(images=1, frames=1, rows=24, cols=32)       # a 768-token image
    odd = dict(images=1, frames=1, rows=46, cols=46)         # 2116 tokens
    pair = dict(images=2, frames=1, rows=64, cols=64)        # two 4096-token images
    video = dict(images=1, frames=16, rows=32, cols=32)      # 16,384 tokens
    return [
        # one user's revisit of 32 tokens of one image: the smallest step, latency alone
        dict(name="revisit-8b-k32", op="revisit", seqs=1, revisits=1, k=32, pos_lo=900, pos_hi=900, **b8, **flat, **small),
        # a small serving batch, one revisit of about 512 tokens each, paged cache
        dict(name="revisit-7b-b8", op="revisit", seqs=8, revisits=1, k=512, pos_lo=1000, pos_hi=4000, **b7, **paged, **odd),
        # a large serving batch, four revisits of ragged sizes per sequence: the most data a revisit step moves
        dict(name="revisit-8b-b16", op="revisit", seqs=16, revisits=4, k=640, pos_lo=1000, pos_hi=4000, **b8, **paged, **pair),
        # prefill of eight requests, one image each: raw rows to the store, rotated rows to the cache
        dict(name="capture-7b-b8", op="capture", seqs=8, pos_lo=0, pos_hi=0, **b7, **paged, **odd),
        # the same rows into the raw store only (a program that writes its own cache), one request
        dict(name="store-7b-b1", op="store", seqs=1, **b7, **odd),
        # which tokens of one 768-token image to revisit: the smallest selection
        dict(name="select-8b-b1", op="select", seqs=1, k=32, pos_lo=900, pos_hi=900, **b8, **small),
        # the same over a batch of 16,384-token videos: the largest selection
        dict(name="select-video-b32", op="select", seqs=32, k=4096, pos_lo=8000, pos_hi=30000, **dict(b8, layers=1), **video),
        # selection from the rows that the decoder's paged cache already holds
        dict(name="cached-8b-b16", op="cached", seqs=16, k=640, pos_lo=9000, pos_hi=12000, **dict(b8, layers=2), **paged, **pair),
        # one user's decode step, every layer: a short context, so mostly latency
        dict(name="decode-8b-b1", op="decode", seqs=1, max_len=933, **b8, **flat),
        # a small serving batch with an odd GQA group, ragged lengths
        dict(name="decode-7b-b8", op="decode", seqs=8, max_len=4096, **b7, **paged),
        # a serving batch at head_dim 256 (8 query heads per KV head): the largest decode step
        dict(name="decode-d256-b16", op="decode", seqs=16, max_len=4096, layers=26, kv_heads=4, group=8, head_dim=256, sec_t=48,
             layout="sectioned", **paged),
        # one user's whole revisit: choose 32 tokens, rebind and append them, decode over the grown cache
        dict(name="pipeline-8b-k32", op="pipeline", seqs=1, revisits=1, k=32, pos_lo=900, pos_hi=900, **b8, **flat, **small),
    ]


_MOST = 10.0e9  # bytes of a drawn case's pass: below the largest listed one's


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    op = rng.choice(["revisit", "revisit", "store", "capture", "select", "select", "cached", "cached", "decode", "decode", "decode",
                     "pipeline"])
    D = rng.choice([64, 128, 128, 128, 128, 256])
    H = rng.choice([1, 2, 3, 4, 4, 5, 8, 8])
    g = rng.choice([1, 2, 3, 4, 4, 6, 7, 8])
    while H * g * D > 8192 or H * g > 64:
        g = max(1, g // 2)
    c = dict(op=op, kv_heads=H, group=g, head_dim=D, layers=_log_int(rng, 2, 36), sec_t=rng.randint(D // 16, D // 4),
             layout=rng.choice(["sectioned", "sectioned", "interleaved"]))
    if op != "decode":
        frames = rng.choice([1, 1, 1, 2, 5, 16])
        c.update(images=rng.choice([1, 1, 2]), frames=frames, rows=_log_int(rng, 8, 64 if frames == 1 else 32),
                 cols=_log_int(rng, 8, 64 if frames == 1 else 32))
    if op in ("revisit", "capture", "cached", "decode", "pipeline"):
        c.update(rng.choice([dict(cache="contiguous", block=1), dict(cache="paged", block=16),
                             dict(cache="paged", block=rng.choice([8, 16, 32, 64, 7]))]))
    if op == "decode":
        c.update(seqs=_log_int(rng, 1, 16), max_len=_log_int(rng, 64, 8192))
    elif op in ("store", "capture"):
        c.update(seqs=_log_int(rng, 1, 8), pos_lo=0, pos_hi=0)
    else:
        lo = _log_int(rng, 200, 12000)
        top = max(2, n_tokens(c) // 2)
        c.update(seqs=_log_int(rng, 1, {"revisit": 16, "pipeline": 4}.get(op, 32)), pos_lo=lo, pos_hi=lo + rng.randint(0, 3000),
                 k=_log_int(rng, min(16, top), min(1024, top)))
        if op in ("revisit", "pipeline"):
            c.update(revisits=rng.choice([1, 1, 2, 4]) if op == "revisit" else 1)
    if op in ("select", "cached"):
        c["layers"] = rng.choice([1, 2])
    if op == "store":
        del c["pos_lo"], c["pos_hi"]
    while work(c)["bytes"] > _MOST or _state_bytes(c) > 3 * _MOST:
        if c["seqs"] > 1:
            c["seqs"] = (c["seqs"] + 1) // 2
        else:
            c["layers"] = (c["layers"] + 1) // 2
    return c


# ----------------------------------------------------------------------------
# what follows from the case alone
# ----------------------------------------------------------------------------
def n_tokens(c):
    return c["images"] * c["frames"] * c["rows"] * c["cols"]


def _sections(c):
    P = c["head_dim"] // 2
    h = (P - c["sec_t"]) // 2
    return (c["sec_t"], h, P - c["sec_t"] - h)


def _fixed(c, what):
    """Random numbers that belong to the case and not to the seed."""
    return np.random.default_rng([sum(map(ord, what)), c["seqs"], c.get("k", 0), c.get("max_len", 0), c["layers"]])


def _rects(c):
    """(rows, columns) of the rectangle of each revisit: [sequence][revisit]; areas from 2/5 to 8/5 of k."""
    rng, R, C = _fixed(c, "rects"), c["rows"], c["cols"]
    out = []
    for _ in range(c["seqs"]):
        out.append([])
        for _ in range(c["revisits"]):
            area = c["k"] if c["seqs"] * c["revisits"] == 1 else int(c["k"] * rng.uniform(0.4, 1.6))
            area = max(1, min(area, R * C))
            nr = int(rng.integers(-(-area // C), min(R, area) + 1))
            if c["k"] == 32 and area == 32:
                nr = 4
            out[-1].append((nr, max(1, min(C, area // nr))))
    return out


def _appended(c):
    if c["op"] == "pipeline":
        return [c["k"]] * c["seqs"]
    return [sum(r * w for r, w in revs) for revs in _rects(c)]


def _contexts(c):
    """Slots each sequence's cache holds before the call."""
    return [int(x) for x in _fixed(c, "contexts").integers(c["pos_lo"], c["pos_hi"] + 1, size=c["seqs"])]


def _lengths(c):
    n = _fixed(c, "lengths").integers(max(1, c["max_len"] // 4), c["max_len"] + 1, size=c["seqs"])
    n[-1] = c["max_len"]
    return [int(x) for x in n]


def _row_bytes(c):
    return 2 * c["kv_heads"] * c["head_dim"]


def work(c):
    row, H, D = _row_bytes(c), c["kv_heads"], c["head_dim"]
    Hq, B, L = H * c["group"], c["seqs"], c["layers"]

    def revisit(tokens):  # K and V rows read and written; index, position, slot of each token
        return tokens * (L * 4 * row + 4 + 24 + 4 + 12), tokens * L * H * D * 3

    def select(layer_tokens, coords):  # keys and queries read, relevances and indices written
        return layer_tokens * (row + (12 if coords else 0) + 4) + B * (Hq * D * 2 + 4 * c["k"]), layer_tokens * Hq * (2 * D + 8)

    def decode(slots):
        return slots * L * 2 * row + B * L * Hq * D * 6, slots * L * Hq * (4 * D + 8)

    if c["op"] == "revisit":
        b, f = revisit(sum(_appended(c)))
    elif c["op"] == "store":
        b, f = B * n_tokens(c) * (L * 4 * row + 24), 0
    elif c["op"] == "capture":
        b, f = B * n_tokens(c) * (L * 6 * row + 24), B * n_tokens(c) * L * H * D * 3
    elif c["op"] in ("select", "cached"):
        b, f = select(B * n_tokens(c), c["op"] == "select")
    elif c["op"] == "decode":
        b, f = decode(sum(_lengths(c)))
    else:
        parts = [select(B * n_tokens(c), True), revisit(B * c["k"]), decode(sum(_contexts(c)) + B + B * c["k"])]
        b, f = (sum(p[i] for p in parts) for i in (0, 1))
    return {"bytes": float(b), "flops": float(f)}


def _state_bytes(c):
    row, B, L = _row_bytes(c), c["seqs"], c["layers"]
    if c["op"] == "decode":
        return B * c["max_len"] * L * 2 * row
    M = n_tokens(c)
    n = B * M * L * 2 * row
    if c["op"] == "capture":
        return 3 * n
    if c["op"] in ("store", "cached"):
        return 2 * n
    if c["op"] in ("revisit", "pipeline"):
        n += B * (max(_contexts(c)) + max(_appended(c)) + 64) * L * 2 * row
    return n


def tolerance(c):
    """Measured on the GPU against the 64-bit result (rounded to bf16 where the output is), times about four."""
    if c["op"] == "store":
        return "exact"  # copies
    if c["op"] in ("revisit", "capture"):
        # bf16 keys: an element near a rounding boundary may fall to its neighbour (2^-7 of the value at most)
        return {"rel": 6e-5, "max": 8e-3}
    if c["op"] in ("select", "cached"):
        return {"rel": 4e-6, "max": 1e-4}  # the relevances; the indices have no near tie at the cut (see _no_near_tie)
    if c["op"] == "decode":
        return {"rel": 2e-5, "max": 2e-4}
    return {"rel": 6e-5, "max": 8e-3}  # the chain: the cache's keys are the widest


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _gen(seed, which):
    return torch.Generator(device=DEV).manual_seed(1000003 * (int(seed) % (1 << 40)) + which)


def _normal(shape, gen):
    return torch.randn(shape, generator=gen, device=DEV, dtype=torch.bfloat16)


def _coords(c):
    """[B, M, 3] int32: token (f, r, w) of an image with base s at (s + f, s + r, s + w), images apart by some text."""
    out, s = [], 16
    for _ in range(c["images"]):
        f, r, w = np.meshgrid(np.arange(c["frames"]), np.arange(c["rows"]), np.arange(c["cols"]), indexing="ij")
        out.append(np.stack([s + f.ravel(), s + r.ravel(), s + w.ravel()], 1))
        s += max(c["frames"], c["rows"], c["cols"]) + 24
    one = np.concatenate(out).astype(np.int32)
    return torch.from_numpy(np.broadcast_to(one, (c["seqs"],) + one.shape).copy()).to(DEV)


def _to(a, dtype):
    return torch.as_tensor(np.asarray(a), dtype=dtype).to(DEV)


def _cfg(c):
    return prcr.rope_cfg(c["layers"], c["kv_heads"], c["head_dim"], _sections(c), THETA,
                         prcr.LAYOUT_INTERLEAVED if c["layout"] == "interleaved" else prcr.LAYOUT_SECTIONED)


def _cache(c, first, last, rng, gen):
    """A cache whose slots first[b] .. last[b] - 1 are backed: (k, v, block table or None). Rows are N(0, 1) as a model's
    context is, or zero (gen None) where the call fills them."""
    B, L, H, D, bs = c["seqs"], c["layers"], c["kv_heads"], c["head_dim"], c["block"]
    if c["cache"] == "contiguous":
        shape, bt = (B, L, max(last) + 8, H, D), None
    else:
        lo, hi = [f // bs for f in first], [-(-e // bs) for e in last]
        total = sum(h - l for l, h in zip(lo, hi))
        perm = rng.permutation(total + 3)[:total]  # a few blocks of the pool stay unused
        table = np.full((B, max(hi) + 1), -1, dtype=np.int32)
        n = 0
        for b in range(B):
            table[b, lo[b]:hi[b]] = perm[n:n + hi[b] - lo[b]]
            n += hi[b] - lo[b]
        shape, bt = (L, total + 3, bs, H, D), _to(table, torch.int32)
    make = (lambda: _normal(shape, gen)) if gen is not None else (lambda: torch.zeros(shape, dtype=torch.bfloat16, device=DEV))
    return make(), make(), bt


def _cache_desc(k, v, bt):
    return prcr.cache_contiguous(k, v) if bt is None else prcr.cache_paged(k, v, bt)


def _store(c, seed):
    shape = (c["seqs"], c["layers"], n_tokens(c), c["kv_heads"], c["head_dim"])
    return _normal(shape, _gen(seed, 1)), _normal(shape, _gen(seed, 2)), _coords(c)


def _positions(c, rng):
    """The latest text positions: behind the context's slot count, as M-RoPE compresses images."""
    return np.asarray([int(n * f) + 40 for n, f in zip(_contexts(c), rng.uniform(0.5, 1.0, c["seqs"]))])


def _selection(c, rng):
    """Revisit offsets and indices: every revisit a rectangle at a random place of one frame of one image."""
    sro, rto, idx = [0], [0], []
    R, C = c["rows"], c["cols"]
    for revs in _rects(c):
        for nr, nc in revs:
            frame = int(rng.integers(0, c["images"] * c["frames"]))
            r0, c0 = int(rng.integers(0, R - nr + 1)), int(rng.integers(0, C - nc + 1))
            r, w = np.meshgrid(np.arange(r0, r0 + nr), np.arange(c0, c0 + nc), indexing="ij")
            idx.append((frame * R * C + r * C + w).ravel())
            rto.append(rto[-1] + nr * nc)
        sro.append(len(rto) - 1)
    return sro, rto, np.concatenate(idx)


def _no_near_tie(rows_of, c, q, q_pos, relevance):
    """Keeps the k-th and the (k+1)-th relevance of every sequence apart by 5e-5 of their value, far more than sums in
    float32 differ by: one flipped near tie would shift the sorted indices behind it. Tokens too close to the cut lose
    their key (rows_of(b): that sequence's [M, H, D] keys, changed in place)."""
    k, M = c["k"], n_tokens(c)
    if k >= M:
        return
    for b in range(c["seqs"]):
        keys = rows_of(b)
        for _ in range(12):
            rel = relevance(b, keys.double())
            top, order = rel.topk(k + 1)
            cut, below = float(top[k - 1]), float(top[k])
            if cut - below > 5e-5 * cut:
                break
            near = ((rel - cut).abs() < 1e-4 * cut).nonzero().flatten()
            keys[near[near != order[0]]] = 0


def _select_state(c, seed, keys_are_rotated):
    """Queries, positions and outputs of a selection."""
    B, Hq, M = c["seqs"], c["kv_heads"] * c["group"], n_tokens(c)
    rng = np.random.default_rng([int(seed) % (1 << 40), 5])
    s = dict(q=_normal((B, Hq, c["head_dim"]), _gen(seed, 5)), q_pos=_to(_positions(c, rng), torch.int64),
             idx=torch.zeros(B * c["k"], dtype=torch.int32, device=DEV), sro=torch.zeros(B + 1, dtype=torch.int32, device=DEV),
             rto=torch.zeros(B + 1, dtype=torch.int32, device=DEV), score=torch.zeros((B, M), dtype=torch.float32, device=DEV),
             ws=torch.empty(prcr.select_workspace_size(B, Hq, M), dtype=torch.uint8, device=DEV))
    return s


def _prepare_select(c, seed):
    s = dict(_select_state(c, seed, False), c=c, cfg=_cfg(c), layer=c["layers"] - 1)
    s["store_k"], s["store_v"], s["coords"] = _store(c, seed)
    _no_near_tie(lambda b: s["store_k"][b, s["layer"]], c, s["q"], s["q_pos"],
                 lambda b, k: _relevance(c, s["q"][b], int(s["q_pos"][b]), k, s["coords"][b]))
    s["store"] = prcr.store_desc(s["store_k"], s["store_v"], s["coords"])
    return s


def _prepare_cached(c, seed):
    s = dict(_select_state(c, seed, True), c=c, cfg=_cfg(c), layer=c["layers"] - 1)
    rng = np.random.default_rng([int(seed) % (1 << 40), 6])
    M, B = n_tokens(c), c["seqs"]
    first = [int(x) for x in _fixed(c, "prefix").integers(3, 60, size=B)]  # a text prefix before the image
    k, v, bt = _cache(c, [0] * B, [f + M + 5 for f in first], rng, _gen(seed, 3))
    s.update(cache_k=k, cache_v=v, bt=bt, cache=_cache_desc(k, v, bt), slot0=_to(first, torch.int32), first=first,
             status=torch.zeros(1, dtype=torch.int32, device=DEV))
    for b in range(B):  # a row view cannot be taken of a paged cache: change a copy and write it back
        rows = _rows(c, k, bt, b, s["layer"], first[b], M)
        before = rows.clone()
        one = dict(c, seqs=1)
        _no_near_tie(lambda _: rows, one, s["q"], s["q_pos"], lambda _, x: _relevance(c, s["q"][b], int(s["q_pos"][b]), x, None))
        for m in (rows != before).any(-1).any(-1).nonzero().flatten().tolist():
            if bt is None:
                k[b, s["layer"], first[b] + m] = 0
            else:
                k[s["layer"], int(bt[b, (first[b] + m) // c["block"]]), (first[b] + m) % c["block"]] = 0
    return s


def _rows(c, cache, bt, b, layer, first, n):
    """Slots first .. first + n - 1 of sequence b at a layer: [n, H, D]."""
    if bt is None:
        return cache[b, layer, first:first + n].clone()
    s = torch.arange(first, first + n, device=DEV)
    return cache[layer][bt[b].long()[s // c["block"]], s % c["block"]]


def _prepare_revisit(c, seed):
    rng = np.random.default_rng([int(seed) % (1 << 40), 7])
    s = dict(c=c)
    s["store_k"], s["store_v"], s["coords"] = _store(c, seed)
    s["p"], s["len"] = _positions(c, rng), _contexts(c)
    sro, rto, idx = _selection(c, rng)
    s["sro"], s["rto"], s["idx"] = sro, rto, idx
    # paged: the blocks that the appended rows fall into; the context's own are not touched by this call
    k, v, bt = _cache(c, s["len"], [n + a for n, a in zip(s["len"], _appended(c))], rng, None)
    s.update(cache_k=k, cache_v=v, bt=bt)
    s["rv"] = prcr.Revisit(_cfg(c), s["store_k"], s["store_v"], s["coords"], k, v, bt, _to(sro, torch.int32), _to(rto, torch.int32),
                           _to(idx, torch.int32), _to(s["p"], torch.int64), _to(s["len"], torch.int32), L=LEFT)
    return s


def _prepare_fill(c, seed):
    """Prefill rows [B, n_L, M, H, D] and their coordinates, and the store (and cache) that they go to."""
    s = dict(c=c, cfg=_cfg(c))
    s["src_k"], s["src_v"], s["src_coords"] = _store(c, seed)
    s["store_k"], s["store_v"] = torch.zeros_like(s["src_k"]), torch.zeros_like(s["src_v"])
    s["coords"] = torch.zeros_like(s["src_coords"])
    s["store"] = prcr.store_desc(s["store_k"], s["store_v"], s["coords"])
    if c["op"] == "capture":
        rng = np.random.default_rng([int(seed) % (1 << 40), 8])
        M, B = n_tokens(c), c["seqs"]
        s["first"] = [int(x) for x in _fixed(c, "prefix").integers(3, 60, size=B)]
        k, v, bt = _cache(c, [0] * B, [f + M for f in s["first"]], rng, None)
        s.update(cache_k=k, cache_v=v, bt=bt, cache=_cache_desc(k, v, bt), status=torch.zeros(1, dtype=torch.int32, device=DEV))
    return s


def _decode_state(c, seed, cfg, max_len):
    B, L, Hq, D = c["seqs"], c["layers"], c["kv_heads"] * c["group"], c["head_dim"]
    n = prcr.decode_workspace_size(cfg, B, Hq, max_len)
    return dict(dq=_normal((B, L, Hq, D), _gen(seed, 9)), out=torch.zeros((B, L, Hq, D), dtype=torch.float32, device=DEV),
                dstatus=torch.zeros(1, dtype=torch.int32, device=DEV), max_len=max_len,
                dws=torch.empty(n, dtype=torch.uint8, device=DEV) if n else None)


def _prepare_decode(c, seed):
    rng = np.random.default_rng([int(seed) % (1 << 40), 10])
    lens, cfg = _lengths(c), _cfg(c)
    k, v, bt = _cache(c, [0] * c["seqs"], lens, rng, _gen(seed, 4))
    s = dict(_decode_state(c, seed, cfg, max(lens)), c=c, cfg=cfg, cache_k=k, cache_v=v, bt=bt, cache=_cache_desc(k, v, bt), lens=lens)
    s["q_pos"] = _to([int(n * f) + 40 for n, f in zip(lens, rng.uniform(0.5, 1.0, c["seqs"]))], torch.int64)
    s["seq_len"] = _to(lens, torch.int32)
    return s


def _prepare_pipeline(c, seed):
    s = _prepare_select(c, seed)
    rng = np.random.default_rng([int(seed) % (1 << 40), 11])
    s["len"] = [n + 1 for n in _contexts(c)]
    last = [n + c["k"] for n in s["len"]]
    k, v, bt = _cache(c, [0] * c["seqs"], last, rng, _gen(seed, 4))
    s.update(cache_k=k, cache_v=v, bt=bt)
    s["rv"] = prcr.Revisit(s["cfg"], s["store_k"], s["store_v"], s["coords"], k, v, bt, s["sro"], s["rto"], s["idx"], s["q_pos"],
                           _to(s["len"], torch.int32), L=LEFT)
    s.update(_decode_state(c, seed, s["cfg"], max(last)))
    return s


def prepare(case, seed):
    return {"revisit": _prepare_revisit, "store": _prepare_fill, "capture": _prepare_fill, "select": _prepare_select,
            "cached": _prepare_cached, "decode": _prepare_decode, "pipeline": _prepare_pipeline}[case["op"]](case, seed)


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------
def _run_select(s):
    prcr.select_topk(s["cfg"], s["store"], s["layer"], s["q"], s["q_pos"], s["c"]["k"], s["idx"], s["sro"], s["rto"], s["ws"], s["score"])


def _run_decode(s, cache, q_pos, seq_len):
    prcr.decode_attention(s["cfg"], cache, s["dq"], q_pos, seq_len, s["max_len"], s["out"], s["dstatus"], s["dws"])


def run(s):
    op = s["c"]["op"]
    if op == "revisit":
        rv = s["rv"]
        rv.run()
        return dict(cache_k=s["cache_k"], cache_v=s["cache_v"], pos=rv.pos, slot=rv.slot, cache_len=rv.cache_len_out,
                    next_pos=rv.next_pos, status=rv.status)
    if op == "store":
        for b in range(s["c"]["seqs"]):
            prcr.store_raw(s["cfg"], s["store"], b, 0, 0, s["src_k"][b], s["src_v"][b], s["src_coords"][b])
        return dict(store_k=s["store_k"], store_v=s["store_v"], coords=s["coords"])
    if op == "capture":
        for b in range(s["c"]["seqs"]):
            prcr.prefill_capture(s["cfg"], s["store"], s["cache"], b, 0, 0, s["first"][b], s["src_k"][b], s["src_v"][b],
                                 s["src_coords"][b], s["status"])
        return dict(store_k=s["store_k"], store_v=s["store_v"], coords=s["coords"], cache_k=s["cache_k"], cache_v=s["cache_v"],
                    status=s["status"])
    if op == "select":
        _run_select(s)
        return dict(idx=s["idx"], seq_rev_off=s["sro"], rev_tok_off=s["rto"], score=s["score"])
    if op == "cached":
        prcr.select_topk_cached(s["cfg"], s["cache"], s["layer"], s["q"], s["q_pos"], s["slot0"], n_tokens(s["c"]), s["c"]["k"],
                                s["idx"], s["sro"], s["rto"], s["status"], s["ws"], s["score"])
        return dict(idx=s["idx"], seq_rev_off=s["sro"], rev_tok_off=s["rto"], score=s["score"], status=s["status"])
    if op == "decode":
        _run_decode(s, s["cache"], s["q_pos"], s["seq_len"])
        return dict(out=s["out"], status=s["dstatus"])
    rv = s["rv"]
    _run_select(s)
    rv.run()
    _run_decode(s, rv.cache, rv.next_pos, rv.cache_len_out)
    return dict(idx=s["idx"], score=s["score"], cache_k=s["cache_k"], cache_v=s["cache_v"], pos=rv.pos, slot=rv.slot,
                cache_len=rv.cache_len_out, next_pos=rv.next_pos, out=s["out"], status=rv.status)


# ----------------------------------------------------------------------------
# the same in 64 bits, in plain torch
# ----------------------------------------------------------------------------
def _axis_of_pair(c):
    P = c["head_dim"] // 2
    t, h, w = _sections(c)
    if c["layout"] == "interleaved":
        return torch.tensor([1 if i % 3 == 1 and i < 3 * h else 2 if i % 3 == 2 and i < 3 * w else 0 for i in range(P)], device=DEV)
    return torch.tensor([0] * t + [1] * h + [2] * w, device=DEV)


def _turn(c, x, pos):
    """M-RoPE of x [..., n, H, D] (float64) at pos [n, 3] (float64)."""
    D = c["head_dim"]
    rate = THETA ** (-2.0 * torch.arange(D // 2, device=DEV, dtype=torch.float64) / D)
    ang = pos[:, _axis_of_pair(c)] * rate
    cos, sin = ang.cos()[:, None], ang.sin()[:, None]
    a, b = x[..., :D // 2], x[..., D // 2:]
    return torch.cat([a * cos - b * sin, b * cos + a * sin], -1)


def _turn_query(c, q, p):
    return _turn(c, q.double()[None], torch.full((1, 3), float(p), dtype=torch.float64, device=DEV))[0]


def _relevance(c, q, p, keys, coords):
    """[M] relevances of one sequence: q [Hq, D] raw, keys [M, H, D] float64 (raw with coords, else already turned)."""
    if coords is not None:
        keys = _turn(c, keys, coords.double())
    M, H, D = keys.shape
    qr = _turn_query(c, q, p).view(H, c["group"], D)
    logits = torch.einsum("mhd,hgd->hgm", keys, qr) / math.sqrt(D)
    return logits.softmax(-1).mean((0, 1))


def _rebound(c, s, sro, rto, idx, p, lens, cache_k, cache_v):
    """(positions, slots) of a revisit, and its rows written into the float64 caches."""
    pos_all, slot_all = [], []
    for b in range(c["seqs"]):
        t0 = rto[sro[b]]
        for r in range(sro[b], sro[b + 1]):
            m = torch.as_tensor(idx[rto[r]:rto[r + 1]], device=DEV).long()
            K = m.numel()
            x = s["coords"][b].long()[m]
            lo, span = x.amin(0), x.amax(0) - x.amin(0)
            den = torch.where(span > 0, (K + 1) * span, torch.full_like(span, K + 1))
            tail = torch.where(span > 0, (LEFT + 1) * (span + (K - 1) * (x - lo)), torch.full_like(x, LEFT + 1))
            pos = ((int(p[b]) - LEFT) * den + tail).double() / den.double()
            slot = torch.arange(K, device=DEV) + (int(lens[b]) + rto[r] - t0)
            k = _turn(c, s["store_k"][b][:, m].double(), pos)
            v = s["store_v"][b][:, m].double()
            if s["bt"] is None:
                cache_k[b][:, slot], cache_v[b][:, slot] = k.to(cache_k.dtype), v.to(cache_v.dtype)
            else:
                blk, off = s["bt"][b].long()[slot // c["block"]], slot % c["block"]
                cache_k[:, blk, off], cache_v[:, blk, off] = k.to(cache_k.dtype), v.to(cache_v.dtype)
            pos_all.append(pos)
            slot_all.append(slot)
    return torch.cat(pos_all), torch.cat(slot_all)


def _attention(c, cache_k, cache_v, bt, q, p, lens):
    """[B, n_L, Hq, D]: the decode step, a layer of a sequence at a time."""
    H, g, D = c["kv_heads"], c["group"], c["head_dim"]
    out = torch.zeros(q.shape, dtype=torch.float64, device=DEV)
    for b in range(c["seqs"]):
        for l in range(c["layers"]):
            k = _rows(c, cache_k, bt, b, l, 0, lens[b]).double()
            v = _rows(c, cache_v, bt, b, l, 0, lens[b]).double()
            qr = _turn_query(c, q[b, l], int(p[b])).view(H, g, D)
            w = (torch.einsum("nhd,hgd->hgn", k, qr) / math.sqrt(D)).softmax(-1)
            out[b, l] = torch.einsum("hgn,nhd->hgd", w, v).reshape(H * g, D)
    return out


def exact(case, seed):
    c, op = case, case["op"]
    s = prepare(case, seed)
    if op == "store":
        return dict(store_k=s["src_k"].double(), store_v=s["src_v"].double(), coords=None)
    if op == "capture":
        k, v = torch.zeros_like(s["cache_k"], dtype=torch.float64), torch.zeros_like(s["cache_v"], dtype=torch.float64)
        for b in range(c["seqs"]):
            slot = torch.arange(n_tokens(c), device=DEV) + s["first"][b]
            kr, vr = _turn(c, s["src_k"][b].double(), s["src_coords"][b].double()), s["src_v"][b].double()
            if s["bt"] is None:
                k[b][:, slot], v[b][:, slot] = kr, vr
            else:
                blk, off = s["bt"][b].long()[slot // c["block"]], slot % c["block"]
                k[:, blk, off], v[:, blk, off] = kr, vr
        return dict(store_k=s["src_k"].double(), store_v=s["src_v"].double(), coords=None, cache_k=k, cache_v=v, status=None)
    if op == "revisit":
        k, v = torch.zeros_like(s["cache_k"], dtype=torch.float64), torch.zeros_like(s["cache_v"], dtype=torch.float64)
        pos, _ = _rebound(c, s, s["sro"], s["rto"], s["idx"], s["p"], s["len"], k, v)
        return dict(cache_k=k, cache_v=v, pos=pos, slot=None, cache_len=None, next_pos=None, status=None)
    if op == "decode":
        return dict(out=_attention(c, s["cache_k"], s["cache_v"], s["bt"], s["dq"], s["q_pos"], s["lens"]), status=None)
    M, lay = n_tokens(c), s["layer"]
    if op == "cached":
        score = torch.stack([_relevance(c, s["q"][b], int(s["q_pos"][b]), _rows(c, s["cache_k"], s["bt"], b, lay, s["first"][b], M).double(),
                                        None) for b in range(c["seqs"])])
        return dict(idx=None, seq_rev_off=None, rev_tok_off=None, score=score, status=None)
    score = torch.stack([_relevance(c, s["q"][b], int(s["q_pos"][b]), s["store_k"][b, lay].double(), s["coords"][b])
                         for b in range(c["seqs"])])
    if op == "select":
        return dict(idx=None, seq_rev_off=None, rev_tok_off=None, score=score)
    idx = torch.cat([row.topk(c["k"]).indices.sort().values for row in score]).tolist()
    off = list(range(c["seqs"] + 1))
    k, v = s["cache_k"].double(), s["cache_v"].double()
    pos, _ = _rebound(c, s, off, [c["k"] * b for b in off], idx, s["q_pos"], s["len"], k, v)
    # the decode step reads the cache's bf16 keys
    out = _attention(c, k.to(torch.bfloat16), v.to(torch.bfloat16), s["bt"], s["dq"], s["q_pos"] + 1, [n + c["k"] for n in s["len"]])
    return dict(idx=None, score=score, cache_k=k, cache_v=v, pos=pos, slot=None, cache_len=None, next_pos=None, out=out, status=None)
