"""GPU parity of prcr_decode_attention (Eq. "decode_with_active_cache")
against the oracle's fp64 decode_attention.

1. Decode over a populated input cache (contiguous and paged, GQA groups
   1 / 4 / 7, head_dim 64 / 128 / 256, sequences long enough to be split).
   Bar: max |o_gpu - o_ref| <= 1e-4 * max |V| (float32 logits, exp and
   accumulation over at most a few thousand slots per chunk stay ~1e-6).
2. End to end: revisit rows appended by prcr_rebind_inject into a cache whose
   context rows are data, then decoded at next_pos over cache_len_out. The
   expected cache is the context plus the oracle's rebound keys rounded to
   bf16 (the value a correct kernel stores); bar 1e-3 * max |V|.
3. Relative positions only (Eq. "direct_reuse_score"): a cache made only of
   revisited rows decoded at p + 1 gives the same output when the text
   position moves by a constant (up to the bf16 rounding of the keys).
"""
import numpy as np
import pytest
import torch

from oracle import prcr_oracle as O
from workloads import Workload, get, make_batch, make_decode_inputs

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _f64(t):
    return O.bf16_bits_to_f64(t.contiguous().view(torch.int16).cpu().numpy())


def _cache_rows(cache_k, cache_v, block_table, b, n, paged):
    """[n, n_L, H, D] value arrays of slots 0..n-1 of sequence b (input data)."""
    s = torch.arange(n, device=cache_k.device)
    if not paged:
        return _f64(cache_k[b, :, :n].transpose(0, 1)), _f64(cache_v[b, :, :n].transpose(0, 1))
    bs = cache_k.shape[2]
    blk = block_table[b][s // bs].long()
    off = s % bs
    return _f64(cache_k[:, blk, off].transpose(0, 1)), _f64(cache_v[:, blk, off].transpose(0, 1))


def _run_decode(cfg, cache_desc, q, q_pos, seq_len, max_len):
    import paper_2606_26631_gb300 as prcr
    out = torch.full(q.shape, float("nan"), dtype=torch.float32, device=DEV)
    status = torch.zeros(1, dtype=torch.int32, device=DEV)
    nbytes = prcr.decode_workspace_size(cfg, q.shape[0], q.shape[2], max_len)
    ws = torch.empty(max(nbytes, 16), dtype=torch.uint8, device=DEV)
    prcr.decode_attention(cfg, cache_desc, q, q_pos, seq_len, max_len, out, status, ws)
    torch.cuda.synchronize()
    return out, int(status.item())


CASES = [  # (B, layers, H, Hq, D, max_len, paged)
    (3, 3, 8, 32, 128, 3000, True),
    (2, 2, 2, 14, 64, 700, False),
    (2, 2, 4, 4, 256, 1200, True),
    (5, 1, 4, 28, 128, 9000, True),
    # one sequence of the Table 3 shape (a team of six warps per KV head, unsplit)
    (1, 36, 8, 32, 128, 933, False),
    (2, 2, 8, 16, 64, 500, True),
    # teams at the ends of the GQA range: 1 and 8 query heads per KV head
    (1, 2, 8, 8, 128, 500, False),
    (1, 2, 8, 64, 128, 300, True),
]


@pytest.mark.parametrize("case", CASES, ids=[f"B{c[0]}L{c[1]}H{c[2]}Hq{c[3]}D{c[4]}S{c[5]}{'p' if c[6] else 'c'}" for c in CASES])
def test_decode_parity(case):
    import paper_2606_26631_gb300 as prcr
    B, nL, H, Hq, D, max_len, paged = case
    sec = (D // 8, D // 8 + (D // 2 - 3 * (D // 8)) // 2, 0)
    sec = (sec[0], sec[1], D // 2 - sec[0] - sec[1])
    inp = make_decode_inputs(B, nL, H, Hq, D, max_len, paged, device=DEV, seed=7)
    cfg = prcr.rope_cfg(nL, H, D, sec, 1e6)
    cd = (prcr.cache_paged(inp["cache_k"], inp["cache_v"], inp["block_table"]) if paged
          else prcr.cache_contiguous(inp["cache_k"], inp["cache_v"]))
    out, st = _run_decode(cfg, cd, inp["q"], inp["q_pos"], inp["seq_len"], max_len)
    assert st == 0
    got = out.cpu().numpy()
    qv = _f64(inp["q"])
    for b in range(B):
        n = int(inp["seq_len"][b])
        K, V = _cache_rows(inp["cache_k"], inp["cache_v"], inp["block_table"], b, n, paged)
        for l in range(nL):
            ref = O.decode_attention(qv[b, l], int(inp["q_pos"][b]), K[:, l], V[:, l], D, sec, 1e6)
            err = np.abs(got[b, l] - ref).max() / np.abs(V[:, l]).max()
            assert err <= 1e-4, (b, l, err)


@pytest.mark.parametrize("H,Hq,D,paged", [(8, 32, 128, False), (4, 16, 128, True), (2, 14, 64, False),
                                         (4, 8, 256, True)])
def test_decode_empty_and_single_slot(H, Hq, D, paged):
    """A sequence with no slots gets zeros; one with a single slot gets that
    slot's V row exactly (its softmax weight is exactly 1); a longer one
    beside them still matches the oracle. Head dims 64, 128 and 256; the kernel
    of one warp per chunk has its own such lengths in test_decode_large."""
    import paper_2606_26631_gb300 as prcr
    B, nL, max_len = 3, 2, 300
    sec = (D // 8, D // 8 + (D // 2 - 3 * (D // 8)) // 2, 0)
    sec = (sec[0], sec[1], D // 2 - sec[0] - sec[1])
    inp = make_decode_inputs(B, nL, H, Hq, D, max_len, paged, device=DEV, seed=19)
    seq_len = torch.tensor([0, 1, max_len], dtype=torch.int32, device=DEV)
    cfg = prcr.rope_cfg(nL, H, D, sec, 1e6)
    cd = (prcr.cache_paged(inp["cache_k"], inp["cache_v"], inp["block_table"]) if paged
          else prcr.cache_contiguous(inp["cache_k"], inp["cache_v"]))
    out, st = _run_decode(cfg, cd, inp["q"], inp["q_pos"], seq_len, max_len)
    assert st == 0
    got = out.cpu().numpy()
    assert np.all(got[0] == 0.0)
    g = Hq // H
    K1, V1 = _cache_rows(inp["cache_k"], inp["cache_v"], inp["block_table"], 1, 1, paged)
    for l in range(nL):
        for h in range(Hq):
            assert np.array_equal(got[1, l, h], V1[0, l, h // g].astype(np.float32)), (l, h)
    K, V = _cache_rows(inp["cache_k"], inp["cache_v"], inp["block_table"], 2, max_len, paged)
    qv = _f64(inp["q"])
    for l in range(nL):
        ref = O.decode_attention(qv[2, l], int(inp["q_pos"][2]), K[:, l], V[:, l], D, sec, 1e6)
        assert np.abs(got[2, l] - ref).max() / np.abs(V[:, l]).max() <= 1e-4


def test_decode_device_errors():
    """Device-detected errors: an unmapped block in a sequence's range sets
    PRCR_ST_NO_BLOCK and its slots are left out of the softmax; a length
    beyond the capacity sets PRCR_ST_CAPACITY and is clamped to it; a length
    above max_len sets PRCR_ST_CAPACITY too. Outputs stay the oracle's
    attention over the slots that remain (where those are defined)."""
    import paper_2606_26631_gb300 as prcr
    nL, H, Hq, D, sec = 2, 2, 8, 64, (8, 12, 12)
    cfg = prcr.rope_cfg(nL, H, D, sec, 1e6)
    # (a) paged: block 3 of sequence 1 (its slots 48..63) unmapped
    inp = make_decode_inputs(2, nL, H, Hq, D, 200, True, device=DEV, seed=23)
    bt = inp["block_table"].clone()
    bt[1, 3] = -1
    cd = prcr.cache_paged(inp["cache_k"], inp["cache_v"], bt)
    out, st = _run_decode(cfg, cd, inp["q"], inp["q_pos"], inp["seq_len"], 200)
    assert st & prcr.ST_NO_BLOCK
    got = out.cpu().numpy()
    qv = _f64(inp["q"])
    n1 = int(inp["seq_len"][1])
    K, V = _cache_rows(inp["cache_k"], inp["cache_v"], inp["block_table"], 1, n1, True)
    keep = np.array([s for s in range(n1) if s // 16 != 3])
    for l in range(nL):
        ref = O.decode_attention(qv[1, l], int(inp["q_pos"][1]), K[keep, l], V[keep, l], D, sec, 1e6)
        assert np.abs(got[1, l] - ref).max() / np.abs(V[:, l]).max() <= 1e-4
    K0, V0 = _cache_rows(inp["cache_k"], inp["cache_v"], inp["block_table"], 0, int(inp["seq_len"][0]),
                         True)
    for l in range(nL):
        ref = O.decode_attention(qv[0, l], int(inp["q_pos"][0]), K0[:, l], V0[:, l], D, sec, 1e6)
        assert np.abs(got[0, l] - ref).max() / np.abs(V0[:, l]).max() <= 1e-4
    # (b) contiguous, capacity 208 slots: a length of 300 is clamped to 208
    inp = make_decode_inputs(1, nL, H, Hq, D, 200, False, device=DEV, seed=24)
    cap = inp["cache_k"].shape[2]
    cd = prcr.cache_contiguous(inp["cache_k"], inp["cache_v"])
    seq_len = torch.tensor([300], dtype=torch.int32, device=DEV)
    out, st = _run_decode(cfg, cd, inp["q"], inp["q_pos"], seq_len, cap)
    assert st & prcr.ST_CAPACITY
    got = out.cpu().numpy()
    qv = _f64(inp["q"])
    K, V = _cache_rows(inp["cache_k"], inp["cache_v"], None, 0, cap, False)
    for l in range(nL):
        ref = O.decode_attention(qv[0, l], int(inp["q_pos"][0]), K[:, l], V[:, l], D, sec, 1e6)
        assert np.abs(got[0, l] - ref).max() / np.abs(V[:, l]).max() <= 1e-4
    # (c) a length above the max_len the call was split for
    seq_len = torch.tensor([150], dtype=torch.int32, device=DEV)
    out, st = _run_decode(cfg, cd, inp["q"], inp["q_pos"], seq_len, 100)
    assert st & prcr.ST_CAPACITY
    assert torch.isfinite(out).all()


def test_decode_query_position_range():
    """A query position of 2^31 or more is beyond the fixed-point angle
    reduction: PRCR_ST_POS_RANGE, and that sequence reads no slot (its output
    is zeros) while the other sequence of the batch matches the oracle. Teams
    of warps, split and unsplit sequences."""
    import paper_2606_26631_gb300 as prcr
    sec = (16, 24, 24)
    for H, Hq, max_len in ((8, 32, 300), (2, 8, 300), (8, 32, 3000)):
        inp = make_decode_inputs(2, 2, H, Hq, 128, max_len, False, device=DEV, seed=5)
        cfg = prcr.rope_cfg(2, H, 128, sec, 1e6)
        cd = prcr.cache_contiguous(inp["cache_k"], inp["cache_v"])
        qp = inp["q_pos"].clone()
        qp[0] = 2 ** 31
        out, st = _run_decode(cfg, cd, inp["q"], qp, inp["seq_len"], max_len)
        assert st == prcr.ST_POS_RANGE
        got = out.cpu().numpy()
        assert np.all(got[0] == 0.0)
        n = int(inp["seq_len"][1])
        K, V = _cache_rows(inp["cache_k"], inp["cache_v"], None, 1, n, False)
        qv = _f64(inp["q"])
        for l in range(2):
            ref = O.decode_attention(qv[1, l], int(qp[1]), K[:, l], V[:, l], 128, sec, 1e6)
            assert np.abs(got[1, l] - ref).max() / np.abs(V[:, l]).max() <= 1e-4
        qp[0] = -(2 ** 31)
        out, st = _run_decode(cfg, cd, inp["q"], qp, inp["seq_len"], max_len)
        assert st == prcr.ST_POS_RANGE and bool((out[0] == 0).all().item())
        qp[0] = 2 ** 31 - 1
        _, st = _run_decode(cfg, cd, inp["q"], qp, inp["seq_len"], max_len)
        assert st == 0


def test_decode_unaligned_query():
    """Query rows only 4-byte aligned (the ABI's minimum) take the scalar
    loads of the rotation: the output is bit-identical to the aligned call."""
    import paper_2606_26631_gb300 as prcr
    B, nL, H, Hq, D, max_len = 1, 4, 8, 32, 128, 933
    inp = make_decode_inputs(B, nL, H, Hq, D, max_len, False, device=DEV, seed=3)
    cfg = prcr.rope_cfg(nL, H, D, (16, 24, 24), 1e6)
    cd = prcr.cache_contiguous(inp["cache_k"], inp["cache_v"])
    q = inp["q"]
    buf = torch.empty(q.numel() + 2, dtype=torch.bfloat16, device=DEV)
    q_odd = buf[2:].view(q.shape)
    q_odd.copy_(q)
    assert q_odd.data_ptr() % 16 == 4
    ref, st0 = _run_decode(cfg, cd, q, inp["q_pos"], inp["seq_len"], max_len)
    got, st1 = _run_decode(cfg, cd, q_odd, inp["q_pos"], inp["seq_len"], max_len)
    assert st0 == 0 and st1 == 0
    assert torch.equal(ref, got)


# slots at the edges of a 16-slot tile, of a round of the head_dim 256 CTA's
# three warps (48) and of a chunk (512, 576), one per sequence of the batch;
# head counts that leave a CTA's last warps without a unit; the group's ends
@pytest.mark.parametrize("H,Hq,D,paged,bs", [(1, 8, 256, True, 7), (3, 3, 256, False, 16), (4, 28, 256, True, 16),
                                             (1, 8, 128, True, 7), (5, 5, 128, False, 16), (3, 21, 64, True, 16)])
@pytest.mark.parametrize("n_layers", [1, 9, 19, 40])
def test_decode_edges(H, Hq, D, paged, bs, n_layers):
    """Few layers: teams of warps per chunk (1) or per whole sequence (9, 19 and
    40: of 12, 6, 4 and 2; head_dim 64 at 40: one warp per chunk). head_dim 256: every product has 24 significant bits and is summed in
    float32, so a logit (sum of ~10 in magnitude over 48 MMAs) is off by about
    sqrt(48) 2^-24 10 = 4e-6 and the output by no more than twice that. Below,
    the file's bar: 16 significant bits per operand, 10 * 2^-17 = 8e-5."""
    import paper_2606_26631_gb300 as prcr
    sec = (D // 8, D // 4, D // 8)
    lens = [1, 15, 16, 17, 47, 48, 49, 511, 512, 513, 575, 576, 577, 593, 0, 1153]
    B, max_len = len(lens), 1153
    inp = make_decode_inputs(B, n_layers, H, Hq, D, max_len, paged, device=DEV, seed=31, block_size=bs)
    if paged:  # every sequence's table maps all of its slots
        nblk = -(-max_len // bs)
        pool = inp["cache_k"].shape[1]
        bt = (torch.arange(B * nblk, device=DEV, dtype=torch.int32).view(B, nblk) * 5) % pool
        inp["block_table"] = bt.contiguous()
    seq_len = torch.tensor(lens, dtype=torch.int32, device=DEV)
    cfg = prcr.rope_cfg(n_layers, H, D, sec, 1e6)
    cd = (prcr.cache_paged(inp["cache_k"], inp["cache_v"], inp["block_table"]) if paged
          else prcr.cache_contiguous(inp["cache_k"], inp["cache_v"]))
    out, st = _run_decode(cfg, cd, inp["q"], inp["q_pos"], seq_len, max_len)
    assert st == 0
    got, qv, l = out.cpu().numpy(), _f64(inp["q"]), n_layers - 1
    for b, n in enumerate(lens):
        if n == 0:
            assert np.all(got[b] == 0.0)
            continue
        s = torch.arange(n, device=DEV)
        if paged:
            blk = inp["block_table"][b][s // bs].long()
            K, V = (_f64(inp[x][l][blk, s % bs]) for x in ("cache_k", "cache_v"))
        else:
            K, V = (_f64(inp[x][b, l, :n]) for x in ("cache_k", "cache_v"))
        ref = O.decode_attention(qv[b, l], int(inp["q_pos"][b]), K, V, D, sec, 1e6)
        assert np.abs(got[b, l] - ref).max() / np.abs(V).max() <= (8e-6 if D == 256 else 1e-4), (b, n)


# (B, layers, H, Hq, D, max_len, paged), and what the host launches on 152 SMs
# (warps of a team or 0, chunks of max_len), which test_launch_cpu checks
LARGE = [
    ((1, 11, 3, 12, 128, 2000, True), (0, 42)),     # one warp per chunk, the merge of over 32
    ((16, 23, 5, 10, 128, 600, False), (0, 1)),     # one warp per sequence: more than 12 units per SM, 5 of 8 warps in use
    ((8, 23, 5, 10, 128, 700, True), (4, 1)),       # a large batch: teams of four, a chunk per sequence
    ((8, 23, 5, 10, 128, 2049, False), (4, 2)),     # and just over a chunk's 2048
    ((4, 28, 4, 28, 128, 4100, True), (4, 3)),      # and over two
    ((3, 25, 8, 8, 128, 4097, False), (4, 5)),      # few long sequences: chunks of 1024 at most
    ((16, 23, 5, 10, 64, 600, True), (0, 1)),       # head_dim 64
    ((8, 23, 5, 10, 64, 1100, False), (0, 3)),
]


@pytest.mark.parametrize("case", [c for c, _ in LARGE], ids=["B%dL%dH%dHq%dD%dS%d" % c[:6] for c, _ in LARGE])
def test_decode_large(case):
    """Many units or long sequences: sequences of no slot, one, a tile and its
    neighbours, a chunk of this call's and its neighbours, and max_len, at the
    first and last layer. The file's bar."""
    import paper_2606_26631_gb300 as prcr
    B, nL, H, Hq, D, max_len, paged = case
    sec = (D // 8, D // 4, D // 8)
    c = -(-(-(-max_len // 16)) // dict(LARGE)[case][1]) * 16
    lens = ([max_len, 0, 1, 17, c - 1, c, c + 1, 16] * 2)[:B] if B > 4 else [max_len, c + 1, c, 15][:B]
    lens = [min(n, max_len) for n in lens]
    g = torch.Generator(device=DEV).manual_seed(B + max_len)
    bs, nblk = 16, -(-max_len // 16)
    shape = (nL, B * nblk, bs, H, D) if paged else (B, nL, max_len, H, D)
    ck, cv = (torch.randn(shape, device=DEV, generator=g, dtype=torch.bfloat16) for _ in range(2))
    bt = torch.randperm(B * nblk, device=DEV, generator=g).to(torch.int32).view(B, nblk) if paged else None
    q = torch.randn((B, nL, Hq, D), device=DEV, generator=g, dtype=torch.bfloat16)
    q_pos = torch.arange(B, device=DEV, dtype=torch.int64) * 977 + max_len
    cfg = prcr.rope_cfg(nL, H, D, sec, 1e6)
    cd = prcr.cache_paged(ck, cv, bt) if paged else prcr.cache_contiguous(ck, cv)
    out, st = _run_decode(cfg, cd, q, q_pos, torch.tensor(lens, dtype=torch.int32, device=DEV), max_len)
    assert st == 0
    got, qv = out.cpu().numpy(), _f64(q)
    for b, n in enumerate(lens):
        if n == 0:
            assert np.all(got[b] == 0.0)
            continue
        s = torch.arange(n, device=DEV)
        for l in (0, nL - 1):
            K, V = (_f64(x[l][bt[b][s // bs].long(), s % bs] if paged else x[b, l, :n]) for x in (ck, cv))
            ref = O.decode_attention(qv[b, l], int(q_pos[b]), K, V, D, sec, 1e6)
            assert np.abs(got[b, l] - ref).max() / np.abs(V).max() <= 1e-4, (b, l, n)


def test_inject_then_decode():
    import paper_2606_26631_gb300 as prcr
    import parity_util as pu
    for name in ("qwen2vl-2b", "qwen25vl-7b"):
        wl = get(name)
        batch = make_batch(wl, device=DEV, context="random")
        B, nL, H, D = wl.n_seqs, wl.n_layers, wl.n_kv_heads, wl.head_dim
        Hq = {"qwen2vl-2b": 12, "qwen25vl-7b": 28}[name]
        # expected cache: context rows as given + the oracle's rows at the slots
        ctx_k = batch.cache_k.clone()
        ctx_v = batch.cache_v.clone()
        rv = pu.make_revisit(batch)
        rv.run()
        torch.cuda.synchronize()
        assert rv.status_value() == 0
        pl = pu.oracle_plan(batch)
        g = torch.Generator(device=DEV)
        g.manual_seed(11)
        q = torch.randn((B, nL, Hq, D), generator=g, device=DEV).to(torch.bfloat16)
        max_len = int(pl["cache_len_out"].max())
        cfg = rv.cfg
        out, st = _run_decode(cfg, rv.cache, q, rv.next_pos, rv.cache_len_out, max_len)
        assert st == 0
        got = out.cpu().numpy()
        qv = _f64(q)
        idx = batch.idx.cpu().numpy()
        for b in range(B):
            n_ctx = int(batch.cache_len_in[b])
            n_all = int(pl["cache_len_out"][b])
            K, V = _cache_rows(ctx_k, ctx_v, batch.block_table, b, n_all, batch.paged)
            toks = np.nonzero(pl["seq"] == b)[0]
            slots = pl["slot"][toks]
            k_raw = pu.bits(batch.store_k[b][:, torch.as_tensor(idx[toks], device=DEV).long()]
                            .transpose(0, 1))
            v_raw = pu.bits(batch.store_v[b][:, torch.as_tensor(idx[toks], device=DEV).long()]
                            .transpose(0, 1))
            k_hat = O.rebind_keys(k_raw, pl["pos"][toks], D, wl.sections, wl.theta)
            K[slots] = O.f64_to_bf16_rne(k_hat)
            V[slots] = O.bf16_bits_to_f64(v_raw)
            assert n_ctx + len(toks) == n_all
            for l in range(nL):
                ref = O.decode_attention(qv[b, l], int(pl["next_pos"][b]), K[:, l], V[:, l], D,
                                         wl.sections, wl.theta)
                err = np.abs(got[b, l] - ref).max() / np.abs(V[:, l]).max()
                assert err <= 1e-3, (name, b, l, err)


def test_decode_sees_only_relative_positions():
    import paper_2606_26631_gb300 as prcr
    import parity_util as pu
    wl = Workload(name="rel", n_layers=2, n_kv_heads=4, head_dim=128, sections=(16, 24, 24),
                  n_seqs=2, grids=((1, 24, 24),), selection="random", cache="contiguous",
                  cur_pos=("fixed", 3000), extra=(1, 1, 200, 300))
    outs = []
    for shift in (0, 12345):
        batch = make_batch(wl, device=DEV, seed=3)
        batch.p_txt += shift
        batch.cache_len_in.zero_()  # the cache holds only the revisited rows
        rv = pu.make_revisit(batch)
        rv.run()
        g = torch.Generator(device=DEV)
        g.manual_seed(5)
        q = torch.randn((2, 2, 16, 128), generator=g, device=DEV).to(torch.bfloat16)
        out, st = _run_decode(rv.cfg, rv.cache, q, rv.next_pos, rv.cache_len_out,
                              int(rv.cache_len_out.max()))
        assert st == 0 and rv.status_value() == 0
        outs.append(out.cpu().numpy())
    vmax = float(torch.abs(batch.store_v.float()).max())
    assert np.abs(outs[0] - outs[1]).max() / vmax <= 2e-3


def _layer_rows(inp, b, l, n):
    """[n, H, D] value arrays of slots 0..n-1 of sequence b at layer l (paged)."""
    s = torch.arange(n, device=inp["cache_k"].device)
    bs = inp["cache_k"].shape[2]
    blk = inp["block_table"][b][s // bs].long()
    off = s % bs
    return _f64(inp["cache_k"][l, blk, off]), _f64(inp["cache_v"][l, blk, off])


@pytest.mark.slow
def test_decode_full_size_sampled():
    """The decode configuration bench.py times (qwen3vl-8b shape: 16 sequences
    of up to 8192 slots, 36 layers, 8 KV heads, 32 query heads, paged, the same
    seed, so the same chunk split and merge launch); sampled (sequence, layer)
    pairs, every query head, against the oracle."""
    import paper_2606_26631_gb300 as prcr
    wl = get("qwen3vl-8b")
    B, nL, H, D = wl.n_seqs, wl.n_layers, wl.n_kv_heads, wl.head_dim
    Hq, max_len = 4 * H, 8192
    inp = make_decode_inputs(B, nL, H, Hq, D, max_len, True, device=DEV, seed=1)
    cfg = prcr.rope_cfg(nL, H, D, wl.sections, wl.theta)
    cd = prcr.cache_paged(inp["cache_k"], inp["cache_v"], inp["block_table"])
    out, st = _run_decode(cfg, cd, inp["q"], inp["q_pos"], inp["seq_len"], max_len)
    assert st == 0
    got = out.cpu().numpy()
    qv = _f64(inp["q"])
    for b in (0, B // 2, B - 1):
        n = int(inp["seq_len"][b])
        for l in (0, nL // 2, nL - 1):
            K, V = _layer_rows(inp, b, l, n)
            ref = O.decode_attention(qv[b, l], int(inp["q_pos"][b]), K, V, D, wl.sections, wl.theta)
            err = np.abs(got[b, l] - ref).max() / np.abs(V).max()
            assert err <= 1e-4, (b, l, n, err)
    del inp
    torch.cuda.empty_cache()


@pytest.mark.parametrize("max_len,paged,nL", [(100, False, 1), (1200, True, 2), (5000, False, 30)])
def test_decode_infinities_d256(max_len, paged, nL):
    """head_dim 256, where operands are split into pieces: a key whose logit is
    -inf has weight 0 (the output is the attention over the other slots), one
    whose logit is +inf makes its head NaN, an infinite value stays infinite in
    its dimension and touches no other. Unsplit, few and many chunks."""
    import paper_2606_26631_gb300 as prcr
    H, Hq, D, dim, slot = 2, 6, 256, 37, max_len - 30
    P, g = D // 2, Hq // H
    inp = make_decode_inputs(1, nL, H, Hq, D, max_len, paged, device=DEV, seed=12)
    ck, cv, bt = inp["cache_k"], inp["cache_v"], inp["block_table"]

    def put(cache, h, d, x):
        if paged:
            cache[:, int(bt[0, slot // 16]), slot % 16, h, d] = x
        else:
            cache[0, :, slot, h, d] = x

    cfg = prcr.rope_cfg(nL, H, D, (48, 40, 40), 1e6)
    cd = prcr.cache_paged(ck, cv, bt) if paged else prcr.cache_contiguous(ck, cv)
    p, l = int(inp["q_pos"][0]), nL - 1
    qv = _f64(inp["q"])[0, l]
    K, V = (x[:, l] for x in _cache_rows(ck, cv, bt, 0, max_len, paged))
    others = np.arange(max_len) != slot
    full = O.decode_attention(qv, p, K, V, D, (48, 40, 40), 1e6)
    without = O.decode_attention(qv, p, K[others], V[others], D, (48, 40, 40), 1e6)
    angle = p * 1e6 ** (-2.0 * dim / D)
    rot = qv[:, dim] * np.cos(angle) - qv[:, dim + P] * np.sin(angle)  # the query's component that meets the infinite key
    vmax = np.abs(V).max()
    for sign in (-1.0, 1.0):
        kept = ck.clone()
        put(ck, 0, dim, sign * float("inf"))
        out, st = _run_decode(cfg, cd, inp["q"], inp["q_pos"], inp["seq_len"], max_len)
        ck.copy_(kept)
        got = out[0, l].cpu().numpy()
        assert st == 0
        for h in range(Hq):
            if h < g and sign * rot[h] > 0:
                assert np.all(np.isnan(got[h])), h
            else:
                assert np.abs(got[h] - (without if h < g else full)[h]).max() <= 8e-6 * vmax, h
    kept = cv.clone()
    put(cv, 1, 200, float("-inf"))
    out, st = _run_decode(cfg, cd, inp["q"], inp["q_pos"], inp["seq_len"], max_len)
    cv.copy_(kept)
    got = out[0, l].cpu().numpy()
    assert st == 0 and np.all(np.isneginf(got[g:, 200]))
    got[g:, 200] = full[g:, 200]
    assert np.abs(got - full).max() <= 8e-6 * vmax
