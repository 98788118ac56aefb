"""GPU checks of prcr_select_topk (attention-driven selection, Sec. 2.1 /
Eq. 3, under the reading in the oracle's header).

Relevance: float32 on the GPU against the oracle's float64 ads_relevance,
relative error <= 1e-4. Selection: where floating point decides an integer,
the check is that (a) the set is exactly the top-k of the relevance the
kernel itself reports (ties to the lower index), (b) it is a valid top-k of
the oracle's relevance up to the measured relevance error, and (c) it equals
the oracle's ads_select whenever the oracle's k-th and (k+1)-th values are
further apart than that error. Ties are forced with an all-zero key layer.
"""
import numpy as np
import pytest
import torch

from oracle import prcr_oracle as O
from workloads import Workload, get, make_batch

pytestmark = pytest.mark.gpu

DEV = "cuda:0"


def _select(batch, layer, Hq, k, q, q_pos):
    import paper_2606_26631_gb300 as prcr
    wl = batch.wl
    B, M = wl.n_seqs, wl.n_tokens
    cfg = prcr.rope_cfg(wl.n_layers, wl.n_kv_heads, wl.head_dim, wl.sections, wl.theta)
    sd = prcr.store_desc(batch.store_k, batch.store_v, batch.coords)
    idx = torch.full((B * k,), -7, dtype=torch.int32, device=DEV)
    sro = torch.full((B + 1,), -7, dtype=torch.int32, device=DEV)
    rto = torch.full((B + 1,), -7, dtype=torch.int32, device=DEV)
    score = torch.full((B, M), -1.0, dtype=torch.float32, device=DEV)
    ws = torch.empty(prcr.select_workspace_size(B, Hq, M), dtype=torch.uint8, device=DEV)
    prcr.select_topk(cfg, sd, layer, q, q_pos, k, idx, sro, rto, ws, score)
    torch.cuda.synchronize()
    return idx.view(B, k).cpu().numpy(), sro.cpu().numpy(), rto.cpu().numpy(), score.cpu().numpy()


def _topk_by(values, k):
    order = np.lexsort((np.arange(len(values)), -values))
    return np.sort(order[:k])


# odd shapes: head_dim 48 (3 of 4 lanes per row active), 3 KV heads with a
# GQA group of 3, two grids per sequence; head_dim 256 with a group of 2;
# token counts that leave a ragged last tile
SHAPES = {
    "sel-odd": Workload(name="sel-odd", n_layers=2, n_kv_heads=3, head_dim=48, sections=(8, 8, 8),
                        n_seqs=3, grids=((3, 5, 5), (1, 4, 4)), selection="random",
                        cache="contiguous", cur_pos=("uniform", 100, 4000), extra=(0, 3, 0, 37)),
    "sel-d256": Workload(name="sel-d256", n_layers=1, n_kv_heads=2, head_dim=256,
                         sections=(40, 44, 44), n_seqs=2, grids=((2, 10, 13),), selection="random",
                         cache="contiguous", cur_pos=("uniform", 500, 900), extra=(1, 2, 1, 40)),
    # 1500 tokens over 24 tiles of 64 (ragged last tile), 16 query heads
    "sel-1500": Workload(name="sel-1500", n_layers=1, n_kv_heads=4, head_dim=128,
                         sections=(16, 24, 24), n_seqs=2, grids=((1, 30, 50),), selection="random",
                         cache="contiguous", cur_pos=("uniform", 2000, 9000), extra=(1, 1, 1, 40)),
}


@pytest.mark.parametrize("name,Hq,k,layer", [("qwen25vl-7b", 28, 64, 5), ("qwen3vl-8b", 32, 300, 35),
                                             ("tiny", 2, 16, 1), ("qwen2vl-2b", 4, 100, 20),
                                             ("sel-odd", 9, 20, 1), ("sel-d256", 4, 30, 0),
                                             ("sel-1500", 16, 200, 0)])
def test_select_parity(name, Hq, k, layer):
    wl = SHAPES.get(name) or get(name)
    batch = make_batch(wl, device=DEV)
    B, M, D = wl.n_seqs, wl.n_tokens, wl.head_dim
    g = torch.Generator(device=DEV)
    g.manual_seed(17)
    q = (3.0 * torch.randn((B, Hq, D), generator=g, device=DEV)).to(torch.bfloat16)
    idx, sro, rto, score = _select(batch, layer, Hq, k, q, batch.p_txt)
    assert np.array_equal(sro, np.arange(B + 1))
    assert np.array_equal(rto, k * np.arange(B + 1))
    qv = O.bf16_bits_to_f64(q.view(torch.int16).cpu().numpy())
    coords = batch.coords.cpu().numpy()
    for b in range(min(B, 4)):
        k_raw = batch.store_k[b, layer].view(torch.int16).cpu().numpy()
        ref = O.ads_relevance(qv[b], int(batch.p_txt[b]), k_raw, coords[b], D, wl.sections, wl.theta)
        rel_err = np.abs(score[b] - ref) / ref
        assert rel_err.max() <= 1e-4, rel_err.max()
        sel = idx[b]
        assert len(set(sel.tolist())) == k and np.all(np.diff(sel) > 0)
        assert np.array_equal(sel, _topk_by(score[b].astype(np.float64), k))  # (a)
        tol = 2 * np.abs(score[b] - ref).max() + 1e-12
        chosen = np.zeros(M, dtype=bool)
        chosen[sel] = True
        if k < M:
            assert ref[chosen].min() >= ref[~chosen].max() - tol  # (b)
            srt = np.sort(ref)[::-1]
            if srt[k - 1] - srt[k] > tol:
                assert np.array_equal(sel, O.ads_select(ref, k))  # (c)


def test_select_ties_and_full_set():
    wl = get("qwen2vl-2b")
    batch = make_batch(wl, device=DEV)
    batch.store_k[:, 3].zero_()  # every logit of layer 3 is 0: all relevances tie
    B, M, D = 1, wl.n_tokens, wl.head_dim
    q = torch.randn((B, 2, D), device=DEV).to(torch.bfloat16)
    idx, _, _, score = _select(batch, 3, 2, 100, q, batch.p_txt)
    assert np.array_equal(idx[0], np.arange(100))
    assert np.allclose(score[0], 1.0 / M, rtol=1e-6)
    idx, _, _, _ = _select(batch, 7, 2, M, q, batch.p_txt)
    assert np.array_equal(idx[0], np.arange(M))


def test_select_feeds_rebind_inject():
    """The selection's outputs are a valid revisit batch for prcr_rebind_inject."""
    import paper_2606_26631_gb300 as prcr
    wl = get("qwen25vl-7b")
    batch = make_batch(wl, device=DEV)
    B, k = wl.n_seqs, 48
    q = torch.randn((B, 4, wl.head_dim), device=DEV).to(torch.bfloat16)
    cfg = prcr.rope_cfg(wl.n_layers, wl.n_kv_heads, wl.head_dim, wl.sections, wl.theta)
    sd = prcr.store_desc(batch.store_k, batch.store_v, batch.coords)
    idx = torch.empty(B * k, dtype=torch.int32, device=DEV)
    sro = torch.empty(B + 1, dtype=torch.int32, device=DEV)
    rto = torch.empty(B + 1, dtype=torch.int32, device=DEV)
    ws = torch.empty(prcr.select_workspace_size(B, 4, wl.n_tokens), dtype=torch.uint8, device=DEV)
    prcr.select_topk(cfg, sd, 0, q, batch.p_txt, k, idx, sro, rto, ws)
    # a cache with room for k slots after each sequence's context
    clen = batch.cache_len_in
    nblk = int(((clen.max() + k) // 16 + 2).item())
    bt = torch.arange(B * nblk, dtype=torch.int32, device=DEV).view(B, nblk).contiguous()
    ck = torch.full((wl.n_layers, B * nblk, 16, wl.n_kv_heads, wl.head_dim), -1,
                    dtype=torch.int16, device=DEV).view(torch.bfloat16)
    cv = ck.clone()
    rv = prcr.Revisit(cfg, batch.store_k, batch.store_v, batch.coords, ck, cv, bt, sro, rto, idx,
                      batch.p_txt, clen)
    rv.run()
    torch.cuda.synchronize()
    assert rv.status_value() == 0
    assert torch.equal(rv.cache_len_out, clen + k)
    assert torch.equal(rv.next_pos, batch.p_txt + 1)
    written = int((ck.view(torch.int16) != -1).sum().item())
    assert written == B * k * wl.n_layers * wl.n_kv_heads * wl.head_dim


@pytest.mark.slow
def test_select_full_size_sampled():
    """The selection configuration bench.py times on the stress shape (32
    sequences x 16,384 tokens, 32 query heads, k = 4096, last layer); sampled
    sequences checked like test_select_parity."""
    wl = get("stress")
    batch = make_batch(wl, device=DEV)
    B, M, H, D = wl.n_seqs, wl.n_tokens, wl.n_kv_heads, wl.head_dim
    Hq, k, layer = 4 * H, batch.total_k // B, wl.n_layers - 1
    q = torch.randn((B, Hq, D), device=DEV, generator=torch.Generator(device=DEV).manual_seed(3)
                    ).to(torch.bfloat16)
    idx, sro, rto, score = _select(batch, layer, Hq, k, q, batch.p_txt)
    assert np.array_equal(sro, np.arange(B + 1))
    assert np.array_equal(rto, k * np.arange(B + 1))
    qv = O.bf16_bits_to_f64(q.view(torch.int16).cpu().numpy())
    coords = batch.coords.cpu().numpy()
    for b in (0, B // 2, B - 1):
        k_raw = batch.store_k[b, layer].view(torch.int16).cpu().numpy()
        ref = O.ads_relevance(qv[b], int(batch.p_txt[b]), k_raw, coords[b], D, wl.sections, wl.theta)
        assert (np.abs(score[b] - ref) / ref).max() <= 1e-4
        sel = idx[b]
        assert np.array_equal(sel, _topk_by(score[b].astype(np.float64), k))
        tol = 2 * np.abs(score[b] - ref).max() + 1e-12
        chosen = np.zeros(M, dtype=bool)
        chosen[sel] = True
        assert ref[chosen].min() >= ref[~chosen].max() - tol
    del batch
    torch.cuda.empty_cache()


def test_select_interleaved_layout():
    """The interleaved M-RoPE band layout (pair i to h when i % 3 == 1, to w
    when i % 3 == 2, within their sections) on both logits kernels: head_dim
    128 (tensor cores) and 48 (CUDA cores)."""
    import paper_2606_26631_gb300 as prcr
    for wl, Hq, k, layer in ((get("qwen2vl-2b"), 8, 100, 9), (SHAPES["sel-odd"], 9, 20, 1)):
        batch = make_batch(wl, device=DEV)
        B, M, D = wl.n_seqs, wl.n_tokens, wl.head_dim
        cfg = prcr.rope_cfg(wl.n_layers, wl.n_kv_heads, D, wl.sections, wl.theta,
                            O.LAYOUT_INTERLEAVED)
        sd = prcr.store_desc(batch.store_k, batch.store_v, batch.coords)
        q = (3.0 * torch.randn((B, Hq, D), device=DEV,
                               generator=torch.Generator(device=DEV).manual_seed(8))).to(torch.bfloat16)
        idx = torch.empty(B * k, dtype=torch.int32, device=DEV)
        sro = torch.empty(B + 1, dtype=torch.int32, device=DEV)
        rto = torch.empty(B + 1, dtype=torch.int32, device=DEV)
        score = torch.empty((B, M), dtype=torch.float32, device=DEV)
        ws = torch.empty(prcr.select_workspace_size(B, Hq, M), dtype=torch.uint8, device=DEV)
        prcr.select_topk(cfg, sd, layer, q, batch.p_txt, k, idx, sro, rto, ws, score)
        torch.cuda.synchronize()
        qv = O.bf16_bits_to_f64(q.view(torch.int16).cpu().numpy())
        coords = batch.coords.cpu().numpy()
        sc = score.cpu().numpy()
        sel = idx.view(B, k).cpu().numpy()
        for b in range(B):
            k_raw = batch.store_k[b, layer].view(torch.int16).cpu().numpy()
            ref = O.ads_relevance(qv[b], int(batch.p_txt[b]), k_raw, coords[b], D, wl.sections,
                                  wl.theta, O.LAYOUT_INTERLEAVED)
            assert (np.abs(sc[b] - ref) / ref).max() <= 1e-4, wl.name
            assert np.array_equal(sel[b], _topk_by(sc[b].astype(np.float64), k))


# Coordinate structures beyond one image per sequence: two images of widths
# 4 and 16 in one sequence, a 24-wide video with a t section that ends inside
# an 8-pair group, head_dim 64 with a GQA group of 8, and a sequence whose
# coordinates are shuffled (no token shares a row or column with its index
# neighbours). The relevance must not depend on any grid regularity.
GRID_SHAPES = {
    "rot-w4-w16": (Workload(name="rot-w4-w16", n_layers=1, n_kv_heads=2, head_dim=128,
                            sections=(24, 20, 20), n_seqs=2, grids=((2, 6, 4), (1, 9, 16)),
                            selection="random", cache="contiguous", cur_pos=("uniform", 300, 5000),
                            extra=(1, 1, 1, 20)), 8, False),
    "rot-t20": (Workload(name="rot-t20", n_layers=1, n_kv_heads=4, head_dim=128,
                         sections=(20, 20, 24), n_seqs=2, grids=((3, 11, 24),), selection="random",
                         cache="contiguous", cur_pos=("uniform", 300, 5000), extra=(1, 1, 1, 20)),
                16, False),
    "rot-d64-g8": (Workload(name="rot-d64-g8", n_layers=1, n_kv_heads=2, head_dim=64,
                            sections=(8, 12, 12), n_seqs=2, grids=((1, 20, 24),), selection="random",
                            cache="contiguous", cur_pos=("uniform", 300, 5000), extra=(1, 1, 1, 20)),
                   16, False),
    "rot-shuffled": (get("qwen2vl-2b"), 8, True),
}


@pytest.mark.parametrize("name", sorted(GRID_SHAPES))
def test_select_coordinate_structures(name):
    wl, Hq, shuffle = GRID_SHAPES[name]
    batch = make_batch(wl, device=DEV)
    B, M, D = wl.n_seqs, wl.n_tokens, wl.head_dim
    if shuffle:
        perm = torch.randperm(M, generator=torch.Generator().manual_seed(5)).to(DEV)
        batch.coords[0] = batch.coords[0][perm].clone()
    k = min(40, M - 1)
    g = torch.Generator(device=DEV)
    g.manual_seed(29)
    q = (3.0 * torch.randn((B, Hq, D), generator=g, device=DEV)).to(torch.bfloat16)
    idx, sro, rto, score = _select(batch, 0, Hq, k, q, batch.p_txt)
    qv = O.bf16_bits_to_f64(q.view(torch.int16).cpu().numpy())
    coords = batch.coords.cpu().numpy()
    for b in range(B):
        k_raw = batch.store_k[b, 0].view(torch.int16).cpu().numpy()
        ref = O.ads_relevance(qv[b], int(batch.p_txt[b]), k_raw, coords[b], D, wl.sections, wl.theta)
        rel_err = np.abs(score[b] - ref) / ref
        assert rel_err.max() <= 1e-4, (b, rel_err.max())
        assert np.array_equal(idx[b], _topk_by(score[b].astype(np.float64), k))


# Shapes whose logits work divides unevenly over the persistent grid of a
# 152-SM GB300 (two CTAs per SM): the last items are split in halves by KV
# heads, here over groups of 3 KV heads (halves of 2 and 1) and 5 (3 and 2,
# then 2 and 1 for the group of 2). The split items are the last ones, i.e.
# the last sequences', which the test checks against the oracle.
HALVES = {
    "halves-h6": (Workload(name="halves-h6", n_layers=1, n_kv_heads=6, head_dim=128,
                           sections=(16, 24, 24), n_seqs=24, grids=((1, 40, 40),), selection="random",
                           cache="contiguous", cur_pos=("uniform", 2000, 9000), extra=(1, 1, 1, 40)), 12),
    "halves-h5-d64": (Workload(name="halves-h5-d64", n_layers=1, n_kv_heads=5, head_dim=64,
                               sections=(8, 12, 12), n_seqs=20, grids=((1, 40, 50),), selection="random",
                               cache="contiguous", cur_pos=("uniform", 2000, 9000), extra=(1, 1, 1, 40)), 15),
}


@pytest.mark.parametrize("name", sorted(HALVES))
def test_select_leftover_halves(name):
    wl, Hq = HALVES[name]
    batch = make_batch(wl, device=DEV)
    B, M, D = wl.n_seqs, wl.n_tokens, wl.head_dim
    k = 100
    g = torch.Generator(device=DEV)
    g.manual_seed(29)
    q = (3.0 * torch.randn((B, Hq, D), generator=g, device=DEV)).to(torch.bfloat16)
    idx, _, _, score = _select(batch, 0, Hq, k, q, batch.p_txt)
    qv = O.bf16_bits_to_f64(q.view(torch.int16).cpu().numpy())
    coords = batch.coords.cpu().numpy()
    for b in (0, B - 3, B - 2, B - 1):
        k_raw = batch.store_k[b, 0].view(torch.int16).cpu().numpy()
        ref = O.ads_relevance(qv[b], int(batch.p_txt[b]), k_raw, coords[b], D, wl.sections, wl.theta)
        assert (np.abs(score[b] - ref) / ref).max() <= 1e-4, b
        assert np.array_equal(idx[b], _topk_by(score[b].astype(np.float64), k))


# raw keys through the one-kernel path (a cluster per sequence) and past it:
# a pass of cos/sin holds 16 tiles of 16 tokens at head_dim 64, 8 at 128 and 4
# at 256; an odd KV-head count; the last rank of a cluster short or empty
RAW_SIZES = [  # (B, M, k, H, Hq, D)
    (1, 33, 5, 1, 8, 128), (2, 769, 32, 3, 3, 128), (1, 2065, 700, 5, 20, 64), (9, 1030, 50, 2, 14, 256), (1, 5000, 64, 2, 8, 256),
    (150, 200, 9, 1, 2, 64), (30, 2500, 100, 4, 16, 128),
]


@pytest.mark.parametrize("B,M,k,H,Hq,D", RAW_SIZES, ids=[f"B{c[0]}M{c[1]}k{c[2]}H{c[3]}Hq{c[4]}D{c[5]}" for c in RAW_SIZES])
def test_select_raw_sizes(B, M, k, H, Hq, D):
    """Relevances within the file's bar, and exactly the top-k of them."""
    import paper_2606_26631_gb300 as prcr
    sec = (D // 8, D // 4 - D // 16, D // 2 - D // 8 - (D // 4 - D // 16))
    g = torch.Generator(device=DEV).manual_seed(200 + M)
    store_k = torch.randn((B, 1, M, H, D), device=DEV, generator=g).to(torch.bfloat16)
    coords = torch.randint(0, 60, (B, M, 3), device=DEV, generator=g, dtype=torch.int32)
    coords[..., 2] = torch.arange(M, device=DEV, dtype=torch.int32) % 40
    q = (2.0 * torch.randn((B, Hq, D), device=DEV, generator=g)).to(torch.bfloat16)
    q_pos = torch.arange(B, device=DEV, dtype=torch.int64) * 41 + 700
    idx = torch.full((B * k,), -7, dtype=torch.int32, device=DEV)
    sro = torch.full((B + 1,), -7, dtype=torch.int32, device=DEV)
    rto = torch.full((B + 1,), -7, dtype=torch.int32, device=DEV)
    score = torch.full((B, M), -1.0, dtype=torch.float32, device=DEV)
    ws = torch.empty(prcr.select_workspace_size(B, Hq, M), dtype=torch.uint8, device=DEV)
    cfg = prcr.rope_cfg(1, H, D, sec, 1e6)
    prcr.select_topk(cfg, prcr.store_desc(store_k, torch.zeros_like(store_k), coords), 0, q, q_pos, k, idx, sro, rto, ws, score)
    torch.cuda.synchronize()
    got, sel = score.cpu().numpy(), idx.view(B, k).cpu().numpy()
    assert np.array_equal(sro.cpu().numpy(), np.arange(B + 1)) and np.array_equal(rto.cpu().numpy(), k * np.arange(B + 1))
    qv = O.bf16_bits_to_f64(q.view(torch.int16).cpu().numpy())
    for b in sorted({0, B // 2, B - 1}):
        ref = O.ads_relevance(qv[b], int(q_pos[b]), store_k[b, 0].view(torch.int16).cpu().numpy(), coords[b].cpu().numpy(), D, sec, 1e6)
        assert (np.abs(got[b] - ref) / ref).max() <= 1e-4
    for b in range(B):
        assert np.array_equal(sel[b], _topk_by(got[b].astype(np.float64), k)), b


@pytest.mark.parametrize("M", [70, 9000])  # one kernel, and two
def test_select_infinite_key_d256(M):
    """head_dim 256, where the keys are split into pieces: a key whose logit is
    -inf has relevance 0 and leaves the others as they are without it."""
    import paper_2606_26631_gb300 as prcr
    D, P, m, k, sec = 256, 128, 41, 9, (48, 40, 40)
    g = torch.Generator(device=DEV).manual_seed(7)
    store_k = torch.randn((1, 1, M, 1, D), device=DEV, generator=g).to(torch.bfloat16)
    coords = torch.randint(0, 60, (1, M, 3), device=DEV, generator=g, dtype=torch.int32)
    q = torch.randn((1, 1, D), device=DEV, generator=g).to(torch.bfloat16)
    q_pos = torch.full((1,), 700, dtype=torch.int64, device=DEV)
    qv = O.bf16_bits_to_f64(q.view(torch.int16).cpu().numpy())[0]
    kv, cv = store_k[0, 0].view(torch.int16).cpu().numpy(), coords[0].cpu().numpy()
    others = np.arange(M) != m
    ref = O.ads_relevance(qv, 700, kv[others], cv[others], D, sec, 1e6)
    for i in range(P):  # a pair both of whose turned components meet the query with one sign
        angle = float(cv[m, 0 if i < 48 else 1 if i < 88 else 2] - 700) * 1e6 ** (-2.0 * i / D)
        x, y = qv[0, i] * np.cos(angle), qv[0, i + P] * np.sin(angle)
        if x * y > 1e-3:
            break
    store_k[0, 0, m, 0, i] = -float("inf") if x > 0 else float("inf")
    idx, sro, rto = (torch.zeros(n, dtype=torch.int32, device=DEV) for n in (k, 2, 2))
    score = torch.full((1, M), -1.0, dtype=torch.float32, device=DEV)
    ws = torch.empty(prcr.select_workspace_size(1, 1, M), dtype=torch.uint8, device=DEV)
    prcr.select_topk(prcr.rope_cfg(1, 1, D, sec, 1e6), prcr.store_desc(store_k, store_k, coords), 0, q, q_pos, k, idx, sro, rto, ws, score)
    got = score[0].cpu().numpy()
    assert got[m] == 0.0
    assert (np.abs(got[others] - ref) / ref).max() <= 1e-4
    assert np.array_equal(idx.cpu().numpy(), _topk_by(got.astype(np.float64), k))


@pytest.mark.parametrize("B,M,H,Hq,D", [(3, 8192, 4, 32, 256), (2, 4099, 4, 28, 96), (16, 600, 4, 32, 256)])
def test_select_weights_sum_to_one(B, M, H, Hq, D):
    """Raw keys where the logits have float32's accuracy (head dims other than
    64 and 128): the relevances of a sequence sum to 1 within half a unit in the
    last place, 2^-24. Their rounding errors, and the heads' normalisers', are
    thousands of independent ones that average out; what would remain is an
    exp in the denominators that is off to one side."""
    import paper_2606_26631_gb300 as prcr
    sec = (D // 8, D // 4, D // 8)
    g = torch.Generator(device=DEV).manual_seed(M)
    store_k = torch.randn((B, 1, M, H, D), device=DEV, generator=g).to(torch.bfloat16)
    coords = torch.randint(0, 60, (B, M, 3), device=DEV, generator=g, dtype=torch.int32)
    q = torch.randn((B, Hq, D), device=DEV, generator=g).to(torch.bfloat16)
    q_pos = torch.arange(B, device=DEV, dtype=torch.int64) * 41 + 700
    idx, sro, rto = (torch.zeros(n, dtype=torch.int32, device=DEV) for n in (B, B + 1, B + 1))
    score = torch.zeros((B, M), dtype=torch.float32, device=DEV)
    ws = torch.empty(prcr.select_workspace_size(B, Hq, M), dtype=torch.uint8, device=DEV)
    prcr.select_topk(prcr.rope_cfg(1, H, D, sec, 1e6), prcr.store_desc(store_k, store_k, coords), 0, q, q_pos, 1, idx, sro, rto, ws, score)
    assert float((score.double().sum(1) - 1.0).mean().abs()) <= 2.0 ** -24


@pytest.mark.parametrize("M", [33, 70, 2050, 9000])  # one kernel, and two
@pytest.mark.parametrize("D", [96, 128, 256])
def test_select_nan_key(D, M):
    """A NaN key makes every relevance of its head NaN, wherever it lies."""
    import paper_2606_26631_gb300 as prcr
    sec = (D // 8, D // 4, D // 8)
    g = torch.Generator(device=DEV).manual_seed(5)
    store_k = torch.randn((1, 1, M, 1, D), device=DEV, generator=g).to(torch.bfloat16)
    coords = torch.randint(0, 60, (1, M, 3), device=DEV, generator=g, dtype=torch.int32)
    q = torch.randn((1, 1, D), device=DEV, generator=g).to(torch.bfloat16)
    q_pos = torch.full((1,), 700, dtype=torch.int64, device=DEV)
    idx, sro, rto = (torch.zeros(n, dtype=torch.int32, device=DEV) for n in (3, 2, 2))
    score = torch.zeros((1, M), dtype=torch.float32, device=DEV)
    ws = torch.empty(prcr.select_workspace_size(1, 1, M), dtype=torch.uint8, device=DEV)
    for m in (0, M // 2, M - 1):
        keep = store_k[0, 0, m].clone()
        store_k[0, 0, m, 0, 3] = float("nan")
        prcr.select_topk(prcr.rope_cfg(1, 1, D, sec, 1e6), prcr.store_desc(store_k, store_k, coords), 0, q, q_pos, 3, idx, sro, rto, ws, score)
        store_k[0, 0, m] = keep
        assert bool(torch.isnan(score).all()) and idx.tolist() == [0, 1, 2], m
