"""CPU checks of what the host side launches, against a CUDA runtime that only
keeps the launches (fake_gpu)."""
import ctypes as C
import threading

import pytest

import fake_gpu as F


def test_shared_memory_limits_only_rise():
    """The limit belongs to the kernel, not to the call: a call that lowers it
    fails another thread's launch. Calls of one kernel with different needs
    (decode teams of 12, 6, 4, 3 and 2 warps, one warp per chunk and head_dim
    256; cached and raw selections past one cluster), from several threads."""
    b8, b256, small = F.cfg(36, 8, 128), F.cfg(26, 4, 256), F.cfg(2, 4, 128)
    calls = [(lambda c=c, n=n, m=m: F.decode(c, n, 4, m, 1 << 40)) for c in (small, b8, b256) for n, m in ((1, 200), (1, 933), (3, 933), (16, 300), (16, 8192))]
    calls += [(lambda H=H, D=D, n=n, m=m: F.select_cached(F.cfg(1, H, D), n, 4, m))
              for H, D in ((8, 128), (2, 128)) for n, m in ((1, 32768), (4, 16384), (32, 8192))]
    calls += [(lambda H=H, D=D, n=n: F.select_raw(F.cfg(1, H, D), n, 4, 16384))
              for H, D in ((8, 128), (2, 128), (2, 96), (8, 96), (4, 256)) for n in (1, 32)]
    F.lib()
    bad, done = [], []

    def work(first):
        for i in range(3 * len(calls)):
            which = (i + first) % len(calls)
            rc = calls[which]()
            if rc:
                bad.append((which, rc))
        done.append(first)

    threads = [threading.Thread(target=work, args=(7 * t,)) for t in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    names = {n for n, _ in F.launches()}
    for part in ("decode_kernelILi128ELb1E", "decode_kernelILi128ELb0E", "decode_wide", "select_logits", "ads_logits_mma", "ads_logits_kernel"):
        assert any(part in n for n in names), part
    assert not bad and len(done) == len(threads), bad[:5]
    assert F.lib().fake_lowered() == 0


@pytest.mark.parametrize("D", [64, 128, 256])
def test_decode_workspace_holds_shorter_calls(D):
    """A workspace sized once, for the longest length, is enough for every
    shorter one: no length needs more chunks than the size for it holds, and
    sizes fall nowhere as max_len grows. Lengths around the rules' lines."""
    for layers, H in ((1, 1), (1, 4), (2, 4), (4, 1), (26, 4), (36, 8), (3, 3)):
        c = F.cfg(layers, H, D)
        for seqs in (1, 2, 5, 16):
            unit = seqs * layers * H * (D + 2) * 4  # one head per KV head
            lengths = sorted({*range(1, 700, 7), *range(1, 40000, 391), *(m * e + d for m in (16, 48, 512, 576, 640, 2048, 4080, 4096)
                                                                       for e in (1, 2, 3, 9, 38, 76) for d in (-1, 0, 1)), 30000, 200000})
            before = 0
            for n in lengths:
                size = F.workspace(c, seqs, 1, n)
                assert size >= before, (layers, H, seqs, n)
                before = size
                F.launches()
                assert F.decode(c, seqs, 1, n, 1 << 40) == 0
                splits = F.launches()[0][1][5]
                assert size >= (unit * splits if splits > 1 else 0), (layers, H, seqs, n, splits)
    # the calls that were refused: (layers, KV heads, sequences, longest, shorter)
    for layers, H, seqs, longest, shorter in ((1, 4, 1, 3649, 3601), (2, 4, 1, 1825, 1777), (1, 4, 5, 721, 673), (1, 1, 2, 7297, 7249)):
        c = F.cfg(layers, H, D)
        assert F.decode(c, seqs, 2, shorter, F.workspace(c, seqs, 2, longest)) == 0


def test_rebind_looks_ahead_only_behind_its_own_plan():
    """The rebind kernel reads the batch before its wait only where this call's
    plan kernel, which waits first, stands before it. prcr_rebind_apply may
    follow any kernel, one that still writes the batch among them."""
    c = F.cfg(28, 4, 128)
    F.launches()
    assert F.revisit(c, 8, 512) == 0
    plan, rebind = F.launches()
    assert "plan_kernel" in plan[0] and "rebind_kernel" in rebind[0] and rebind[1][5] > 0
    assert F.revisit(c, 8, 512, "plan") == 0 and F.revisit(c, 8, 512, "apply") == 0
    plan, alone = F.launches()
    assert "plan_kernel" in plan[0] and "rebind_kernel" in alone[0]
    assert alone[1][:5] == rebind[1][:5] and alone[1][5] == 0


@pytest.mark.parametrize("D", [64, 128, 256])
@pytest.mark.parametrize("max_len", [2 ** 31 - 17, 2 ** 31 - 1, 2 ** 31, 2 ** 32, 2 ** 40])
def test_decode_any_max_len(D, max_len):
    """A paged cache's capacity, and max_len with it, may exceed an int32 (a
    sequence's length cannot): the split still covers every length."""
    for layers, H, seqs in ((1, 1, 1), (36, 8, 1), (36, 8, 16)):
        c = F.cfg(layers, H, D)
        F.launches()
        assert F.decode(c, seqs, 2, max_len, 1 << 60, F.paged(c, seqs, 2 ** 30, 2 ** 10)) == 0
        splits, chunk = F.launches()[0][1][5:7]
        assert 0 < chunk <= 2 ** 30 and splits * chunk >= 2 ** 31 - 17, (splits, chunk)


@pytest.mark.parametrize("n_tokens", [64, 16384])  # one kernel, and two
def test_cached_selection_of_a_cache_without_rows(n_tokens):
    """A token without a cache row reads the cache's first row (and drops it);
    a cache that has none is no readable memory, so the workspace stands in."""
    c = F.cfg(1, 8, 128)
    for cache, first_row in ((F.paged(c, 4, 2048, 16), 1), (F.contiguous(c, 4, n_tokens), 1), (F.paged(c, 4, 2048, 16, n_blocks=0), 0),
                             (F.paged(c, 4, 0, 16), 0), (F.contiguous(c, 4, 0), 0)):
        F.launches()
        assert F.select_cached(c, 4, 4, n_tokens, cache) == 0
        assert F.launches()[0][1][5] == first_row


def test_few_heads_take_longer_layer_groups():
    """A CTA's cos/sin cost as much for one KV head as for eight: with few heads
    a CTA walks more layers (rebind and capture), with eight as few as four and
    two."""
    for H, D, L, tokens, rebind, capture in ((1, 256, 21, 2916, 3, None), (2, 128, 23, 20000, 4, None), (8, 128, 36, 4000, 9, None),
                                             (1, 128, 18, 3410, None, 3), (2, 128, 12, 6048, None, 4), (8, 128, 12, 6048, None, 6)):
        c = F.cfg(L, H, D)
        F.launches()
        if rebind:
            assert F.revisit(c, 1, tokens) == 0 and F.launches()[1][1][1] == rebind, (H, D)
        else:
            assert F.capture(c, tokens) == 0 and F.launches()[0][1][1] == capture, (H, D)


def test_decode_chunks_of_few_long_sequences():
    """Two or three long sequences under four waves of teams take chunks of 1024
    slots, which even out their last wave; more sequences, more waves, or a
    group of more than 4 query heads 2048."""
    for L, H, seqs, group, n, want in ((36, 8, 2, 4, 4096, 1024), (36, 8, 3, 4, 3000, 1008), (11, 8, 3, 1, 8192, 1024), (36, 8, 2, 4, 8192, 2048),
                                       (36, 4, 6, 4, 4096, 2048), (28, 4, 3, 7, 8192, 2048), (36, 8, 16, 4, 4096, 2048)):
        F.launches()
        assert F.decode(F.cfg(L, H, 128), seqs, group, n, 1 << 40) == 0
        assert F.launches()[0][1][6:] == [want, 4], (L, H, seqs, group, n)


def test_decode_large_cases_reach_their_kernels():
    """The GPU test's shapes take the kernel, the team and the split they name."""
    from test_decode_gpu import LARGE
    for (B, layers, H, Hq, D, max_len, _), (team, splits) in LARGE:
        F.launches()
        assert F.decode(F.cfg(layers, H, D), B, Hq // H, max_len, 1 << 40) == 0
        kernel, *merge = F.launches()
        assert f"decode_kernelILi{D}ELb{int(team > 0)}E" in kernel[0]
        assert [kernel[1][5], kernel[1][7]] == [splits, team] and len(merge) == (splits > 1), (B, layers, H)
        if splits > 1:
            assert ("warp" in merge[0][0]) == (splits <= 32)


@pytest.mark.parametrize("D,ctas", [(64, 4), (128, 2), (256, 2)])
def test_cached_logits_fill_the_gpu_once(D, ctas):
    """A large cached selection's logits: one wave of four CTAs per SM at
    head_dim 64 (whose rows are half as long), of two above."""
    F.launches()
    assert F.select_cached(F.cfg(1, 4, D), 8, 4, 16384) == 0
    logits, tail = F.launches()
    assert "select_logits" in logits[0] and "select_tail" in tail[0]
    assert 0.9 * 152 * ctas < logits[1][0] <= 152 * ctas


def test_capture_of_wide_rows_keeps_two_ctas_per_sm():
    """A row of 512 threads takes the capture kernel of 64 registers a thread."""
    for H, D, wide in ((8, 128, False), (32, 128, False), (48, 128, False), (64, 128, True), (32, 256, True)):
        F.launches()
        assert F.capture(F.cfg(2, H, D), 900) == 0
        assert ("capture_kernelILi512E" in F.launches()[0][0]) == wide, (H, D)


def test_selection_takes_the_faster_path():
    """Points where one kernel and two were measured at least a tenth apart."""
    for cached, D, H, g, seqs, tokens, one in ((False, 128, 8, 4, 1, 768, True), (False, 128, 8, 4, 1, 4096, False), (False, 64, 8, 4, 1, 4096, False),
                                               (False, 64, 8, 4, 7, 1536, True), (False, 64, 8, 4, 40, 2048, False), (False, 256, 8, 4, 1, 1024, True),
                                               (True, 64, 8, 4, 40, 3072, False), (True, 64, 32, 3, 1, 214, True), (True, 64, 64, 1, 8, 311, True),
                                               (True, 128, 8, 4, 1, 1024, True), (True, 128, 8, 4, 16, 4096, False), (True, 128, 2, 4, 1, 8192, False),
                                               (True, 256, 8, 4, 7, 512, True), (True, 256, 8, 4, 16, 2048, False)):
        F.launches()
        assert (F.select_cached if cached else F.select_raw)(F.cfg(1, H, D), seqs, g, tokens) == 0
        assert ("select_fused" in F.launches()[0][0]) == one, (cached, D, H, g, seqs, tokens)
