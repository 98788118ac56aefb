"""The library's host side on a CPU: its objects linked against a CUDA runtime
that keeps the launches instead of running them (fake_cudart.cpp, 152 SMs)."""
import ctypes as C
import functools
import os
import subprocess
import tempfile

from paper_2606_26631_gb300 import _binding as B
from paper_2606_26631_gb300 import _build

FAKE = 1 << 40  # a device address, never dereferenced
WORK = FAKE + (1 << 30)  # a selection's workspace


@functools.lru_cache(None)
def lib():
    _build.build()
    objs = [os.path.join(_build.BUILD, s.replace(".cu", ".o")) for s in _build.SOURCES]
    if not all(os.path.exists(o) for o in objs):
        _build.build(force=True)
    out = os.path.join(tempfile.mkdtemp(), "libprcr_fake.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(_build.nvcc())), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-fvisibility=hidden", "-Wl,-Bsymbolic", "-I", cuda, "-I", _build.INCLUDE,
                    "-I", _build.CSRC, os.path.join(os.path.dirname(__file__), "fake_cudart.cpp"), *objs, "-o", out], check=True)
    L, real = C.CDLL(out), B.lib()
    for name in B.EXPORTS:
        f, r = getattr(L, name), getattr(real, name)
        f.argtypes, f.restype = r.argtypes, r.restype
    return L


def launches():
    """[(kernel's mangled name, numbers)] since the last call."""
    buf = C.create_string_buffer(1 << 20)
    lib().fake_log(buf, C.c_size_t(len(buf)))
    return [(w[0], [int(x) for x in w[1:]]) for w in (line.split() for line in buf.value.decode().splitlines())]


def cfg(layers, H, D):
    return B.rope_cfg(layers, H, D, (D // 2, 0, 0))


def contiguous(c, seqs, slots):
    row = c.n_kv_heads * c.head_dim
    return B.CacheDesc(kind=0, block_size=1, k=FAKE, v=FAKE, seq_stride=c.n_layers * slots * row, layer_stride=slots * row, block_stride=0,
                       slot_stride=row, block_table=None, bt_stride=0, n_blocks=0, max_slots=min(slots, 2 ** 31 - 1), n_seqs=seqs)


def workspace(c, seqs, group, max_len):
    return lib().prcr_decode_workspace_size(C.byref(c), seqs, c.n_kv_heads * group, max_len)


def decode(c, seqs, group, max_len, ws_bytes, cache=None):
    cache = cache or contiguous(c, seqs, max_len)
    return lib().prcr_decode_attention(C.byref(c), C.byref(cache), seqs, c.n_kv_heads * group, FAKE, FAKE, FAKE, max_len, FAKE, FAKE, FAKE,
                                       ws_bytes, None)


def select_cached(c, seqs, group, n_tokens, cache=None):
    cache = cache or contiguous(c, seqs, n_tokens)
    Hq = c.n_kv_heads * group
    return lib().prcr_select_topk_cached(C.byref(c), C.byref(cache), seqs, 0, Hq, n_tokens, FAKE, FAKE, FAKE, 1, FAKE, FAKE, FAKE, None, FAKE,
                                         WORK, lib().prcr_select_workspace_size(seqs, Hq, n_tokens), None)


def store(c, seqs, n_tokens):
    row = c.n_kv_heads * c.head_dim
    return B.StoreDesc(k=FAKE, v=FAKE, coords=FAKE, seq_stride=c.n_layers * n_tokens * row, layer_stride=n_tokens * row, token_stride=row,
                       coord_seq_stride=3 * n_tokens, n_seqs=seqs, n_tokens=n_tokens)


def select_raw(c, seqs, group, n_tokens):
    s = store(c, seqs, n_tokens)
    Hq = c.n_kv_heads * group
    return lib().prcr_select_topk(C.byref(c), C.byref(s), seqs, 0, Hq, FAKE, FAKE, 1, FAKE, FAKE, FAKE, None, FAKE,
                                  lib().prcr_select_workspace_size(seqs, Hq, n_tokens), None)


def revisit(c, seqs, tokens, entry="inject"):
    """A batch of one revisit of `tokens` per sequence: prcr_rebind_inject, prcr_plan or prcr_rebind_apply."""
    total = seqs * tokens
    st, ca = store(c, seqs, tokens), contiguous(c, seqs, 2 * tokens)
    b = B.RevisitBatch(seq_rev_off=FAKE, rev_tok_off=FAKE, idx=FAKE, p_txt=FAKE, cache_len_in=FAKE, n_seqs=seqs, n_revisits=seqs,
                       total_k=total)
    o = B.Outputs(cache_len_out=FAKE + 4096, next_pos_out=FAKE, pos_out=None, slot_out=None, status=FAKE)
    f = {"inject": lib().prcr_rebind_inject, "plan": lib().prcr_plan, "apply": lib().prcr_rebind_apply}[entry]
    return f(C.byref(c), C.byref(st), C.byref(ca), C.byref(b), C.byref(o), 0, 2, 0, FAKE, lib().prcr_workspace_size(total), None)


def paged(c, seqs, blocks_per_seq, block, n_blocks=1024):
    row = c.n_kv_heads * c.head_dim
    return B.CacheDesc(kind=1, block_size=block, k=FAKE, v=FAKE, seq_stride=0, layer_stride=1024 * block * row, block_stride=block * row,
                       slot_stride=row, block_table=FAKE, bt_stride=blocks_per_seq, n_blocks=n_blocks, max_slots=0, n_seqs=seqs)


def capture(c, tokens):
    st, ca = store(c, 1, tokens), contiguous(c, 1, tokens)
    row = c.n_kv_heads * c.head_dim
    return lib().prcr_prefill_capture(C.byref(c), C.byref(st), C.byref(ca), 0, 0, c.n_layers, 0, tokens, 0, FAKE, FAKE, tokens * row, row,
                                      FAKE, FAKE, None)
