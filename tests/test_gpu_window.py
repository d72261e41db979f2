"""Residual window of recent full-precision tokens for K and V (Sec. 4.1's 64-token residual buffer) through the
C-ABI: pages and window bytes bit for bit against the oracle under any chunking, dequantize bit for bit, decode
attention (one and several query rows, ragged and short sequences, rotated keys) within tolerance."""
import numpy as np
import pytest
import torch

from paper_2502_15075_b200 import workloads as wl

import kvq_testlib as tl
from test_gpu_rows import decode_rows, make_q_rows

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kvq():
    from paper_2502_15075_b200 import build
    build.build()
    from paper_2502_15075_b200 import kvq as mod
    return mod


W8 = wl.LLAMA_8B.with_(n_kv_heads=2, n_q_heads=8)


@pytest.mark.parametrize("name,w,R,T,chunks", [
    ("k4v2-r64-bulk", W8, 64, 64 * 5 + 37, [64 * 5 + 37]),
    ("k4v2-r64-steps", W8, 64, 200, [63, 1, 1, 70, 64, 1]),
    ("k4v2-r128", W8, 128, 128 * 2 + 100, [300, 56]),
    ("k8v4-r64", W8.with_(kb=8, vb=4), 64, 150, [150]),
    ("k3v6-r64", W8.with_(kb=3, vb=6), 64, 150, [100, 50]),
    ("1b-d64-r64", wl.LLAMA_1B.with_(n_kv_heads=2, n_q_heads=8), 64, 64 * 3 + 5, [64 * 3 + 5]),
    ("70b-g8-r64", wl.LLAMA_70B.with_(n_kv_heads=2, n_q_heads=16), 64, 300, [300]),
    ("k4v2-r64-exact-blocks", W8, 64, 256, [256]),
])
def test_window_parity(kvq, name, w, R, T, chunks):
    B = 2
    cap = ((T + 127) // 128) * 128 + 128
    k, v = wl.make_kv(w, tokens=T, batch=B)
    cfg, gc, oc = tl.build_both(kvq, w, k, v, chunks, cap, residual=R)
    assert kvq.kvq_check_status(gc) == 0
    tl.assert_caches_equal(gc, oc)
    ko = torch.zeros((B, w.n_kv_heads, cap, w.head_dim), dtype=w.torch_dtype, device="cuda")
    vo = torch.zeros_like(ko)
    kvq.kvq_dequantize(cfg, gc, ko, vo, 0, cap)
    kr = np.zeros((B, w.n_kv_heads, cap, w.head_dim), np.uint16)
    vr = np.zeros_like(kr)
    oc.dequantize(kr, vr, 0, cap)
    assert np.array_equal(tl.bits_of(ko), kr) and np.array_equal(tl.bits_of(vo), vr)
    assert np.array_equal(tl.bits_of(ko)[:, :, (T // R) * R:T], tl.bits_of(k)[:, :, (T // R) * R:T])   # the window is exact
    q = wl.make_q(w, batch=B)
    if name in ("k3v6-r64",):       # the plain-ALU kernel does not merge a window
        with pytest.raises(kvq.KvqError):
            tl.gpu_decode(kvq, cfg, gc, q)
        return
    want = tl.oracle_on_gpu_codes(gc, w).decode(tl.bits_of(q))
    tl.assert_attention_close(tl.gpu_decode(kvq, cfg, gc, q), want)


def test_window_with_rows_ragged_short_and_rotated(kvq):
    w, R, B, cap = W8, 64, 4, 512
    signs = np.where(np.random.default_rng(5).random(128) < 0.5, -1, 1).astype(np.int8)
    k, v = wl.make_kv(w, tokens=cap, batch=B)
    cfg, gc, oc = tl.build_both(kvq, w, k, v, [cap - 3], cap, k_signs=signs, residual=R)
    lens = [0, 2, 63, 64 * 6 + 9]                  # empty; shorter than the window; window only; pages + window
    # rebuild with ragged lengths: append per length through seq_len manipulation is not possible for a ring,
    # so build separate caches of batch 1 and compare each
    for n in lens:
        cfg1, g1, o1 = tl.build_both(kvq, w, k[:1, :, :n], v[:1, :, :n], [n] if n else [], cap, k_signs=signs, residual=R)
        tl.assert_caches_equal(g1, o1)
        q = make_q_rows(w, 1, 2, n)
        want = o1.decode_rows(tl.bits_of(q))
        got = decode_rows(kvq, cfg1, g1, q)
        tl.assert_attention_close(got, want)
        if n == 0:
            assert not got.any()


def test_window_improves_attention_accuracy(kvq):
    """The recent tokens carry no quantization error: against exact attention on the unquantized cache the error
    with a 64-token window is below the error without one."""
    w, T = W8, 64 * 4 + 40
    k, v = wl.make_kv(w, tokens=T, batch=2)
    q = wl.make_q(w, batch=2)
    logits = torch.einsum("bhd,bhtd->bht", q.double(), k.double().repeat_interleave(4, 1)) / np.sqrt(128)
    exact = torch.einsum("bht,bhtd->bhd", torch.softmax(logits, -1), v.double().repeat_interleave(4, 1)).numpy()
    errs = []
    for R in (0, 64):
        cfg, gc, _ = tl.build_both(kvq, w, k, v, [T], 512, residual=R)
        errs.append(np.linalg.norm(tl.gpu_decode(kvq, cfg, gc, q) - exact))
    assert errs[1] < errs[0]


@pytest.mark.parametrize("D,heads,rows", [(128, 1, 1), (128, 3, 1), (128, 2, 2), (128, 4, 2), (128, 7, 1), (128, 8, 1),
                                          (64, 1, 1), (64, 3, 1), (64, 2, 2)])      # (head_dim 64 serves four pairs)
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("R,T", [(64, 1), (64, 63), (64, 128 + 33), (128, 127), (128, 128 + 65)])
def test_window_tokens_only_and_with_pages(kvq, D, heads, rows, dtype, R, T):
    """Window lengths around the kernel's token passes, every number of (row, head) pairs, with and without pages."""
    g = 128 if D == 128 else 64
    w = wl.LLAMA_8B.with_(n_kv_heads=2, n_q_heads=2 * heads, head_dim=D, gk=g, gv=g, dtype=dtype)
    k, v = wl.make_kv(w, tokens=T, batch=2)
    cfg, gc, oc = tl.build_both(kvq, w, k, v, [T], 384, residual=R)
    q = make_q_rows(w, 2, rows, T)
    tl.assert_attention_close(decode_rows(kvq, cfg, gc, q), oc.decode_rows(tl.bits_of(q)))


@pytest.mark.parametrize("w,R,rows,lens", [
    (W8, 64, 1, [0, 40, 64 * 3 + 9, 128 * 20 + 70, 128 * 70 + 13, 128]),        # windows in gaps, with first pages, without pages, empty
    (W8, 64, 2, [2, 63, 65, 1000, 1001]),
    (W8.with_(kb=8, vb=4), 128, 1, [127, 300, 128 * 9 + 127]),                   # no gaps between the streams
    (wl.LLAMA_70B.with_(n_kv_heads=2, n_q_heads=16), 128, 1, [50, 128 * 3 + 127, 128 * 40 + 1]),
    (wl.LLAMA_1B.with_(n_kv_heads=2, n_q_heads=8), 128, 1, [50, 128 * 3 + 127, 128 * 40 + 1]),
    (W8, 64, 1, [64 * (i % 9) + 7 * i % 64 for i in range(90)]),                  # many short streams
    (wl.LLAMA_8B.with_(n_kv_heads=1, n_q_heads=4), 128, 1, [128 * 60 + 99]),      # one stream over many shares
])
def test_windows_of_uneven_batches(kvq, w, R, rows, lens):
    """Whoever takes a stream's window - a share inside the gap in front of it, the share with its first page, or a stream without
    pages - and whatever the other streams do: each sequence gives what it gives alone, checked against the oracle."""
    T, cap = max(lens), -(-max(lens) // 128) * 128
    cfg = tl.gpu_config_for(kvq, w, len(lens), cap, R)
    gc = kvq.Cache(cfg)
    cfg1 = tl.gpu_config_for(kvq, w, 1, cap, R)
    k, v = wl.make_kv(w, tokens=T, batch=1, device="cuda")
    pages, win = gc.pages_view(), gc.window_view()
    win.fill_(-1)                                  # rows that hold no token are NaN
    for b, n in enumerate(lens):
        one = kvq.Cache(cfg1)
        one.window_view().fill_(-1)
        if n:
            kvq.kvq_quantize_append(cfg1, one, k[:, :, T - n:], v[:, :, T - n:])
        pages[b], win[b] = one.pages_view()[0], one.window_view()[0]
    gc.seq_len.copy_(torch.tensor(lens, dtype=torch.int32))
    q = make_q_rows(w, len(lens), rows, 3)
    got = decode_rows(kvq, cfg, gc, q)
    assert np.array_equal(got, decode_rows(kvq, cfg, gc, q))
    check = range(len(lens)) if len(lens) < 10 else range(0, len(lens), 7)
    for b in check:
        sub = kvq.Cache(cfg1)
        sub.pages_view()[0], sub.window_view()[0] = pages[b], win[b]
        sub.seq_len.fill_(lens[b])
        oc = tl.oracle_on_gpu_codes(sub, w)
        tl.assert_attention_close(got[b:b + 1], oc.decode_rows(tl.bits_of(q[b:b + 1])))


@pytest.mark.parametrize("kb,vb", [(4, 4), (4, 2), (8, 4)])
def test_windows_longer_than_the_ring(kvq, kb, vb):
    """Windows around what fits a CTA's ring of pages (96 tokens), taken by shares inside the gaps of a short batch (none at K8V4)."""
    lens = [128 * 3 + 96, 97, 128 * 20 + 102, 128 * 9 + 111, 128 * 2 + 103, 128 + 104, 128 * 5 + 112, 128 * 4 + 95]
    test_windows_of_uneven_batches(kvq, W8.with_(kb=kb, vb=vb), 128, 1, lens)


def test_a_window_that_never_arrives_sets_the_status(kvq):
    """The copy of a window taken by a share inside a gap: its wait runs out, the call returns (after it has waited once more for what may
    be on its way), the status says so, and the next call on the same cache and workspace gives the bytes it gave before."""
    B, T, R = 3, 64 * 5 + 37, 64
    cfg = tl.gpu_config_for(kvq, W8, B, 384, R)
    gc = kvq.Cache(cfg)
    kvq.kvq_quantize_append(cfg, gc, *wl.make_kv(W8, 0, "cuda", tokens=T, batch=B))
    q = wl.make_q(W8, batch=B).cuda()
    ws = torch.empty(kvq.kvq_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    good, out = (torch.zeros(tuple(q.shape), dtype=torch.float32, device="cuda") for _ in range(2))
    kvq.kvq_decode_attention(cfg, gc, q, good, ws)
    assert kvq.kvq_check_status(gc) == 0
    for stream in range(B * W8.n_kv_heads):
        kvq.kvq_debug_decode_stall(cfg, gc, q, out, ws, -2 - 3 * stream, 2000)        # (three pages a stream)
        assert kvq.kvq_check_status(gc) == -7                   # KVQ_ERR_DEVICE_TIMEOUT
        gc.status.zero_()
        out.fill_(7.0)
        kvq.kvq_decode_attention(cfg, gc, q, out, ws)
        assert kvq.kvq_check_status(gc) == 0 and torch.equal(out, good)
    kvq.kvq_debug_decode_stall(cfg, gc, q, out, ws, -2 - 1, 50000)                  # no stream starts with page 1
    assert kvq.kvq_check_status(gc) == 0 and torch.equal(out, good)
