"""Quantize-append against the oracle, byte for byte, at the sizes where its kernels change over: single tokens, ends of
blocks, completed and incomplete blocks, both input types, all widths, rotated and plain keys, strided inputs, values at
the ends of the 16-bit ranges."""
import numpy as np
import pytest
import torch

from paper_2502_15075_b200 import workloads as wl

import kvq_testlib as tl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kvq():
    from paper_2502_15075_b200 import build
    build.build()
    from paper_2502_15075_b200 import kvq as mod
    return mod


def edge_values(w, T, B, seed, rotated=False):
    """Keys and values with constant groups, signed zeros, subnormal ranges and entries at the ends of the 16-bit type."""
    k, v = wl.make_kv(w.with_(number=seed), tokens=T, batch=B)
    big = 65504.0 if w.dtype == "fp16" else 1.0e30 if rotated else 3.0e38      # (a rotation sums 128 of them: finite)
    for x in (k, v):
        x[:, :, 0] = 0.25                                   # a constant row
        if T > 3:
            x[:, :, 1] = -0.0
            x[:, :, 2] *= 2.0 ** -14                         # scales in the fp16 subnormals, some of them zero
            x[:, 0, 3, :2] = torch.tensor([big, -big])
        if T > 5:
            x[:, 0, 5] = 100.0 + x[:, 0, 5] * 2.0 ** -6      # the rounding of the minimum exceeds the step: codes clamp
    return k, v


def check(kvq, w, B, chunks, signs=None, residual=0, strided=False, seed=1):
    T = sum(chunks)
    cap = -(-T // 128) * 128 + 128
    k, v = edge_values(w, T, B, seed, signs is not None)
    if strided:                                              # [B, T, H, D] in memory, as a projection leaves it
        k, v = (x.transpose(1, 2).contiguous().transpose(1, 2) for x in (k, v))
    cfg, gc, oc = tl.build_both(kvq, w, k, v, chunks, cap, k_signs=signs, residual=residual)
    assert kvq.kvq_check_status(gc) == 0
    tl.assert_caches_equal(gc, oc)


CHUNKS = {"steps": [126, 1, 1, 1], "block": [128], "over": [129, 127, 3], "ragged": [5, 250, 1, 140]}
SIGNS = np.random.default_rng(3).choice([-1, 1], 128).astype(np.int8)


@pytest.mark.parametrize("chunks", list(CHUNKS))
@pytest.mark.parametrize("kb", [2, 4, 8])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("rotated", [False, True])
def test_channelwise_keys(kvq, chunks, kb, dtype, rotated):
    w = wl.SHAPED_14B.with_(n_kv_heads=3, n_q_heads=3, kb=kb, dtype=dtype)
    check(kvq, w, 2, CHUNKS[chunks], SIGNS if rotated else None, strided=chunks == "over")


FEW = [1, 1, 2, 5, 16, 17, 103, 1, 15]          # single tokens and short runs around the page's 16-, 32- and 128-token marks


@pytest.mark.parametrize("kb,vb", [(2, 8), (4, 2), (8, 4)])
@pytest.mark.parametrize("D,gk,gv", [(128, 128, 32), (128, 32, 64), (64, 64, 32), (64, 32, 64)])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("form", ["plain", "rotated", "window", "rotated window"])
def test_few_tokens(kvq, kb, vb, D, gk, gv, dtype, form):
    heads = 9 if D == 64 else 3                  # more and fewer heads than CTAs of a cluster
    w = wl.LLAMA_8B.with_(n_kv_heads=heads, n_q_heads=heads, head_dim=D, kb=kb, vb=vb, gk=gk, gv=gv, dtype=dtype)
    check(kvq, w, 2, FEW, SIGNS[:D] if "rotated" in form else None, 64 if "window" in form else 0, strided=D == 64)


def test_few_tokens_beyond_the_capacity(kvq):
    """A sequence without room keeps its bytes and its length and sets the status; the others take their tokens."""
    w = wl.LLAMA_8B.with_(n_kv_heads=2, n_q_heads=2)
    k, v = edge_values(w, 128, 2, 1)
    cfg, gc, _ = tl.build_both(kvq, w, k, v, [128], 256)
    gc.seq_len.copy_(torch.tensor([255, 128], dtype=torch.int32))
    before = gc.pages_view()[0].clone()
    kvq.kvq_quantize_append(cfg, gc, k[:, :, :2].cuda(), v[:, :, :2].cuda())
    assert gc.seq_len.tolist() == [255, 130] and torch.equal(gc.pages_view()[0], before)
    assert kvq.kvq_check_status(gc) == -5


RUNS = {"odd": [131, 70, 259], "exact": [256, 160], "inside": [200, 65, 66]}       # whole, partial and interior 32-token tasks


@pytest.mark.parametrize("kb,vb", [(2, 8), (4, 2), (8, 4)])
@pytest.mark.parametrize("D,gk,gv", [(128, 128, 32), (128, 32, 128), (128, 64, 64), (64, 64, 32), (64, 32, 64)])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("runs,form", [("odd", "plain"), ("exact", "plain"), ("odd", "rotated"), ("inside", "rotated window")])
def test_runs_of_tokens(kvq, kb, vb, D, gk, gv, dtype, runs, form):
    w = wl.LLAMA_8B.with_(n_kv_heads=2, n_q_heads=2, head_dim=D, kb=kb, vb=vb, gk=gk, gv=gv, dtype=dtype)
    check(kvq, w, 2, RUNS[runs], SIGNS[:D] if "rotated" in form else None, 64 if "window" in form else 0, strided=runs == "odd")


@pytest.mark.parametrize("kb", [2, 4, 8])
@pytest.mark.parametrize("rotated", [False, True])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
def test_a_nan_row_gives_the_same_bytes_at_once_and_in_pieces(kvq, kb, rotated, dtype):
    """Non-finite inputs are outside of what the quantizer defines, but the bytes must not depend on how many tokens a call has."""
    w = wl.LLAMA_8B.with_(n_kv_heads=2, n_q_heads=2, kb=kb, dtype=dtype)
    k, v = wl.make_kv(w, tokens=140, batch=1)
    for t in (3, 70, 139):
        k[:, :, t, 17] = float("nan")
    k[:, 0, 40] = v[:, 1, 41] = float("nan")
    pages = []
    for chunks in ([140], [64, 12, 64]):
        cfg = tl.gpu_config_for(kvq, w, 1, 256)
        gc = kvq.Cache(cfg, k_signs=torch.from_numpy(SIGNS) if rotated else None)
        for part in torch.split(torch.arange(140), chunks):
            kvq.kvq_quantize_append(cfg, gc, k[:, :, part].cuda(), v[:, :, part].cuda())
        pages.append(gc.pages.cpu())
    assert torch.equal(*pages)


# appends of at most 64 tokens that complete a block and leave tokens behind it, or end with it
BLOCKS = {"behind": [120, 20, 64, 60], "behind and ahead": [100, 64, 1, 64], "exact": [64, 64, 1, 63, 64]}


@pytest.mark.parametrize("chunks", list(BLOCKS))
@pytest.mark.parametrize("heads", [9, 10])              # two heads for some or all CTAs of a cluster: the scratch is used again
@pytest.mark.parametrize("kb", [4, 8])
@pytest.mark.parametrize("rotated", [False, True])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
def test_short_appends_of_channelwise_keys_over_blocks(kvq, chunks, heads, kb, rotated, dtype):
    w = wl.SHAPED_14B.with_(n_kv_heads=heads, n_q_heads=heads, kb=kb, dtype=dtype)
    check(kvq, w, 2, BLOCKS[chunks], SIGNS if rotated else None, strided=chunks == "exact")


@pytest.mark.parametrize("D,heads,n", [(128, 1, 64), (64, 8, 128), (128, 16, 32), (64, 16, 64), (128, 24, 21)])
@pytest.mark.parametrize("form", ["plain", "rotated", "window"])
def test_both_sides_of_the_short_append(kvq, D, heads, n, form):
    """The largest append that takes one launch and the one beyond it, for few and many heads."""
    if form != "plain" and heads > 8:
        n = n * 40 // 64
    w = wl.LLAMA_8B.with_(n_kv_heads=heads, n_q_heads=heads, head_dim=D, gk=64, gv=64)
    check(kvq, w, 1, [13, n, n + 1, 3, n, n + 1], SIGNS[:D] if form == "rotated" else None, 64 if form == "window" else 0)


@pytest.mark.parametrize("heads,n", [(8, 64), (10, 52), (17, 30)])
def test_both_sides_of_the_short_append_of_channelwise_keys(kvq, heads, n):
    w = wl.SHAPED_14B.with_(n_kv_heads=heads, n_q_heads=heads)
    check(kvq, w, 1, [13, n, n + 1, 3, n, n + 1])


@pytest.mark.parametrize("shape,kb", [("channel", 4), ("channel", 8), ("token", 4)])
@pytest.mark.parametrize("n", [1, 20, 64, 90])
def test_append_to_sequences_of_different_lengths(kvq, shape, kb, n):
    """One sequence completes a block and leaves tokens behind it, one ends with the block, one stays inside it."""
    w = (wl.SHAPED_14B if shape == "channel" else wl.LLAMA_8B).with_(n_kv_heads=9, n_q_heads=9, kb=kb)
    k, v = edge_values(w, 120 + n, 3, 5)
    cfg, gc, oc = tl.build_both(kvq, w, k[:, :, :120], v[:, :, :120], [120], 256)
    lens = [120, 128 - n, 3]
    gc.seq_len.copy_(torch.tensor(lens, dtype=torch.int32))
    oc.seq_len[:] = lens
    kvq.kvq_quantize_append(cfg, gc, k[:, :, 120:].cuda(), v[:, :, 120:].cuda())
    oc.append(tl.bits_of(k)[:, :, 120:], tl.bits_of(v)[:, :, 120:])
    assert kvq.kvq_check_status(gc) == 0
    tl.assert_caches_equal(gc, oc)


@pytest.mark.parametrize("axis,kb,vb", [("token", 4, 2), ("token", 2, 8), ("token", 8, 4), ("channel", 4, 2), ("channel", 8, 4)])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
def test_values_below_the_normal_fp16_numbers(kvq, axis, kb, vb, dtype):
    """Magnitudes from 2^-26 to 2^3 side by side (a bf16 key of a channel-wise block is rounded to fp16 in the sum), groups that
    need no clamp next to groups that do: one block of three, and single rows, reach the ends of the 16-bit type."""
    w = (wl.SHAPED_14B if axis == "channel" else wl.LLAMA_8B).with_(n_kv_heads=2, n_q_heads=2, kb=kb, vb=vb, dtype=dtype)
    T, B = 405, 2
    g = torch.Generator().manual_seed(7)
    k, v = wl.make_kv(w, tokens=T, batch=B)
    for x in (k, v):
        x *= torch.exp2(torch.randint(-24, 2, x.shape, generator=g).to(torch.float32)).to(x.dtype)
        x[:, :, 50:60] = (x[:, :, 50:60].float() * 2.0 ** -10).to(x.dtype)
        for t in (140, 141, 200):
            x[:, 0, t, 3:5] = torch.tensor([65504.0, -65504.0]).to(x.dtype)
    cfg, gc, oc = tl.build_both(kvq, w, k, v, [3, 402], 512)
    assert kvq.kvq_check_status(gc) == 0
    tl.assert_caches_equal(gc, oc)
    _, gc, oc = tl.build_both(kvq, w, k, v, [405], 512)
    tl.assert_caches_equal(gc, oc)


@pytest.mark.parametrize("axis,kb,vb,D", [("token", 4, 2, 128), ("token", 2, 8, 128), ("token", 8, 4, 64), ("channel", 4, 2, 128), ("channel", 8, 4, 128)])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
def test_a_long_append_gives_the_bytes_of_its_pieces(kvq, axis, kb, vb, D, dtype):
    """60 streams x 5,989 tokens: several passes or blocks per warp or CTA, the next one's loads in flight; pieces have one each."""
    w = (wl.SHAPED_14B if axis == "channel" else wl.LLAMA_8B).with_(n_kv_heads=20, n_q_heads=20, kb=kb, vb=vb, dtype=dtype, head_dim=D, gk=64, gv=64)
    if axis == "channel":
        w = w.with_(gk=128)
    T, B = 5989, 3
    k, v = wl.make_kv(w, tokens=T, batch=B, device="cuda")
    for t in (40, 1000, 2500, 2501, 5980):
        k[:, t % 20, t, 3] = v[:, t % 20, t, 5] = 60000.0
    pages = []
    for piece in (T, 640):
        cfg = tl.gpu_config_for(kvq, w, B, 6144)
        gc = kvq.Cache(cfg)
        for t in range(0, T, piece):
            kvq.kvq_quantize_append(cfg, gc, k[:, :, t:t + piece], v[:, :, t:t + piece])
        assert kvq.kvq_check_status(gc) == 0 and gc.seq_len.tolist() == [T] * B
        pages.append((gc.pages.cpu(), gc.tail_view()[:, :, :T % 128].cpu() if axis == "channel" else None))
    assert torch.equal(pages[0][0], pages[1][0])
    assert axis == "token" or torch.equal(pages[0][1], pages[1][1])


@pytest.mark.parametrize("B,D,heads,n", [(8, 128, 8, 64), (9, 128, 8, 64), (12, 64, 8, 128), (13, 128, 8, 32), (13, 64, 8, 64), (14, 128, 16, 16)])
@pytest.mark.parametrize("form", ["plain", "rotated"])
def test_the_short_append_of_several_sequences(kvq, B, D, heads, n, form):
    """More threads per CTA up to eight sequences, fewer tokens beyond twelve: the largest append of one launch and the one beyond it."""
    if form == "rotated" and heads > 8:
        n = min(n, 20)
    w = wl.LLAMA_8B.with_(n_kv_heads=heads, n_q_heads=heads, head_dim=D, gk=64, gv=64)
    check(kvq, w, B, [13, n, n + 1], SIGNS[:D] if form == "rotated" else None)


@pytest.mark.parametrize("heads,n", [(8, 64), (10, 36), (17, 20)])
def test_the_short_append_of_channelwise_keys_and_the_one_beyond(kvq, heads, n):
    w = wl.SHAPED_14B.with_(n_kv_heads=heads, n_q_heads=heads)
    check(kvq, w, 2, [13, n, n + 1, 3, n, n + 1])


@pytest.mark.parametrize("D,gk", [(128, 32), (128, 64), (128, 128), (64, 32), (64, 64)])
@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
def test_keys_at_two_bits_of_long_appends(kvq, D, gk, dtype):
    """Two tokens of a lane per pass: parts of tasks and whole ones, groups of two and four lanes and two groups a lane, and groups that clamp."""
    w = wl.LLAMA_8B.with_(n_kv_heads=3, n_q_heads=3, head_dim=D, kb=2, vb=4, gk=gk, gv=D, dtype=dtype)
    k, v = wl.make_kv(w, tokens=613, batch=2)
    k[:, 1, 300:330, 5:7] = torch.tensor([60000.0, -60000.0]).to(k.dtype)
    k[:, 2, 100:140] *= 2.0 ** -18
    _, gc, oc = tl.build_both(kvq, w, k, v, [129, 1, 483], 640)
    assert kvq.kvq_check_status(gc) == 0
    tl.assert_caches_equal(gc, oc)


@pytest.mark.parametrize("B,D,heads,n,form", [
    (15, 128, 8, 64, "plain"), (16, 128, 8, 40, "plain"), (15, 64, 8, 128, "plain"), (16, 64, 8, 80, "plain"), (16, 128, 16, 20, "plain"),
    (15, 128, 8, 64, "rotated"), (16, 128, 8, 40, "rotated"), (61, 128, 2, 40, "plain"), (60, 128, 2, 64, "plain")])
def test_the_short_append_where_clusters_begin_to_share_sms(kvq, B, D, heads, n, form):
    """The largest append of one launch and the one beyond it, on both sides of 120 CTAs."""
    w = wl.LLAMA_8B.with_(n_kv_heads=heads, n_q_heads=heads, head_dim=D, gk=64, gv=64)
    check(kvq, w, B, [13, n, n + 1], SIGNS[:D] if form == "rotated" else None)


@pytest.mark.parametrize("B,heads,n", [(16, 8, 64), (3, 8, 64), (4, 16, 32)])
def test_the_short_append_with_a_window(kvq, B, heads, n):
    """Up to 64 rows a CTA with a window, however many sequences; the longest of one launch completes a block."""
    w = wl.LLAMA_8B.with_(n_kv_heads=heads, n_q_heads=heads)
    k, v = wl.make_kv(w, tokens=13 + 2 * n + 1, batch=B)
    _, gc, oc = tl.build_both(kvq, w, k, v, [13, n, n + 1], 384, residual=64)
    assert kvq.kvq_check_status(gc) == 0
    tl.assert_caches_equal(gc, oc)
