"""Dequantize bit for bit against the oracle over every form its kernels take: head dims, widths, groups, key axes, rotation,
both 16-bit types; both sides in one launch and each side alone; ranges that start and end inside pages; tails and empty sequences."""
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


FORMS = [(d, kb, vb, g, axis, rot) for d in (64, 128) for kb, vb in ((2, 2), (4, 4), (8, 8), (4, 2)) for g in (32, 64, 128) if g <= d
         for axis, rot in ((0, False), (0, True), (1, False), (1, True))] + [(128, 16, 2, 128, 0, False), (128, 3, 8, 64, 0, False), (64, 6, 16, 32, 0, False)]


@pytest.mark.parametrize("dtype", ["fp16", "bf16"])
@pytest.mark.parametrize("d,kb,vb,g,axis,rot", FORMS)
def test_every_form(kvq, d, kb, vb, g, axis, rot, dtype):
    w = wl.LLAMA_8B.with_(n_kv_heads=2, n_q_heads=2, head_dim=d, kb=kb, vb=vb, gk=g, gv=g, k_axis=axis, dtype=dtype)
    B, T = 3, 300
    signs = None
    if rot:
        signs = np.where(np.random.default_rng(d + kb).random(d) < 0.5, -1, 1).astype(np.int8)
    k, v = wl.make_kv(w, tokens=T, batch=B)
    cfg, gc, oc = tl.build_both(kvq, w, k, v, [T], 384, signs)
    shape = (B, 2, 384, d)

    def same(lens, lo, hi, sides):
        """sides: which outputs the call is given"""
        gc.seq_len.copy_(torch.tensor(lens, dtype=torch.int32))
        oc.seq_len[:] = lens
        out = [torch.full(shape, 7.0, dtype=w.torch_dtype, device="cuda") if s else None for s in sides]
        kvq.kvq_dequantize(cfg, gc, out[0], out[1], lo, hi)
        ref = [tl.bits_of(torch.full(shape, 7.0, dtype=w.torch_dtype)).copy() for _ in range(2)]
        oc.dequantize(ref[0], ref[1], lo, hi)
        for got, want in zip(out, ref):
            if got is not None:
                assert np.array_equal(tl.bits_of(got), want)

    # shorter lengths leave the incomplete last block of channel-wise keys out of the tail: those only where a block ends
    lens = [300, 256, 0] if axis == 1 else [300, 131, 0]
    for lo, hi in ((0, 384), (77, 259)):
        same(lens, lo, hi, (True, True))
    for sides in ((True, False), (False, True)):
        same(lens, 0, 384, sides)


@pytest.mark.parametrize("axis,rot", [(0, False), (1, False), (0, True)])
def test_long_ranges_take_a_launch_per_side(kvq, axis, rot):
    """more than 148 x 8 pages and streams: the same bytes as page by page"""
    w = wl.LLAMA_8B.with_(k_axis=axis)
    B, T = 10, 16 * 128 - 5
    cfg = tl.gpu_config_for(kvq, w, B, 2048)
    signs = None
    if rot:
        signs = torch.ones(128, dtype=torch.int8)
        signs[::3] = -1
    gc = kvq.Cache(cfg, k_signs=signs)
    k, v = (t.cuda() for t in wl.make_kv(w, tokens=T, batch=B))
    kvq.kvq_quantize_append(cfg, gc, k, v)
    whole, paged = ([torch.zeros((B, 8, 2048, 128), dtype=w.torch_dtype, device="cuda") for _ in range(2)] for _ in range(2))
    kvq.kvq_dequantize(cfg, gc, whole[0], whole[1], 0, 2048)
    for t in range(0, 2048, 128):
        kvq.kvq_dequantize(cfg, gc, paged[0], paged[1], t, t + 128)
    assert torch.equal(whole[0], paged[0]) and torch.equal(whole[1], paged[1])
    assert whole[0][:, :, :T].abs().sum() > 0 and not whole[0][:, :, T:].any()
