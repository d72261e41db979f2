"""Decode attention where the fast kernel's pages and blocks end: lengths around a 32-token block and a 128-token page, keys and
values that keep growing (the common reference and the scale limit move on every page), every number of heads it
serves, against the fp64 oracle on the same codes."""
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


FORMS = {
    "k4v2": wl.LLAMA_8B, "k2v4": wl.LLAMA_8B.with_(kb=2, vb=4), "k8v4": wl.LLAMA_8B.with_(kb=8, vb=4),
    "k4v4": wl.LLAMA_8B.with_(vb=4), "k4v2-g32": wl.LLAMA_8B.with_(gk=32), "k4v2-g64": wl.LLAMA_8B.with_(gk=64, gv=64),
    "d64": wl.LLAMA_1B, "d64-g32": wl.TINY, "channel-k4v2": wl.SHAPED_14B, "channel-k8v2": wl.SHAPED_14B.with_(kb=8),
}


@pytest.mark.parametrize("T", [1, 31, 33, 96, 127, 128, 129, 500])
@pytest.mark.parametrize("form,heads", [(f, h) for f in FORMS for h in (1, 4)] + [("k4v2", 8), ("k4v2-g32", 5), ("k4v2-g64", 8)])
def test_growing_logits_and_values(kvq, form, heads, T):
    w = FORMS[form].with_(n_kv_heads=2, n_q_heads=2 * heads)
    k, v = wl.make_kv(w, tokens=T, batch=2)
    ramp = torch.linspace(0.05, 4.0, T).view(1, 1, T, 1)             # later tokens: larger logits, larger value scales
    k, v = (x.float().mul(ramp).to(w.torch_dtype) for x in (k, v))
    cfg, gc, _ = tl.build_both(kvq, w, k, v, [T], 512)
    oc = tl.oracle_on_gpu_codes(gc, w)
    # The absolute bound is for values of unit size: an error d of the logits moves an output by up to 2 d max|v|, and d comes
    # from q in 16-bit fixed point, half a unit of max|q| / 32512 per channel whatever the values are.
    scale = max(1.0, float(v.float().abs().max()))
    for variant in ("normal", "peaked"):
        q = wl.make_q(w, batch=2, variant=variant, k=k)
        tl.assert_attention_close(tl.gpu_decode(kvq, cfg, gc, q), oc.decode(tl.bits_of(q)), mabs=tl.MAX_ABS_TOL * scale)


@pytest.mark.parametrize("form,pages", [("channel-k4v2", [95, 63, 37, 57, 58, 70, 35, 110, 117, 93]), ("k4v2", [472, 1024])])
def test_every_row_of_an_uneven_batch_is_written(kvq, form, pages):
    """Full grids over uneven lengths, where a long stream's partials come close to its slots: against the plain kernel."""
    w = FORMS[form].with_(n_q_heads=FORMS[form].n_kv_heads)
    T, B = 128 * max(pages), len(pages)
    cfg = tl.gpu_config_for(kvq, w, B, T)
    gc = kvq.Cache(cfg)
    kvq.kvq_quantize_append(cfg, gc, *wl.make_kv(w, 0, "cuda", tokens=T, batch=B))
    gc.seq_len.copy_(torch.tensor(pages, dtype=torch.int32) * 128)
    q = wl.make_q(w, batch=B)
    got = tl.gpu_decode(kvq, cfg, gc, q)
    ws = torch.empty(kvq.kvq_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    want = torch.empty(tuple(q.shape), dtype=torch.float32, device="cuda")
    kvq.kvq_debug_decode_generic(cfg, gc, q.cuda(), want, ws)
    tl.assert_attention_close(got, want.double().cpu().numpy())


@pytest.mark.parametrize("form,heads", [("k4v2", 1), ("k4v4", 4), ("k4v2-g64", 1), ("k4v2", 8), ("channel-k4v2", 1)])
def test_streams_of_very_different_values_share_a_cta(kvq, form, heads):
    """More streams than CTAs, neighbours' values a factor of 2^24 apart: a stream's weights are fixed point below the largest
    value scale of that stream, not of the one its CTA served before it."""
    H, B, T = 8, 75, 200
    w = FORMS[form].with_(n_kv_heads=H, n_q_heads=H * heads)
    k, v = wl.make_kv(w, tokens=T, batch=B)
    v = (v.float() * torch.where(torch.arange(B * H) % 2 == 0, 2.0 ** 12, 2.0 ** -12).view(B, H, 1, 1)).to(w.torch_dtype)
    cfg = tl.gpu_config_for(kvq, w, B, 256)
    gc = kvq.Cache(cfg)
    kvq.kvq_quantize_append(cfg, gc, k.cuda(), v.cuda())
    q = wl.make_q(w, batch=B)
    got = tl.gpu_decode(kvq, cfg, gc, q).reshape(B * H, -1)
    want = tl.oracle_on_gpu_codes(gc, w).decode(tl.bits_of(q)).reshape(B * H, -1)
    err = np.linalg.norm(got - want, axis=1) / np.linalg.norm(want, axis=1)
    assert err.max() <= tl.REL_L2_TOL, f"stream {err.argmax()}: rel-L2 {err.max():.2e}"


@pytest.mark.parametrize("form", ["k4v2", "k4v4", "k2v4", "k8v4", "k4v2-g64", "d64", "channel-k4v2"])
@pytest.mark.parametrize("T", [32, 256, 1536])
def test_neighbouring_tokens_cancel_exactly(kvq, form, T):
    """Equal weights, values 2^27 apart that cancel between tokens t and t + 8: a lane adds the two before it goes on to the next
    tile, so what is left is exact.  (Values are constant over a row: codes and scales are 0, a token adds weight x zero-point.)"""
    w = FORMS[form].with_(n_kv_heads=2, n_q_heads=8)
    big, small = 2.0 ** 15, 2.0 ** -12
    t = torch.arange(T) % 32
    row = torch.where(t < 8, big, torch.where(t < 16, -big, small))
    k, v = wl.make_kv(w, tokens=T, batch=2)
    v = row.view(1, 1, T, 1).expand(v.shape).to(w.torch_dtype).contiguous()
    cfg, gc, _ = tl.build_both(kvq, w, k, v, [T], 1536)
    got = tl.gpu_decode(kvq, cfg, gc, torch.zeros((2, 8, w.head_dim), dtype=w.torch_dtype))      # every logit is 0
    assert np.array_equal(got, np.full(got.shape, small / 2))


def test_value_sums_over_more_pages_than_an_integer_accumulator_holds(kvq):
    """Over 350 pages per CTA of equal weights and largest codes: without the fold every 128 pages the 32-bit sums would overflow
    (the second weight byte is 254, the upper code field 192: 344 pages of 128 tokens).  All values of a head are equal, so the
    output is that value whatever the weights; the folds also fall at different distances behind a change of stream."""
    H, P = 8, 22000
    cfg = kvq.make_config(1, H, H, 64, 4, 2, 64, 64, 0, "fp16", 128 * P)
    starts = kvq.kvq_debug_decode_plan(cfg, [128 * P])[2]
    assert np.diff(starts).min() > 344
    gc = kvq.Cache(cfg)
    pages = gc.pages_view()                                  # key codes and metadata stay zero: every logit is 0
    k_bytes, v_codes = 128 * 64 // 2 + 128 * 4, 128 * 64 // 4
    pages[..., k_bytes:k_bytes + v_codes] = 0xFF             # code 3 everywhere
    scales = [0x3FFF, 0x3BFF, 0x3FFF, 0x33FF, 0x3FFF, 0x3FFF, 0x2FFF, 0x3FFF]     # 1.999 and smaller ones, mantissas all ones
    for h, s in enumerate(scales):
        meta = pages[0, h, :, k_bytes + v_codes:].view(P, 128, 4)
        meta[..., 0], meta[..., 1] = s & 255, s >> 8         # (zero-points stay 0)
    gc.seq_len.fill_(128 * P)
    got = tl.gpu_decode(kvq, cfg, gc, torch.ones((1, H, 64), dtype=torch.float16))[0]
    want = 3.0 * torch.tensor(scales, dtype=torch.int16).view(torch.float16).double().numpy()
    assert np.allclose(got, want[:, None], rtol=1e-5, atol=0.0)


def test_the_splits_division_on_the_device(kvq):
    """Exact for every quotient below 2^31, whatever the estimate that it starts from: small and large divisors, multiples and their
    neighbours (the host's copy of the split divides the same way from another estimate)."""
    g = torch.Generator().manual_seed(3)
    d = torch.cat([torch.arange(1, 200), 2 ** torch.arange(0, 44), 2 ** torch.arange(1, 44) - 1,
                   (torch.rand(20000, generator=g, dtype=torch.float64) * 43).exp2().long(), torch.tensor([148 * 1040 * 3, 148 * 1000 * 3 * 2 ** 20])])
    q = torch.cat([torch.arange(0, 200), (torch.rand(d.numel() - 200, generator=g, dtype=torch.float64) * 31).exp2().long()]).clamp_(max=2 ** 31 - 2)
    q = torch.minimum(q, 2 ** 62 // d - 1)
    want = torch.cat([q, q, q])
    n = torch.cat([q * d, q * d + d - 1, q * d + d // 2])
    d = torch.cat([d, d, d])
    assert torch.equal(kvq.kvq_debug_divide(n.cuda(), d.cuda()).cpu(), want) and torch.equal(n // d, want)
