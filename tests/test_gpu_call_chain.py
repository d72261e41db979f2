"""Calls queued behind one another on a stream, each launched as a dependent of the kernel before it, give the bytes they
give when the device is waited for after every call - eagerly, on a side stream and replayed from a graph."""
import pytest
import torch

from paper_2502_15075_b200 import workloads as wl

import kvq_testlib as tl

pytestmark = pytest.mark.gpu
SMALL = wl.LLAMA_8B.with_(n_kv_heads=2, n_q_heads=8)


@pytest.fixture(scope="module")
def kvq():
    from paper_2502_15075_b200 import build
    build.build()
    from paper_2502_15075_b200 import kvq as mod
    return mod


# (workload, rotated, residual window, tokens of the appends in turn): short and long appends, channel-wise blocks and tail, a
# window that fills and is flushed, bit planes and 16-bit keys (generic decode kernel and its merge)
@pytest.mark.parametrize("w,rotated,window,chunks", [
    (SMALL, False, 0, (700, 1, 130, 3)),
    (SMALL, True, 0, (2047, 1, 200, 1)),
    (SMALL, False, 64, (500, 1, 70, 130, 1)),
    (wl.SHAPED_14B.with_(n_kv_heads=2, n_q_heads=8), False, 0, (1000, 1, 30, 300)),
    (SMALL.with_(kb=3, vb=6), False, 0, (300, 1, 90)),
    (SMALL.with_(kb=16), False, 0, (300, 1, 90)),
    (wl.LLAMA_1B.with_(n_kv_heads=2, n_q_heads=8), False, 0, (640, 128, 1)),
])
@pytest.mark.parametrize("how", ["eager", "side stream", "graph"])
def test_queued_calls_equal_calls_one_by_one(kvq, w, rotated, window, chunks, how):
    B, T = 3, sum(chunks)
    cap = -(-T // 128) * 128
    cfg = tl.gpu_config_for(kvq, w, B, cap, window)
    signs = torch.ones(w.head_dim, dtype=torch.int8) if rotated else None
    if rotated:
        signs[1::3] = -1
    k, v = (t.cuda() for t in wl.make_kv(w, tokens=T, batch=B))
    rows = 2 if (w.kb, w.vb, w.k_axis, w.head_dim) == (4, 2, 0, 128) else 1          # (eight virtual heads: this form only)
    q = wl.make_q(w, batch=B * (1 + rows)).cuda()
    q, q_rows = q[:B], q[B:].view(B, rows, w.n_q_heads, w.head_dim)
    ws = torch.empty(kvq.kvq_workspace_bytes_rows(cfg, rows), dtype=torch.uint8, device="cuda")
    error_cfg = kvq.make_config(B, w.n_q_heads, w.n_kv_heads, w.head_dim, 4, 4, w.gk, w.gv, 0, w.torch_dtype, 128)

    def chain(cache, outs, back, sums, between):
        t = 0
        for n, (out, out_rows, out_static) in zip(chunks, outs):
            kvq.kvq_quantize_append(cfg, cache, k[:, :, t:t + n], v[:, :, t:t + n])
            between()
            kvq.kvq_decode_attention(cfg, cache, q, out, ws)
            between()
            kvq.kvq_decode_attention_rows(cfg, cache, q_rows, out_rows, ws)
            between()
            kvq.kvq_decode_attention_static(cfg, cache, q, out_static)
            between()
            t += n
            kvq.kvq_dequantize(cfg, cache, back[0], back[1], 0, t)
            between()
            kvq.kvq_quant_error(error_cfg, back[0][:, :, :t], back[1][:, :, :t], sums)
            between()

    def buffers():
        return (kvq.Cache(cfg, k_signs=signs), [tuple(torch.empty(s, device="cuda") for s in (q.shape, q_rows.shape, q.shape)) for _ in chunks],
                [torch.zeros_like(k[:, :, :1]).expand(-1, -1, cap, -1).contiguous() for _ in range(2)],
                torch.zeros((B, w.n_kv_heads, 4), dtype=torch.float64, device="cuda"))

    want, got = buffers(), buffers()
    chain(*want, torch.cuda.synchronize)
    if how == "eager":
        chain(*got, lambda: None)
    else:
        s = torch.cuda.Stream()
        s.wait_stream(torch.cuda.current_stream())
        if how == "side stream":
            with torch.cuda.stream(s):
                chain(*got, lambda: None)
        else:
            graph = torch.cuda.CUDAGraph()
            with torch.cuda.graph(graph, stream=s):
                chain(*got, lambda: None)
            graph.replay()
            torch.cuda.synchronize()
            # everything that a replay writes starts from something else again
            for t in (got[0].seq_len, got[0].pages, got[3], *got[2]):
                t.zero_()
            for t in (got[0].k_tail, got[0].kv_win, *(x for out in got[1] for x in out)):
                if t is not None:
                    t.fill_(7)
            graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(got[0].seq_len, want[0].seq_len) and torch.equal(got[0].pages, want[0].pages)
    if want[0].k_tail is not None:
        held = T % 128 if how == "graph" else 128              # (slots behind the incomplete block's tokens keep what they had)
        assert torch.equal(got[0].tail_view()[:, :, :held], want[0].tail_view()[:, :, :held])
    if window:
        held = T % window if how == "graph" else window
        assert torch.equal(got[0].window_view()[:, :, :held], want[0].window_view()[:, :, :held])
    for a, b in zip([x for out in got[1] for x in out] + got[2], [x for out in want[1] for x in out] + want[2]):
        assert torch.equal(a, b)
    for out, _, out_static in got[1]:
        assert torch.equal(out, out_static)
    # double atomics add the CTAs' sums in any order: a few units of 2^-53 of the total
    assert torch.allclose(got[3], want[3], rtol=1e-13, atol=0)
    assert kvq.kvq_check_status(got[0]) == 0


@pytest.mark.parametrize("how", ["eager", "graph"])
def test_work_joined_from_a_second_stream_is_waited_for(kvq, how):
    """A call behind an event of another stream: the keys that stream makes, and the cache it appends to, are complete before the call
    reads them - also where the call's own stream has a library kernel right in front."""
    w, B, T, rounds = SMALL, 3, 400, 4
    cfg = tl.gpu_config_for(kvq, w, B, 512)
    k, v = (t.cuda() for t in wl.make_kv(w, tokens=T, batch=B))
    q = wl.make_q(w, batch=B).cuda()
    ws = torch.empty(kvq.kvq_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    caches = [kvq.Cache(cfg) for _ in range(2)]
    kn, vn = torch.empty_like(k), torch.empty_like(v)
    outs = torch.empty((rounds, 2, *q.shape), device="cuda")

    def work(side):
        main = torch.cuda.current_stream()
        for r in range(rounds):
            for c in caches:
                c.seq_len.zero_()
            side.wait_stream(main)
            with torch.cuda.stream(side):
                for _ in range(20):                               # (long enough that the other stream's kernels are through first)
                    torch.mul(k, float(r + 1), out=kn)
                    torch.mul(v, float(r + 1), out=vn)
                kvq.kvq_quantize_append(cfg, caches[1], kn, vn)
            kvq.kvq_quantize_append(cfg, caches[0], k, v)
            kvq.kvq_decode_attention(cfg, caches[0], q, outs[r, 0], ws)
            main.wait_stream(side)
            kvq.kvq_decode_attention(cfg, caches[1], q, outs[r, 1], ws)

    want = torch.empty_like(outs)
    for r in range(rounds):
        for i, scale in enumerate((1.0, float(r + 1))):
            c = kvq.Cache(cfg)
            kvq.kvq_quantize_append(cfg, c, k * scale, v * scale)
            torch.cuda.synchronize()
            kvq.kvq_decode_attention(cfg, c, q, want[r, i], ws)
            torch.cuda.synchronize()
    side = torch.cuda.Stream()
    if how == "eager":
        work(side)
    else:
        graph, main = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        main.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(graph, stream=main):
            work(side)
        for _ in range(2):
            outs.fill_(7.0)
            kn.zero_()
            vn.zero_()
            graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(outs, want)
