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
    q = wl.make_q(w, batch=B).cuda()
    ws = torch.empty(kvq.kvq_workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    error_cfg = kvq.make_config(B, w.n_q_heads, w.n_kv_heads, w.head_dim, 4, 4, w.gk, w.gv, 0, w.torch_dtype, 128)

    def chain(cache, outs, back, sums, between):
        t = 0
        for n, out in zip(chunks, outs):
            kvq.kvq_quantize_append(cfg, cache, k[:, :, t:t + n], v[:, :, t:t + n])
            between()
            kvq.kvq_decode_attention(cfg, cache, q, out, ws)
            between()
            t += n
            kvq.kvq_dequantize(cfg, cache, back[0], back[1], 0, t)
            between()
            kvq.kvq_quant_error(error_cfg, back[0][:, :, :t], back[1][:, :, :t], sums)
            between()

    def buffers():
        return (kvq.Cache(cfg, k_signs=signs), [torch.empty(q.shape, device="cuda") for _ in chunks],
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
            for t in (got[0].seq_len, got[0].pages, got[3]):
                t.zero_()
            graph.replay()
    torch.cuda.synchronize()
    assert torch.equal(got[0].seq_len, want[0].seq_len) and torch.equal(got[0].pages, want[0].pages)
    if want[0].k_tail is not None:
        assert torch.equal(got[0].k_tail, want[0].k_tail)
    for a, b in zip(got[1] + got[2], want[1] + want[2]):
        assert torch.equal(a, b)
    # double atomics add the CTAs' sums in any order: a few units of 2^-53 of the total
    assert torch.allclose(got[3], want[3], rtol=1e-13, atol=0)
    assert kvq.kvq_check_status(got[0]) == 0
