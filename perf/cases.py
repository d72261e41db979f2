"""Workloads of the packed KV cache as a serving loop and the paper's analysis have them, for timing and comparing builds.

A case is one pass of one of four kinds of work, through the library's Python calls:

  step     one decoding step of `layers` layers: per layer, quantize-append `append` new tokens per sequence, decode
           attention over the whole cache (`rows` causal query rows) and, with `restore`, dequantize the newest page;
  append   prefill: quantize-append `tokens` tokens per sequence behind `prior` cached ones, per layer;
  restore  dequantize `tokens` cached tokens of every layer back to 16 bits;
  error    reconstruction-error sums of K and V at several bit widths, per layer.

Shapes and value recipes are those of `paper_2502_15075_b200.workloads`; lengths, batches and layer counts vary.  Layers
of large cases are fewer than the model's, but together never fit the 126 MB L2, as in a model.  `draw` gives further
cases of the same four kinds over every shape, width pair and option that the listed ones stand for.  Bit planes (1, 3
and 6 bits) appear in the error analysis only, which is where the paper's tables use them.
"""
from __future__ import annotations

import math

import torch

from paper_2502_15075_b200 import kvq, workloads as wl

SHAPES = {"tiny": wl.TINY, "1b": wl.LLAMA_1B, "8b": wl.LLAMA_8B, "14b": wl.SHAPED_14B, "70b": wl.LLAMA_70B}
# (key bits, value bits) of the bit-width sweeps each shape is used with
WIDTHS = {"tiny": [(4, 2)], "1b": [(4, 2)], "8b": [(4, 2), (2, 4), (4, 4), (8, 4)], "14b": [(4, 2), (8, 2)], "70b": [(4, 2)]}
DTYPES = {"fp16": torch.float16, "bf16": torch.bfloat16, "fp32": torch.float32}
PAGE = kvq.PAGE_TOKENS
MAX_BYTES = 1.3e9          # a drawn case moves no more than the largest listed one
MIN_CONTEXT = 192          # shortest context of a decoding step


def _case(kind, shape, name=None, **over):
    w = SHAPES[shape]
    c = {"kind": kind, "shape": shape, "layers": 1, "batch": w.batch, "kb": w.kb, "vb": w.vb, "tokens": w.context,
         "append": 1, "prior": 0, "rows": 1, "ragged": False, "rotated": False, "window": 0, "restore": False, "out": "fp32"}
    c.update(over)
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest call of all: one sequence, one short-context layer, where latency and launches are everything
        _case("step", "tiny", "step_tiny_k4v2", out="fp16"),
        # a whole small model: 16 layers take in 128 new tokens per sequence, then decode one step at a 4k context
        _case("step", "1b", "step_1b_append128", layers=16, append=128, out="fp16"),
        # the benchmark's step at 32k tokens: append one token, decode, give back the newest page
        _case("step", "8b", "step_8b_32k", layers=2, restore=True),
        # a small batch of uneven lengths at equal widths (the paper's 4-bit baseline)
        _case("step", "8b", "step_8b_k4v4_ragged", layers=8, batch=5, tokens=9001, vb=4, ragged=True, out="bf16"),
        # channel-wise keys with fp16 tails of every length
        _case("step", "14b", "step_14b_channel_ragged", layers=2, ragged=True),
        # eight query heads per KV head at a 128k context
        _case("step", "70b", "step_70b_128k", layers=2, tokens=131071, out="bf16"),
        # the paper's 64-token residual window at its 2k contexts, with two drafted tokens verified at once
        _case("step", "8b", "step_8b_window_draft", layers=8, batch=4, tokens=2000, append=2, rows=2, window=64, ragged=True, out="bf16"),
        # prefill of one layer, token-wise groups: the largest call
        _case("append", "8b", "prefill_8b_32k", batch=8),
        # prefill with channel-wise keys that ends in an incomplete block
        _case("append", "14b", "prefill_14b_channel", batch=12, tokens=16383),
        # chunked prefill of rotated keys onto a context that ends inside a page
        _case("append", "70b", "chunk_70b_rotated", layers=4, tokens=2047, prior=4101, rotated=True),
        # a whole layer back to 16 bits, as a preempted request's cache is handed to a dense kernel
        _case("restore", "8b", "restore_8b_32k", batch=8),
        # the reconstruction-error table: ten sequences of up to 1000 tokens at 2, 3 and 4 bits
        _case("error", "8b", "error_8b_table1", layers=4, batch=10, tokens=1000),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        kind = rng.choice(["step", "step", "step", "append", "append", "restore", "error"])
        shape = rng.choice(["8b", "8b", "14b", "70b", "1b", "tiny"] if kind != "error" else ["8b", "70b"])
        w = SHAPES[shape]
        c = _case(kind, shape)
        c["kb"], c["vb"] = rng.choice(WIDTHS[shape])
        c["batch"] = _log_int(rng, 1, max(w.batch, 8))
        c["layers"] = _log_int(rng, 1, 8)
        c["out"] = rng.choice([w.dtype, "fp32"])
        if kind == "step":
            c["tokens"] = _log_int(rng, MIN_CONTEXT, w.context)
            c["ragged"] = rng.random() < 0.5
            c["restore"] = not c["ragged"] and rng.random() < 0.3
            if w.k_axis == 0:
                c["rotated"] = rng.random() < 0.25
                extra = rng.random()
                if extra < 0.25:
                    c["window"] = rng.choice([64, 128])
                if extra > 0.75 and shape == "8b" and (c["kb"], c["vb"]) == (4, 2):
                    c["append"] = c["rows"] = 2
                elif extra > 0.5:
                    c["append"] = _log_int(rng, 1, 128) if c["window"] == 0 else 1
        elif kind == "append":
            c["tokens"] = _log_int(rng, 17, w.context)
            c["rotated"] = rng.random() < 0.3
            if rng.random() < 0.4:
                c["prior"] = _log_int(rng, 1, max(1, w.context // 4))
                if w.k_axis == 1:        # a pass has to find the tail as it was: start behind a complete block
                    c["prior"] = -(-c["prior"] // PAGE) * PAGE
        else:
            c["tokens"] = _log_int(rng, 33, w.context if kind == "restore" else 2000)
            c["rotated"] = kind == "restore" and rng.random() < 0.25
        if work(c)["bytes"] <= MAX_BYTES and _resident_bytes(c) <= 6e9:
            return c


# ----------------------------------------------------------------------------------------------------------- inputs
def _workload(c, seed):
    """The case's workload with a seed base of its own."""
    w = SHAPES[c["shape"]]
    return w.with_(batch=c["batch"], kb=c["kb"], vb=c["vb"], layers=c["layers"], number=w.number + 10 * (1 + abs(int(seed)) % 10 ** 9))


def _config(c, w):
    cap = -(-(c["prior"] + c["tokens"]) // PAGE) * PAGE + PAGE
    return kvq.make_config(w.batch, w.n_q_heads, w.n_kv_heads, w.head_dim, w.kb, w.vb, w.gk, w.gv, w.k_axis, w.torch_dtype,
                           cap, c["window"])


def _base_lens(c, w, seed):
    """Cached tokens per sequence before a step, on the CPU."""
    T = c["tokens"]
    lens = wl.ragged_seq_lens(w, T, w.batch, seed % 1000) if c["ragged"] else torch.full((w.batch,), T, dtype=torch.int32)
    base = (lens - c["append"]).clamp_(min=0)
    unit = PAGE if w.k_axis == 1 else c["window"]
    if unit:      # a step that completes a block and also leaves new tokens behind it would not find its tail again
        over = base % unit + c["append"] > unit
        base = torch.where(over, base - c["append"], base).to(torch.int32)
    return base


def prepare(case, seed):
    c, dev = case, "cuda"
    w = _workload(c, seed)
    cfg = _config(c, w)
    T, B, H, D = c["tokens"], w.batch, w.n_kv_heads, w.head_dim
    s = {"case": dict(c), "cfg": cfg, "kvq": kvq}
    if c["kind"] == "error":
        s["kv"] = [wl.make_kv(w, layer, dev, tokens=T) for layer in range(w.layers)]
        s["cfgs"] = [kvq.make_config(B, w.n_q_heads, H, D, b, b, w.gk, w.gv, 0, w.torch_dtype, PAGE) for b in (2, 3, 4)]
        s["sums"] = torch.zeros((w.layers, len(s["cfgs"]), B, H, 4), dtype=torch.float64, device=dev)
        return s
    signs = None
    if c["rotated"]:
        g = torch.Generator().manual_seed(abs(int(seed)) + 1)
        signs = (torch.randint(0, 2, (D,), generator=g, dtype=torch.int8) * 2 - 1).to(dev)
    s["lens"] = torch.zeros((w.layers, B), dtype=torch.int32, device=dev)
    s["caches"] = [kvq.Cache(cfg, device=dev, k_signs=signs, seq_len=s["lens"][i]) for i in range(w.layers)]
    if c["kind"] == "append":
        s["new"] = []
        for i, cache in enumerate(s["caches"]):
            k, v = wl.make_kv(w, i, dev, tokens=c["prior"] + T)
            if c["prior"]:
                kvq.kvq_quantize_append(cfg, cache, k[:, :, :c["prior"]], v[:, :, :c["prior"]])
            s["new"].append((k[:, :, c["prior"]:], v[:, :, c["prior"]:]))
        s["base"] = torch.full((w.layers, B), c["prior"], dtype=torch.int32, device=dev)
        return s
    if c["kind"] == "restore":
        for i, cache in enumerate(s["caches"]):
            kvq.kvq_quantize_append(cfg, cache, *wl.make_kv(w, i, dev, tokens=T))
        s["outs"] = [tuple(torch.zeros((B, H, cfg.capacity_tokens, D), dtype=w.torch_dtype, device=dev) for _ in range(2))
                     for _ in range(w.layers)]
        return s
    base = _base_lens(c, w, abs(int(seed)))
    s["base"] = base.to(dev).unsqueeze(0).repeat(w.layers, 1)
    n, lead = c["append"], min(PAGE, int(base.min()))
    s["new"], s["q"], s["out"] = [], [], []
    qshape = (B, w.n_q_heads, D) if c["rows"] == 1 else (B, c["rows"], w.n_q_heads, D)
    for i, cache in enumerate(s["caches"]):
        k, v = wl.make_kv(w, i, dev, tokens=T)
        kvq.kvq_quantize_append(cfg, cache, k, v)
        if lead:           # the last tokens before the step once more, at each sequence's own length: tails and windows
            cache.seq_len.copy_(s["base"][i] - lead)
            kvq.kvq_quantize_append(cfg, cache, k[:, :, T - lead:], v[:, :, T - lead:])
        s["new"].append(tuple(t.contiguous() for t in wl.make_kv(w, 100 + i, dev, tokens=n)))
        q = wl.make_q(w, i, dev, batch=B * c["rows"])
        s["q"].append(q.view(qshape))
        s["out"].append(torch.zeros(qshape, dtype=DTYPES[c["out"]], device=dev))
        del k, v
    s["ws"] = torch.empty(kvq.kvq_workspace_bytes_rows(cfg, c["rows"]), dtype=torch.uint8, device=dev)
    if c["restore"]:
        s["deq"] = [torch.zeros((B, H, cfg.capacity_tokens, D), dtype=w.torch_dtype, device=dev) for _ in range(2)]
    return s


# ------------------------------------------------------------------------------------------------------------- pass
def run(state):
    c, lib = state["case"], state["kvq"]
    if c["kind"] == "error":
        sums = state["sums"].zero_()
        for i, (k, v) in enumerate(state["kv"]):
            for j, cfg in enumerate(state["cfgs"]):
                lib.kvq_quant_error(cfg, k, v, sums[i, j])
        return sums
    cfg, caches = state["cfg"], state["caches"]
    if c["kind"] == "restore":
        for cache, (k_out, v_out) in zip(caches, state["outs"]):
            lib.kvq_dequantize(cfg, cache, k_out, v_out, 0, c["tokens"])
        return state["outs"]
    state["lens"].copy_(state["base"])       # all layers' lengths, as the scheduler hands them out before a step
    if c["kind"] == "append":
        for cache, (k, v) in zip(caches, state["new"]):
            lib.kvq_quantize_append(cfg, cache, k, v)
        return [[cache.pages for cache in caches], [cache.k_tail for cache in caches], state["lens"]]
    t_end = c["tokens"]
    page0 = (t_end - 1) // PAGE * PAGE
    for cache, (k, v), q, out in zip(caches, state["new"], state["q"], state["out"]):
        lib.kvq_quantize_append(cfg, cache, k, v)
        if c["rows"] == 1:
            lib.kvq_decode_attention(cfg, cache, q, out, state["ws"])
        else:
            lib.kvq_decode_attention_rows(cfg, cache, q, out, state["ws"])
        if c["restore"]:
            lib.kvq_dequantize(cfg, cache, state["deq"][0], state["deq"][1], page0, t_end)
    written = [t[:, :, page0:t_end] for t in state["deq"]] if c["restore"] else []      # all that the last call wrote
    return [state["out"], [cache.pages for cache in caches], [cache.k_tail for cache in caches],
            [cache.kv_win for cache in caches], state["lens"], written]


# ------------------------------------------------------------------------------------------------- what a pass needs
def _resident_bytes(c):
    """16-bit bytes of one state's tokens (inputs or outputs of the largest kind)."""
    w = SHAPES[c["shape"]]
    return 4.0 * c["layers"] * c["batch"] * w.n_kv_heads * w.head_dim * (c["prior"] + c["tokens"])


def work(case):
    c = case
    w = SHAPES[c["shape"]].with_(kb=c["kb"], vb=c["vb"])
    streams = c["layers"] * c["batch"] * w.n_kv_heads
    dense = 4.0 * w.head_dim                              # 16-bit K and V of one token
    packed = wl.packed_bytes_per_token(w)
    if c["kind"] == "error":
        n = streams * c["tokens"]
        return {"bytes": n * dense, "flops": 3 * 10.0 * n * 2 * w.head_dim}
    if c["kind"] == "append":
        n = streams * c["tokens"]
        return {"bytes": n * (dense + packed), "flops": 6.0 * n * 2 * w.head_dim}
    if c["kind"] == "restore":
        n = streams * c["tokens"]
        return {"bytes": n * (dense + packed), "flops": 2.0 * n * 2 * w.head_dim}
    mean = (0.75 if c["ragged"] else 1.0) * c["tokens"]   # ragged lengths are uniform in [tokens / 2, tokens]
    heads = c["rows"] * w.n_q_heads // w.n_kv_heads
    need = mean * packed + c["append"] * (dense + packed)
    need += heads * w.head_dim * (2 + (4 if c["out"] == "fp32" else 2))
    if c["window"]:
        need += min(mean, c["window"] / 2) * (dense - packed)
    elif w.k_axis == 1:
        need += min(mean, PAGE / 2) * (2.0 * w.head_dim - w.head_dim * w.kb / 8)
    if c["restore"]:
        need += (c["tokens"] - (c["tokens"] - 1) // PAGE * PAGE) * (dense + packed)
    return {"bytes": streams * need, "flops": 4.0 * streams * heads * w.head_dim * mean}


def tolerance(case):
    """Packed bytes, tails, windows, restored values and lengths are exact.  Attention: the fixed-point queries and weights
    leave 1.2e-4 (token-wise), 1.7e-4 (2-bit keys) and 2.4e-5 (channel-wise) of relative error against fp64 attention over
    the same codes; a 16-bit output adds the roundings that such a difference turns over (fp16 2^-11, bf16 2^-8 apart).
    The error sums add fp32 squares in double precision."""
    if case["kind"] in ("append", "restore"):
        return "exact"
    if case["kind"] == "error":
        return {"rel": 1e-5, "max": 1e-4}
    return {"fp32": {"rel": 6e-4, "max": 5e-3}, "fp16": {"rel": 1e-3, "max": 6e-3}, "bf16": {"rel": 3e-3, "max": 2e-2}}[case["out"]]


# ---------------------------------------------------------------------------------------------- the same in 64 bits
def _hadamard(x, signs, inverse=False):
    """Randomized Hadamard rotation of the last axis, stage by stage, in x's own precision."""
    D = x.shape[-1]
    y, h = (x if inverse else x * signs.to(x.dtype)), 1
    while h < D:
        p = y.reshape(*y.shape[:-1], D // (2 * h), 2, h)
        y = torch.stack((p[..., 0, :] + p[..., 1, :], p[..., 0, :] - p[..., 1, :]), dim=-2).reshape(x.shape)
        h *= 2
    y = y * torch.tensor(1.0 / math.sqrt(D), dtype=x.dtype, device=x.device)
    return y * signs.to(x.dtype) if inverse else y


def _reconstructed(x, bits, dim):
    """x (fp32, one group along `dim`) quantized with fp16 scale and minimum, and back in 64 bits."""
    qmax = torch.tensor(2.0 ** bits - 1.0, device=x.device)
    lo, hi = x.amin(dim, keepdim=True) + 0.0, x.amax(dim, keepdim=True) + 0.0
    s = ((hi - lo) / qmax).clamp(-65504.0, 65504.0).half().float()
    z = lo.clamp(-65504.0, 65504.0).half().float()
    inv = torch.where(s != 0, torch.ones_like(s) / s, torch.zeros_like(s))
    code = torch.minimum(torch.round((x - z) * inv).clamp(min=0.0), qmax)
    return code.double() * s.double() + z.double()


class _Sequence:
    """One sequence of one layer: its tokens as the cache holds them, in 64 bits (keys rotated where the cache rotates)."""

    def __init__(self, c, w, cap, signs, dev):
        self.c, self.w, self.signs, self.n = c, w, signs, 0
        shape = (w.n_kv_heads, cap, w.head_dim)
        self.k, self.v = (torch.zeros(shape, dtype=torch.float64, device=dev) for _ in range(2))
        self.win = torch.zeros((2, w.n_kv_heads, max(c["window"], 1), w.head_dim), device=dev)
        self.tail = torch.zeros((w.n_kv_heads, PAGE, w.head_dim), device=dev)

    def _tokenwise(self, x, bits, group):
        return _reconstructed(x.reshape(*x.shape[:-1], -1, group), bits, -1).reshape(x.shape)

    def append(self, k, v):
        w, R, t0 = self.w, self.c["window"], self.n
        end = self.n = t0 + k.shape[1]
        k, v = k.float(), v.float()
        qa, qb = (t0 // R * R, end // R * R) if R else (t0, end)
        if R and qb > qa:
            slots = torch.arange(qa, t0, device=k.device) % R
            kq, vq = (torch.cat((self.win[i][:, slots], x), 1)[:, :qb - qa] for i, x in enumerate((k, v)))
        else:
            kq, vq = k[:, :qb - qa], v[:, :qb - qa]
        kr = _hadamard(kq, self.signs) if self.signs is not None else kq
        if qb > qa:
            self.v[:, qa:qb] = self._tokenwise(vq, w.vb, w.gv)
        if w.k_axis == 1:
            first = t0 // PAGE * PAGE
            x = torch.cat((self.tail[:, :t0 - first], kr.clamp(-65504.0, 65504.0).half().float()), 1)
            full = x.shape[1] // PAGE * PAGE
            blocks = x[:, :full].reshape(x.shape[0], -1, PAGE, x.shape[2])
            if full:
                self.k[:, first:first + full] = _reconstructed(blocks, w.kb, 2).flatten(1, 2)
            self.tail[:, :x.shape[1] - full] = x[:, full:]
            self.k[:, first + full:end] = x[:, full:].double()
        elif qb > qa:
            self.k[:, qa:qb] = self._tokenwise(kr, w.kb, w.gk)
        if R:
            keep = torch.arange(max(t0, qb), end, device=k.device)
            self.win[0][:, keep % R], self.win[1][:, keep % R] = k[:, keep - t0], v[:, keep - t0]

    def attend(self, q):
        """q [rows, Hq, D]: causal rows over the last positions."""
        w, R, n = self.w, self.c["window"], self.n
        rows, H, D = q.shape[0], w.n_kv_heads, w.head_dim
        q = q.double().reshape(rows, H, -1, D).transpose(0, 1)                       # [H, rows, G, D]
        qr = _hadamard(q, self.signs) if self.signs is not None else q
        packed = n // R * R if R else n
        logits = torch.einsum("hrgd,htd->hrgt", qr, self.k[:, :packed])
        values = self.v[:, :packed]
        if R:
            slots = torch.arange(packed, n, device=q.device) % R
            logits = torch.cat((logits, torch.einsum("hrgd,htd->hrgt", q, self.win[0][:, slots].double())), -1)
            values = torch.cat((values, self.win[1][:, slots].double()), 1)
        seen = torch.arange(n, device=q.device) <= n - rows + torch.arange(rows, device=q.device)[:, None]
        p = torch.softmax(logits.div(math.sqrt(D)).masked_fill(~seen[None, :, None], -math.inf), -1)
        return torch.einsum("hrgt,htd->hrgd", p, values).transpose(0, 1).reshape(rows, -1, D)


def exact(case, seed):
    """What `run` returns in 64 bits over the same codes; packed bytes, tails, windows and lengths have no such value."""
    c, dev = case, "cuda"
    w = _workload(c, seed)
    T, B, H, D = c["tokens"], w.batch, w.n_kv_heads, w.head_dim
    if c["kind"] == "append":
        return None
    if c["kind"] == "error":
        sums = torch.zeros((w.layers, 3, B, H, 4), dtype=torch.float64, device=dev)
        for i in range(w.layers):
            for side, x in enumerate(wl.make_kv(w, i, dev, tokens=T)):
                x = x.float()
                for j, bits in enumerate((2, 3, 4)):
                    g = x.reshape(B, H, T, -1, (w.gk, w.gv)[side])
                    sums[i, j, :, :, 2 * side] = x.double().square().sum((2, 3))
                    sums[i, j, :, :, 2 * side + 1] = (g.double() - _reconstructed(g, bits, -1)).square().sum((2, 3, 4))
        return sums
    cap = _config(c, w).capacity_tokens
    signs = None
    if c["rotated"]:
        g = torch.Generator().manual_seed(abs(int(seed)) + 1)
        signs = (torch.randint(0, 2, (D,), generator=g, dtype=torch.int8) * 2 - 1).to(dev)
    base = None if c["kind"] == "restore" else _base_lens(c, w, abs(int(seed)))
    n, lead = c["append"], 0 if base is None else min(PAGE, int(base.min()))
    page0 = (T - 1) // PAGE * PAGE
    outs, written = [], []
    for i in range(w.layers):
        k, v = wl.make_kv(w, i, dev, tokens=T)
        if base is None:
            back = tuple(torch.zeros((B, H, cap, D), dtype=torch.float64, device=dev) for _ in range(2))
        else:
            new = wl.make_kv(w, 100 + i, dev, tokens=n)
            q = wl.make_q(w, i, dev, batch=B * c["rows"]).view(B, c["rows"], w.n_q_heads, D)
            out = torch.zeros(q.shape, dtype=torch.float64, device=dev)
            back = tuple(torch.zeros((B, H, T - page0, D), dtype=torch.float64, device=dev) for _ in range(2))
        for b in range(B):
            s = _Sequence(c, w, cap, signs, dev)
            s.append(k[b], v[b])
            if base is not None:
                if lead:
                    s.n = int(base[b]) - lead
                    s.append(k[b][:, T - lead:], v[b][:, T - lead:])
                s.n = int(base[b])
                s.append(new[0][b], new[1][b])
                out[b] = s.attend(q[b])
            if base is None or c["restore"]:
                at = slice(0, T) if base is None else slice(page0, T)
                unrotated = s.k[:, at] if signs is None else _hadamard(s.k[:, at], signs, inverse=True)
                back[0][b, :, :at.stop - at.start], back[1][b, :, :at.stop - at.start] = unrotated, s.v[:, at]
        if base is None:
            outs.append(back)
        else:
            outs.append(out.view(B, w.n_q_heads, D) if c["rows"] == 1 else out)
            written = list(back) if c["restore"] else []
    if base is None:
        return outs
    none = [None] * w.layers
    return [outs, none, none, none, None, written]
