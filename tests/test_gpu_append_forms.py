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


def edge_values(w, T, B, seed):
    """Keys and values with constant groups, signed zeros, subnormal ranges and entries at the ends of the 16-bit type."""
    k, v = wl.make_kv(w.with_(number=seed), tokens=T, batch=B)
    big = 65504.0 if w.dtype == "fp16" else 3.0e38
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
    k, v = edge_values(w, T, B, seed)
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
