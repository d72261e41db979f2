"""Shared memory of the decode kernel, as far as it can be checked without a GPU."""
import collections
import os
import re

import pytest

from paper_2502_15075_b200 import build as kvq_build

CSRC = os.path.join(os.path.dirname(kvq_build.__file__), "csrc")
KERNEL = os.path.join(CSRC, "kvq_decode_mma_kernel.cuh")
INSTANCES = [tuple(int(x) for x in m.split(",")) for m in
             re.findall(r"^KVQ_MMA_DECL\(([^)]*)\)", open(os.path.join(CSRC, "kvq_decode_mma_list.inc")).read(), re.M)]


@pytest.fixture(scope="module")
def kvq():
    kvq_build.build()
    from paper_2502_15075_b200 import kvq as mod
    return mod


def test_a_bookkeeping_word_is_set_in_one_place():
    """A word that is set in two places for two readers, with no barrier between, can be overwritten before a slow warp has read it;
    that warp then leaves, or stays, alone, and the others wait for it at the next barrier.  (The abort flag is cleared at the start
    and set through a pointer.)"""
    source = re.sub(r"//[^\n]*", "", open(KERNEL).read())
    sets = collections.Counter(re.findall(r"sMisc\[(\w+)\]\s*=(?!=)", source))
    assert len(sets) >= 8, "the words are no longer written as this test expects"
    assert {w: n for w, n in sets.items() if n > 1} == {}


@pytest.mark.parametrize("R", [64, 128])
@pytest.mark.parametrize("inst", [i for i in INSTANCES if i[3] == 0], ids=str)        # (no window with channel-wise keys)
def test_a_window_read_from_the_ring_lies_inside_it(kvq, inst, R):
    """The logits of a window read whole tiles of 16 rows of (key, value) in 16 bits each, beyond the rows that were copied."""
    D, kb, vb, axis, ngk, ngv, nh, per_sm = inst
    for batch in (1, 7, 64, 1024):
        cfg = kvq.make_config(batch, 4 * nh, 1, D, kb, vb, D // ngk, D // ngv, 0, "bf16", 256, R)
        ring, longest = kvq.kvq_debug_decode_ring(cfg)
        assert 0 < longest < R and -(-longest // 16) * 16 * 4 * D <= ring
        assert longest == R - 1 or -(-(longest + 1) // 16) * 16 * 4 * D > ring        # (no window is sent the longer way without need)
