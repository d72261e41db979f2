"""Shared memory of the decode kernel, as far as it can be checked without a GPU."""
import collections
import os
import re

from paper_2502_15075_b200 import build as kvq_build

KERNEL = os.path.join(os.path.dirname(kvq_build.__file__), "csrc", "kvq_decode_mma_kernel.cuh")


def test_a_bookkeeping_word_is_set_in_one_place():
    """A word that is set in two places for two readers, with no barrier between, can be overwritten before a slow warp has read it;
    that warp then leaves, or stays, alone, and the others wait for it at the next barrier.  (The abort flag is cleared at the start
    and set through a pointer.)"""
    source = re.sub(r"//[^\n]*", "", open(KERNEL).read())
    sets = collections.Counter(re.findall(r"sMisc\[(\w+)\]\s*=(?!=)", source))
    assert len(sets) >= 8, "the words are no longer written as this test expects"
    assert {w: n for w, n in sets.items() if n > 1} == {}
