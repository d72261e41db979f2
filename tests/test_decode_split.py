"""The decode kernel's split of the pages over its CTAs: every page in one share, every stream's partials counted as the
shares hold them, and never more of them than a stream has slots (a partial without a slot would leave the output unwritten).
The library works the split out on the host with the kernel's own functions.  No GPU needed."""
import random

import numpy as np
import pytest

from paper_2502_15075_b200 import build as kvq_build

PAGE = 128


@pytest.fixture(scope="module")
def kvq():
    kvq_build.build()
    from paper_2502_15075_b200 import kvq as mod
    return mod


def check_split(kvq, cfg, pages, rows=1):
    lens = [PAGE * p - (7 * i) % PAGE if p else 0 for i, p in enumerate(pages)]        # p pages, the last one incomplete
    slots, weighted, starts, parts = kvq.kvq_debug_decode_plan(cfg, lens, rows)
    H, first = cfg.n_kv_heads, 0
    cursors, before = kvq.kvq_debug_decode_cursors(cfg, lens, rows), np.cumsum([0] + [H * p for p in pages])
    for (b, h, page), start in zip(cursors, starts[:-1]):               # the share's first page, said twice
        assert 0 <= h < H and 0 <= page < pages[b] and before[b] + h * pages[b] + page == start
    assert len(cursors) == len(starts) - 1
    assert starts[0] == 0 and starts[-1] == H * sum(pages) and np.all(np.diff(starts) >= 0)
    for b, p in enumerate(pages):
        for h in range(H):
            c0, n = parts[b * H + h]
            if p:
                holds = np.nonzero((starts[1:] > first) & (starts[:-1] < first + p) & (starts[1:] > starts[:-1]))[0]
                assert holds.tolist() == list(range(c0, c0 + n)), f"sequence {b} head {h}: partials {c0}+{n}, shares {holds}"
                assert n <= slots, f"sequence {b} head {h} ({p} pages): {n} partials, {slots} slots"
            else:
                assert (c0, n) == (0, 0)
            first += p
    return weighted


# (key bits, value bits, key axis, query heads per KV head, head_dim, group): three weighted waves with the stream gap of token-wise
# and of channel-wise keys, two weighted waves, equal shares, the gap of head_dim 64
FORMS = {"token": (4, 2, 0, 4, 128, 128), "channel": (4, 2, 1, 4, 128, 128), "eight heads": (4, 2, 0, 8, 128, 128),
         "wide pages": (8, 4, 0, 4, 128, 128), "d64": (4, 2, 0, 4, 64, 64), "d64-g32": (4, 2, 0, 2, 64, 32)}


def config(kvq, form, batch, heads, max_pages, residual=0):
    kb, vb, axis, q_heads, D, group = FORMS[form]
    return kvq.make_config(batch, heads * q_heads, heads, D, kb, vb, group, group, axis, "bf16", PAGE * max_pages, residual)


@pytest.mark.parametrize("form,heads,pages", [
    ("channel", 10, [95, 63, 37, 57, 58, 70, 35, 110, 117, 93]),
    ("token", 8, [472, 1024]),
    ("token", 1, [3000, 900, 5]),
    ("wide pages", 8, [472, 1024]),
    ("d64", 8, [31, 0, 1, 250, 33]),
    ("d64-g32", 3, [1, 1, 700, 2])])
def test_long_streams_of_uneven_batches(kvq, form, heads, pages):
    check_split(kvq, config(kvq, form, len(pages), heads, max(pages)), pages)


@pytest.mark.parametrize("form", list(FORMS))
def test_random_uneven_batches(kvq, form):
    rng, weighted = random.Random(form), 0
    for _ in range(1500):
        heads, batch = rng.randint(1, 10), rng.randint(1, 24)
        top = rng.choice([4, 40, 150, 1200])
        pages = [rng.choice([0, 1, rng.randint(1, top), rng.randint(top // 2, top)]) for _ in range(batch)]
        residual = rng.choice([0, 0, 128]) if form != "channel" else 0
        if residual:            # whole blocks of the window are pages: no incomplete ones
            pages = [max(0, p - 1) for p in pages]
            cfg = config(kvq, form, batch, heads, top, residual)
            slots, _, starts, parts = kvq.kvq_debug_decode_plan(cfg, [PAGE * p + 5 if p else 0 for p in pages])
            assert parts[:, 1].max() <= slots and (sum(pages) == 0 or starts[-1] == heads * sum(pages))
        elif sum(pages):
            weighted += check_split(kvq, config(kvq, form, batch, heads, top), pages)
    assert (weighted > 0) == (form != "wide pages")         # the weighted split is among what was checked


@pytest.mark.parametrize("form,batch,heads", [("d64", 14, 8), ("d64", 16, 8), ("d64-g32", 130, 1), ("d64", 64, 8)])
def test_shares_of_many_streams_hold_pages(kvq, form, batch, heads):
    """head_dim 64, more than 64 streams of 4,096 tokens: a share is not swallowed by the gap in front of a stream, and the largest is
    not far from the mean."""
    starts = kvq.kvq_debug_decode_plan(config(kvq, form, batch, heads, 32), [PAGE * 32] * batch)[2]
    pages = np.diff(starts)
    assert pages.max() <= 1.55 * pages.mean() and (pages == 0).sum() <= len(pages) // 20


def test_empty_caches_have_no_split(kvq):
    slots, weighted, starts, parts = kvq.kvq_debug_decode_plan(config(kvq, "token", 3, 2, 4), [0, 0, 0])
    assert len(starts) == 1 and not parts.any() and not weighted


def test_a_split_is_refused_where_the_kernel_does_not_serve(kvq):
    with pytest.raises(kvq.KvqError) as e:
        kvq.kvq_debug_decode_plan(kvq.make_config(1, 4, 1, 128, 16, 16, 128, 128, 0, "bf16", 256), [5])
    assert e.value.code == -2


@pytest.mark.parametrize("form", [f for f in FORMS if f != "channel"])
def test_windows_are_taken_by_one_cta_that_is_counted(kvq, form):
    """A stream's residual window is taken by the CTA with its first page, or by the first one whose share lies in the gap in front of
    it: an empty share whose cursor is the stream's first page.  The CTAs that are waited for are those with pages and that one."""
    rng, in_gaps, with_pages = random.Random(form), 0, 0
    for _ in range(800):
        heads, batch = rng.randint(1, 10), rng.randint(1, 24)
        top = rng.choice([1, 4, 40, 150, 1200])
        R = rng.choice([64, 128])
        lens = [rng.choice([0, R, rng.randint(1, R - 1), rng.randint(1, PAGE * top), R * rng.randint(1, max(1, PAGE * top // R))]) for _ in range(batch)]
        cfg = config(kvq, form, batch, heads, top, R)
        starts, parts = kvq.kvq_debug_decode_plan(cfg, lens)[2:]
        cursors, windows = kvq.kvq_debug_decode_cursors(cfg, lens), kvq.kvq_debug_decode_windows(cfg, lens)
        empty = {}
        for c, cursor in enumerate(cursors.tolist()):
            if starts[c] == starts[c + 1]:
                empty.setdefault(tuple(cursor), []).append(c)
        for b, n in enumerate(lens):
            for h in range(heads):
                (first, k), (taker, counted) = parts[b * heads + h], windows[b * heads + h]
                if n < R or n % R == 0:
                    assert taker == -1 and counted == (k if n >= R else 0)
                elif taker == first:
                    assert counted == k and (b, h, 0) not in empty
                    with_pages += 1
                else:
                    assert counted == k + 1 and taker == min(empty[b, h, 0]) and taker < first
                    in_gaps += 1
    assert with_pages > 0 and (in_gaps > 0) == (form != "wide pages")
