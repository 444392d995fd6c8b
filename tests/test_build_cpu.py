"""The host Bi-CSR builder against a plain numpy construction, at sizes on both
sides of its one-thread limit and with rows of very different lengths."""
import numpy as np
import pytest


def _reference(n, tails, heads, caps):
    keep = tails != heads
    pairs = np.unique(np.concatenate([tails[keep] * n + heads[keep], heads[keep] * n + tails[keep]]))
    u, v = pairs // n, pairs % n
    row = np.concatenate([[0], np.cumsum(np.bincount(u, minlength=n))])
    arc = np.where(keep, np.searchsorted(pairs, tails * n + heads), -1)
    cap = np.bincount(arc[keep], weights=caps[keep], minlength=len(pairs)).astype(np.int64)
    mult = np.bincount(arc[keep], minlength=len(pairs))
    rev = np.searchsorted(pairs, v * n + u)
    both = (mult + mult[rev]).max() if len(pairs) else 1
    return row, v, rev, cap, arc, (2**31 - 1) // max(1, both)


@pytest.mark.parametrize("n,m,star", [(2, 0, 0), (3, 5, 0), (50, 700, 0), (1000, 16_384, 0), (1001, 70_001, 0),
                                      (5000, 100_000, 3), (40_000, 300_000, 1)])
def test_builder_matches_numpy(n, m, star):
    from paper_2511_05895_gb300 import bicsr_host
    rng = np.random.default_rng(n + m)
    tails = np.sort(rng.integers(0, n, m))
    heads = rng.integers(0, n, m)          # self-loops, parallel and antiparallel edges among them
    if star:                               # a few vertices that most edges enter
        heads = np.where(rng.random(m) < 0.6, rng.integers(0, star, m), heads)
    caps = rng.integers(0, 1000, m)
    row_ptr = np.concatenate([[0], np.cumsum(np.bincount(tails, minlength=n))])
    got = bicsr_host(n, row_ptr, heads, caps, 0, n - 1)
    row, head, rev, cap, arc, limit = _reference(n, tails, heads, caps)
    np.testing.assert_array_equal(got["arc_row"], row)
    np.testing.assert_array_equal(got["head"], head)
    np.testing.assert_array_equal(got["rev"], rev)
    np.testing.assert_array_equal(got["cap"], cap)
    np.testing.assert_array_equal(got["arc_of_edge"], arc)
    assert got["cap_limit"] == limit
