"""Neighbour lists from elements: rows of every length around the sorting networks' widths and the
in-block list's length, alike in all rows of a warp or mixed, and more blocks than one pass of the
scan of their totals takes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def build(n, el, max_row):
    import torch

    from paper_2408_02758_gb300 import ftle as F

    rp, ci = F.ftle_csr_from_elements(n, torch.from_numpy(np.ascontiguousarray(el, dtype=np.int32)).cuda(), max_row)
    return rp.cpu().numpy(), ci.cpu().numpy()


def expected(n, el):
    pairs = np.concatenate([el, el[:, ::-1]]).astype(np.int64)
    key = np.unique(pairs[:, 0] * n + pairs[:, 1])
    return np.concatenate([[0], np.cumsum(np.bincount(key // n, minlength=n))]), key % n


@pytest.mark.parametrize("length", [1, 2, 7, 8, 9, 15, 16, 17, 27, 28, 29, 31, 32, 33, 40])
@pytest.mark.parametrize("mixed", [False, True])
def test_row_lengths(length, mixed):
    n, rng = 300, np.random.default_rng(length)
    # a circulant graph: every node has `length` neighbours (an odd one across the ring)
    i = np.arange(n)
    steps = list(range(3, 3 + length // 2)) + ([n // 2] if length % 2 else [])
    el = np.concatenate([np.stack([i, (i + s) % n], 1) for s in steps])
    if mixed:
        el = el[rng.random(len(el)) < 0.6]
    el = np.concatenate([el, el[: len(el) // 3, ::-1]])[rng.permutation(len(el) + len(el) // 3)]
    label = rng.permutation(n)
    el = label[el]
    rp, ci = build(n, el, 2 * length + 3)
    want = expected(n, el)
    assert np.array_equal(rp, want[0]) and np.array_equal(ci, want[1])


@pytest.mark.parametrize("n", [8192 * 128, 8192 * 128 + 1, 2 * 8192 * 128 + 77])
def test_many_blocks(n):
    i = np.arange(n - 1)
    el = np.stack([i, i + 1], 1)
    rp, ci = build(n, el, 4)
    want = expected(n, el)
    assert np.array_equal(rp, want[0]) and np.array_equal(ci, want[1])
