"""The merged-list form of the CUDA 3x3x3 median (host-side check of the
generated comparator lists; no GPU): the middle ranks of two sorted lists, and
the median taken from them and a third list, against the median network and
against sorting."""
import numpy as np

from test_median_network import _apply, _gen


def _median(ops, outs, lists):
    w = {}
    for k in range(2):
        for i in range(9):
            w[16 * k + i] = lists[k][:, i].copy()
    w = _apply(ops, w)
    m = [w[o] for o in outs]
    r = m[9]
    for i in range(1, 10):
        r = np.minimum(r, np.maximum(lists[2][:, i - 1], m[9 - i]))
    return m, r


def test_merge_and_median():
    ops, outs = _gen().merge9()
    ops3, out3 = _gen().median3x9()
    rng = np.random.default_rng(5)
    for hi in (2, 3, 30, 65536):
        vals = rng.integers(0, hi, size=(20000, 27))
        lists = [np.sort(vals[:, 9 * k: 9 * k + 9], axis=1) for k in range(3)]
        m, r = _median(ops, outs, lists)
        assert np.array_equal(np.stack(m, 1), np.sort(vals[:, :18], axis=1)[:, 4:14]), hi
        assert np.array_equal(r, np.sort(vals, axis=1)[:, 13]), hi
        w = {16 * k + i: lists[k][:, i].copy() for k in range(3) for i in range(9)}
        assert np.array_equal(r, _apply(ops3, w)[out3]), hi


def test_zero_one():
    # sorted 0-1 lists: a number of zeros, then ones
    ops, outs = _gen().merge9()
    z = np.array([(a, b, c) for a in range(10) for b in range(10) for c in range(10)])
    lists = [(np.arange(9)[None, :] >= z[:, k:k + 1]).astype(int) for k in range(3)]
    m, r = _median(ops, outs, lists)
    for k in range(10):
        assert np.array_equal(m[k], (z[:, 0] + z[:, 1] <= 4 + k).astype(int))
    assert np.array_equal(r, (z.sum(1) < 14).astype(int))
