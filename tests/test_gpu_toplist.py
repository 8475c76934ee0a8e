"""Toplist forms against a sort: direct ranking (up to 8192 values), groups with
a pivot, and the radix select that takes over when more values reach the pivot
than the candidate buffer (20480) holds.  Indices and values are exact."""
import numpy as np
import pytest
import torch

import paper_0904_1826_gb300 as lib

pytestmark = pytest.mark.gpu


def _check(v, k, off=0):
    buf = torch.empty(len(v) + off, dtype=torch.float32, device="cuda")
    buf[off:] = torch.from_numpy(v).cuda()
    idx = torch.full((k,), -1, dtype=torch.int64, device="cuda")
    val = torch.full((k,), -1.0, dtype=torch.float32, device="cuda")
    lib.fstat_toplist_noalloc(buf[off:], k, idx, val)
    want = np.lexsort((np.arange(len(v)), -v))[:k]
    np.testing.assert_array_equal(idx.cpu().numpy(), want)
    np.testing.assert_array_equal(val.cpu().numpy(), v[want])


def _values(kind, n, seed):
    r = np.random.default_rng(seed)
    if kind == "chi2":
        return r.chisquare(4, n).astype(np.float32)
    if kind == "ties":      # few levels: many equal values around the threshold
        return r.integers(0, 50, n).astype(np.float32)
    if kind == "equal":
        return np.full(n, 3.25, np.float32)
    if kind == "zero":
        return np.zeros(n, np.float32)
    if kind == "rising":
        return np.arange(n, dtype=np.float32)
    if kind == "falling":
        return np.arange(n, 0, -1).astype(np.float32)
    if kind == "run":       # the largest values side by side, in few groups
        v = r.chisquare(4, n).astype(np.float32)
        v[n // 3:n // 3 + 30000] += 1000.0
        return v
    assert kind == "narrow"  # top 22 bits of the patterns all alike
    return (1.0 + r.integers(0, 900, n) * 2.0 ** -23).astype(np.float32)


@pytest.mark.parametrize("n,k", [(1, 1), (31, 31), (33, 5), (8192, 8192), (8193, 8193), (8195, 1), (20480, 16384),
                                 (20481, 16384), (131072, 1000), (131073, 16384), (1_000_003, 777), (4_194_305, 1000),
                                 (9_000_001, 16384)])
@pytest.mark.parametrize("off", [0, 1, 3])
def test_sizes_and_offsets(n, k, off):
    _check(_values("chi2", n, n + off), k, off)


@pytest.mark.parametrize("kind", ["ties", "equal", "zero", "rising", "falling", "run", "narrow"])
@pytest.mark.parametrize("n,k", [(5000, 300), (60_001, 1000), (2_000_003, 1000), (2_000_003, 16384)])
def test_equal_sorted_and_clustered_values(kind, n, k):
    _check(_values(kind, n, 7), k, 2)


def test_other_calls_between_leave_no_trace():
    """A call that overflowed, then one that does not, then a direct one."""
    for kind, n, k in (("equal", 300_000, 100), ("chi2", 300_000, 100), ("chi2", 700, 20), ("rising", 300_000, 50)):
        _check(_values(kind, n, 3), k)
