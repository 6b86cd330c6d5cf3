"""The bound of the k-th smallest key that cuts the rerank's prefixes, both BF16
pre-filters and (with no slack) the selection's tie class (block_kth_bound): its steps
restated on the CPU with the kernel's 32-bit arithmetic.  At least k keys are at or
below the bound; no more than k + slack are, unless they equal the k-th; with distinct
keys and no slack exactly k; and every counter index lies in the counters."""
import numpy as np
import pytest

M32 = 0xFFFFFFFF


def kth_bound(keys, k, slack, nbins):
    lo, hi = int(keys.min()), int(keys.max())
    log2b = nbins.bit_length() - 1
    # 32 - clz(x) is x's bit length
    shift = max((hi - lo).bit_length() - log2b, 0)
    while True:
        inside = keys[(keys >= lo) & (keys <= hi)]
        bins = ((inside - lo) >> shift).astype(np.int64)
        assert bins.size and bins.max() < nbins
        hist = np.bincount(bins, minlength=nbins)
        ends = np.cumsum(hist)
        part = int(np.searchsorted(ends, k))  # the first part whose end reaches k
        count = int(hist[part])
        first = int(ends[part]) - count
        blo = (lo + (part << shift)) & M32
        rest = ((1 << shift) - 1) & M32
        bhi = hi if hi - blo < rest else blo + rest
        assert lo <= blo <= bhi <= hi
        if shift == 0 or first + count - k <= slack:
            return bhi
        k -= first
        lo, hi = blo, bhi
        shift = max(shift - log2b, 0)


def _keys(case, n, rng):
    if case == "distances":      # a query's squared distances: a narrow range of floats
        return (7.0 + rng.random(n)).astype(np.float32).view(np.uint32).astype(np.int64)
    if case == "equal":
        return np.full(n, int(rng.integers(0, M32 + 1)), dtype=np.int64)
    if case == "full":
        x = rng.integers(0, M32 + 1, size=n, dtype=np.int64)
        x[0], x[-1] = 0, M32
        return x
    if case == "outlier":        # all keys but one in one part
        x = rng.integers(1000, 1000 + 4 * n, size=n, dtype=np.int64)
        x[int(rng.integers(n))] = 0x7F800000
        return x
    if case == "ids":            # distinct ids of a tie class
        return rng.permutation(n * 7)[:n].astype(np.int64)
    if case == "ties":
        return rng.choice(rng.integers(0, M32 + 1, size=5), n).astype(np.int64)
    return np.where(rng.random(n) < 0.9, 0, rng.integers(0, 1 << 20, size=n)).astype(np.int64)


@pytest.mark.parametrize("nbins", [256, 512, 2048])
@pytest.mark.parametrize("case", ["distances", "equal", "full", "outlier", "ids", "ties", "zeros"])
def test_kth_bound(case, nbins):
    rng = np.random.default_rng(nbins + len(case))
    for n in (1, 2, 31, 255, 256, 257, nbins - 1, nbins, nbins + 1, 1000, 4096):
        keys = _keys(case, n, rng)
        ordered = np.sort(keys)
        for k in {1, 2, n // 2, n - 1, n, int(rng.integers(1, n + 1))}:
            if not 1 <= k <= n:
                continue
            for slack in (0, 4, k >> 3):
                U = kth_bound(keys, k, slack, nbins)
                kth, under = int(ordered[k - 1]), int((keys <= U).sum())
                assert under >= k and U >= kth and U <= ordered[-1]
                assert under <= k + slack or U == kth
                if slack == 0 and np.unique(keys).size == n:
                    assert under == k
