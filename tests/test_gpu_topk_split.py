"""tune_topk where the split of the work changes: segment counts around the limits between clusters of 8, 4,
2 and 1 CTAs per segment and a warp per segment, segment lengths around the batch (512 scores), a warp's and
a CTA's share, and the length from which a CTA's warps share a segment, with ties across every boundary.
Selection is exact, so indices and scores equal the oracle's."""

import numpy as np
import pytest

from test_gpu_topk import check, dev  # noqa: F401

pytestmark = pytest.mark.gpu

EDGES = [0, 1, 2, 3, 4, 5, 31, 33, 127, 128, 129, 511, 512, 513, 515, 4095, 4097, 32767, 32768, 32773, 40001]


def segments(n, seed):
    rng = np.random.default_rng(seed)
    lens = rng.permutation(np.concatenate([EDGES[::-1], rng.integers(0, 700, n)])[:n])  # (never all empty)
    off = np.zeros(n + 1, np.int64)
    off[1:] = np.cumsum(lens)
    return rng, off


@pytest.mark.parametrize("k", [1, 10, 16])
@pytest.mark.parametrize("n", [1, 20, 76, 77, 152, 153, 304, 305, 608, 609, 1300, 5000])
def test_split(dev, oracle, n, k):  # noqa: F811
    rng, off = segments(n, 100 * n + k)
    s = np.round(np.exp(rng.uniform(-2, 6, int(off[-1])))).astype(np.float32) - 3.0  # ties, zeros, negatives
    check(dev, oracle, s, off, k)


@pytest.mark.parametrize("n", [2, 100, 700])
@pytest.mark.parametrize("value", [0.0, -0.0, 7.0, -np.inf, 3.4028235e38])
def test_equal_scores(dev, oracle, n, value):  # noqa: F811
    _, off = segments(max(n, len(EDGES)), n)
    check(dev, oracle, np.full(int(off[-1]), value, np.float32), off, 12)


@pytest.mark.parametrize("n", [5, 700])
def test_worst_order(dev, oracle, n):  # noqa: F811
    """Every score below all before it: each enters the list."""
    off = np.arange(n + 1, dtype=np.int64) * (40000 if n < 10 else 1500)
    s = np.arange(int(off[-1]), 0, -1).astype(np.float32)
    check(dev, oracle, s, off, 16)
