"""tune_topk over short segments: up to 32 scores (one per lane, no batch), few candidates (inserted one by one) and more
(sorted and merged), at every alignment of the segments' first score; a warp, a CTA and a cluster per segment. Indices
and scores equal the oracle's."""

import numpy as np
import pytest

from test_gpu_topk import check, dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("k", [1, 2, 8, 9, 16])
@pytest.mark.parametrize("n", [60, 600, 7000])
def test_short_segments(dev, oracle, n, k):  # noqa: F811
    rng = np.random.default_rng(100 * n + k)
    lens = np.resize(np.arange(72), n)  # 0 .. 71, so that starts take every alignment
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    s = np.round(rng.standard_normal(int(off[-1])) * 4).astype(np.float32)
    s[::5] = rng.choice(np.array([np.nan, np.inf, -np.inf, -0.0, 3.4028235e38], np.float32), s[::5].size)
    check(dev, oracle, s, off, k)


@pytest.mark.parametrize("k", [1, 7, 8, 9])
def test_falling_and_rising(dev, oracle, k):  # noqa: F811
    """Every score enters the list, or none after the first k."""
    off = np.arange(0, 40 * 33 + 1, 33, dtype=np.int64)
    s = np.arange(int(off[-1]), dtype=np.float32)
    check(dev, oracle, s, off, k)
    check(dev, oracle, -s, off, k)
