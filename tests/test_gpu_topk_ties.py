"""tune_topk where scores repeat or fall: many candidates in a batch, taken group by group (128 consecutive scores) with
the bound dropping ties in between, and batches with a bound of their own. The lowest indices win among equal scores, on
the paths of a warp, a CTA and a cluster per segment. Indices and scores equal the oracle's."""

import numpy as np
import pytest

from test_gpu_topk import check, dev  # noqa: F401

pytestmark = pytest.mark.gpu

LENGTHS = [65, 127, 128, 129, 200, 384, 511, 512, 513, 640, 1024, 1540, 5000]


@pytest.mark.parametrize("k", [1, 5, 16])
@pytest.mark.parametrize("levels", [1, 2, 3, 9])
@pytest.mark.parametrize("n", [13, 300, 2000])
def test_repeated_scores(dev, oracle, n, levels, k):  # noqa: F811
    rng = np.random.default_rng(1000 * n + 10 * levels + k)
    lens = np.resize(LENGTHS, n)
    off = np.concatenate([[3], 3 + np.cumsum(lens)]).astype(np.int64)
    s = rng.integers(0, levels, int(off[-1])).astype(np.float32)
    s[rng.integers(0, s.size, n // 3)] = -1.0  # a rare smaller one
    check(dev, oracle, s, off, k)


@pytest.mark.parametrize("k", [1, 5, 16])
@pytest.mark.parametrize("n", [13, 700])
def test_falling_with_ties(dev, oracle, n, k):  # noqa: F811
    lens = np.resize(LENGTHS, n)
    off = np.concatenate([[1], 1 + np.cumsum(lens)]).astype(np.int64)
    s = np.floor(np.arange(int(off[-1]), 0, -1) / (3.0 * (1 + np.arange(int(off[-1])) % 2))).astype(np.float32)
    check(dev, oracle, s, off, k)
