"""tune_topk with more segments than resident CTAs: a CTA owns 2, 4 or 8 consecutive segments, by their number, and its
warps share those longer than 32,768 scores at the end, one after the other (several per CTA here, in alternating
buffers). Segment counts on both sides of each line; indices and scores equal the oracle's."""

import numpy as np
import pytest

from test_gpu_topk import check, dev  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [609, 610, 1215, 1216, 1217, 2431, 2432, 2433, 4863, 4864, 4865, 9729])
def test_segment_counts(dev, oracle, n):  # noqa: F811
    rng = np.random.default_rng(n)
    lens = rng.integers(0, 600, n)
    lens[rng.integers(0, n, 6)] = rng.integers(30000, 36000, 6)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    check(dev, oracle, np.round(rng.exponential(50, int(off[-1]))).astype(np.float32), off, 11)


@pytest.mark.parametrize("n,every", [(700, 1), (5000, 7)])
def test_many_long_segments(dev, oracle, n, every):  # noqa: F811
    rng = np.random.default_rng(n)
    lens = rng.integers(0, 100, n)
    lens[::every] = 33000 + rng.integers(0, 9, lens[::every].size)
    off = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    s = rng.standard_normal(int(off[-1]), dtype=np.float32)
    s[::3] = np.round(s[::3])  # ties across the warps' parts
    check(dev, oracle, s, off, 16)
