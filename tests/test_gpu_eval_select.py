"""The ranking pass's walks over grid-size subsets (masks over the increasing order of each B*'s
row), its equal-cost rounds and its numbering of points, against the oracle: indices equal, costs
equal to the bit."""

import numpy as np
import pytest

from workloads import archs, gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    import torch

    assert torch.cuda.is_available()
    return torch.device("cuda")


def _masks(rng, n):
    """Every size of the grid-size set in turn, its members at random; other axes from one value
    to all of them, so that spaces have fewer and more than 32 candidate triples."""
    def bits(m, k):
        return rng.choice(m, k, replace=False).tolist()

    return np.array([gen.mask_bits(bits(32, int(rng.integers(1, 33))), bits(16, 1 + i % 16),
                                   bits(8, int(rng.integers(1, 9))), bits(4, int(rng.integers(1, 5))))
                     for i in range(n)], dtype=np.uint64)


@pytest.mark.parametrize("arch,k,chunk", [("sm_103", 1, 0), ("sm_103", 16, 1), ("sm_20", 5, 2), ("sm_35", 15, 0),
                                          ("sm_60", 10, 1)])
def test_subset_walks_equal_the_oracle(dev, oracle, arch, k, chunk):
    import paper_1701_08547_gb300 as T
    from paper_1701_08547_gb300 import native

    rng = np.random.default_rng(k)
    a, ax = archs.arch(arch), gen.axes()
    d = gen.descriptors(160, 70 + k, "dense128")
    d["space_mask"] = _masks(rng, len(d))
    d["r0"][::9] = 0       # no register limit: tabulated block limits
    d["s0"][::11] = 40000  # few blocks: many invalid points
    for c in range(7):
        d["n"][::13, c] = 0  # every cost 0: ties throughout, walked without the shortcut
    flags = native.TUNE_SCHED_WARP | chunk << 8
    idx, val = T.tune_eval(a, ax, T.descs_to_device(d, dev), k, flags=flags)[:2]
    o = oracle.evaluate(a, ax, d, k)
    assert np.array_equal(idx.cpu().numpy(), o["idx"])
    assert np.array_equal(val.cpu().numpy().view(np.uint32), o["cost"].view(np.uint32))
