"""tune_search's table lookups at the edges of what descriptors and rows may hold: no registers, registers beyond
every limit, blocks of 128 warps, per-block register allocation, no shared-memory allocation, single-entry axes,
and budgets that end inside every kind of step. The trajectory is exact, so everything equals the oracle."""

import numpy as np
import pytest

from test_gpu_search import check, dev  # noqa: F401
from workloads import archs, gen

pytestmark = pytest.mark.gpu


def kernels():
    d = gen.descriptors(40, 77, "uneven")
    d["space_mask"][:4] = [gen.MASK_DENSE, gen.mask_bits([31], [15], [7], [3]), gen.mask_bits(range(32), [0], [0], [0]),
                           gen.mask_bits([0], range(16), range(8), range(4))]
    d["r0"][4:8] = [0, 255, 70000, (1 << 24) - 1]
    d["s0"][8:11] = [0, 232448, 1 << 20]
    return d


@pytest.mark.parametrize("arch", ["sm_103", "sm_20", "sm_52"])
@pytest.mark.parametrize("method,budget", [("nelder_mead", 1), ("nelder_mead", 5), ("nelder_mead", 6), ("nelder_mead", 7),
                                           ("nelder_mead", 8), ("nelder_mead", 13), ("nelder_mead", 200), ("random", 1),
                                           ("random", 64)])
def test_edges(dev, oracle, arch, method, budget):  # noqa: F811
    a, ax, d = archs.arch(arch), gen.axes(), kernels()
    ax["t"][30], ax["t"][31] = 3999, 4096  # blocks of 125 and 128 warps
    check(dev, oracle, a, ax, d, method, budget, 5)
