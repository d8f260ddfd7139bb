"""tune_eval's per-point output where its stretches and 16-byte stores begin and end: odd space sizes and
offsets, arrays whose alignments agree or not, arrays left out, and both register-allocation modes. B* and W*
are integers and costs follow the library's FP32 operation order, so everything equals the oracle bit for bit,
and nothing outside the kernels' points is written."""

import numpy as np
import pytest

from workloads import archs, gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    import torch

    from paper_1701_08547_gb300 import build

    build.build()
    assert torch.cuda.is_available()
    return torch.device("cuda:0")


def kernels():
    """The whole space, single points, and odd subsets of every axis; one r0 = 0 (no register limit)."""
    d = gen.descriptors(48, 31, "uneven")
    d["space_mask"][:6] = [gen.MASK_DENSE, gen.mask_bits([3], [2], [1], [0]), gen.mask_bits(range(32), [0], [7], [3]),
                           gen.mask_bits([0], range(16), range(8), range(4)), gen.mask_bits(range(31), range(15), [0], [1]),
                           gen.mask_bits(range(11), [5, 9, 12], range(7), [0, 1, 3])]
    d["r0"][7] = 0
    d["s0"][8] = 300000  # more than a block may have: no valid point
    return d


@pytest.mark.parametrize("shift", [(0, 0, 0), (1, 1, 1), (3, 3, 3), (0, 1, 2), (2, None, 2), (None, None, 1), (0, 3, None)])
@pytest.mark.parametrize("arch", ["sm_103", "sm_20"])
@pytest.mark.parametrize("gap", [0, 1, 5])
def test_points(dev, oracle, arch, shift, gap):
    import torch

    import paper_1701_08547_gb300 as T

    a, ax, d = archs.arch(arch), gen.axes(), kernels()
    sizes = gen.space_sizes(d)
    off = np.zeros(len(d) + 1, np.int64)
    np.cumsum(sizes + gap, out=off[1:])
    room = int(off[-1]) + 16
    pts = [None if s is None else torch.full((room + s,), -7, dtype=t, device=dev)[s:]
           for s, t in zip(shift, (torch.int32, torch.int32, torch.float32))]
    idx, cost = T.tune_eval(a, ax, T.descs_to_device(d, dev), 10, flags=T.TUNE_EMIT_POINTS, pt_blocks=pts[0],
                            pt_warps=pts[1], pt_cost=pts[2], pt_offsets=torch.from_numpy(off).to(dev))
    o = oracle.evaluate(a, ax, d, 10, emit=True, offsets=off)
    inside = np.zeros(room, bool)
    for i in range(len(d)):
        inside[off[i]:off[i] + sizes[i]] = True
    for got, want in zip(pts, (o["B"], o["W"], o["cost32"])):
        if got is None:
            continue
        g = got.cpu().numpy()
        assert np.array_equal(g[inside].view(np.uint32), want[inside[:len(want)]].view(np.uint32))
        assert (g[~inside] == -7).all()
    assert np.array_equal(idx.cpu().numpy(), o["idx"])
    assert np.array_equal(cost.cpu().numpy().view(np.uint32), o["cost"].view(np.uint32))
