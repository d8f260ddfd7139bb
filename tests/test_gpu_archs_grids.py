"""tune_eval_archs over the ways its rows' launches are laid out: rows side by side (fewer than two descriptors per warp of
a full grid), and full grids whose CTAs start in the places that the row before leaves, with several descriptors per
warp; by CTA-owned descriptors and by work queues. Each row equals tune_eval with that row bit for bit, and a training
step that follows on the stream, whose kernels start early, gives what it gives by itself."""

import numpy as np
import pytest

from workloads import archs, gen
from workloads import mlp as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, 0x10 | (1 << 8), 0x10 | (4 << 8)])
@pytest.mark.parametrize("rows", [2, 5, 8])
@pytest.mark.parametrize("n", [1, 5000, 9700, 9800, 30000])
def test_rows_equal_single_calls(n, rows, flags):
    import torch

    import paper_1701_08547_gb300 as T

    names = (list(archs.ARCHS) * 2)[:rows]
    ax = gen.axes()
    d = gen.descriptors(n, 8, "dense128")
    d["space_mask"][::5] = gen.descriptors(n, 8, "uneven")["space_mask"][::5]
    dd = T.descs_to_device(d)
    idx, cost = T.tune_eval_archs([archs.arch(x) for x in names], ax, dd, 6, flags=flags)
    for i, x in enumerate(names):
        one = T.tune_eval(archs.arch(x), ax, dd, 6)
        assert torch.equal(idx[i], one[0]), x
        assert torch.equal(cost[i].view(torch.int32), one[1].view(torch.int32)), x


def test_training_step_after_a_sweep():
    import torch

    import paper_1701_08547_gb300 as T
    from paper_1701_08547_gb300.surrogate import Surrogate

    g = torch.Generator(device="cuda").manual_seed(4)
    feats = torch.randn((8192, 64), generator=g, device="cuda").bfloat16()
    labels = torch.randn(8192, generator=g, device="cuda")
    rows, ax = [archs.arch(x) for x in archs.ARCHS], gen.axes()
    dd = T.descs_to_device(gen.descriptors(20000, 8, "dense128"))
    out = []
    for sweep in (False, True):
        s = Surrogate(members=5, batch=8192)
        s.set_params(L.init_params(5))
        for _ in range(3):
            if sweep:
                T.tune_eval_archs(rows, ax, dd, 6)
            s.train_step(feats, labels)
        out.append(s.get(s.GET_PARAMS))
        s.check()
    assert np.array_equal(out[0], out[1])
