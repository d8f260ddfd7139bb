"""TUNE_EMIT_POINTS with a single per-point array, where a CTA ranks all its descriptors in one turn: around one and
eight descriptors per CTA of a full grid, each array alone equals the one written with all three, bit for bit, and
the top-k too."""

import numpy as np
import pytest

from workloads import archs, gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 9, 607, 608, 609, 1217, 4863, 4865, 6000])
def test_each_array_alone(n):
    import torch

    import paper_1701_08547_gb300 as T

    a, ax, k = archs.arch("sm_103"), gen.axes(), 3
    d = gen.descriptors(n, 17, "dense128")
    d["space_mask"][::9] = gen.descriptors(n, 17, "uneven")["space_mask"][::9]
    d["space_mask"][n // 2] = np.uint64(gen.MASK_DENSE)
    d["d"][n // 3] = 2.0 if n > 3 else d["d"][n // 3]  # malformed: no points
    off = gen.point_offsets(d)
    dd, po = T.descs_to_device(d), torch.from_numpy(off).cuda()

    def emit(which):
        pts = [torch.full((int(off[-1]),), 7, dtype=t, device="cuda") if i in which else None
               for i, t in enumerate((torch.int32, torch.int32, torch.float32))]
        top = T.tune_eval(a, ax, dd, k, flags=T.TUNE_EMIT_POINTS, pt_blocks=pts[0], pt_warps=pts[1], pt_cost=pts[2],
                          pt_offsets=po)
        return top, pts

    top, pts = emit((0, 1, 2))
    for i in range(3):
        one, alone = emit((i,))
        assert torch.equal(alone[i].view(torch.int32), pts[i].view(torch.int32))
        assert torch.equal(one[0], top[0]) and torch.equal(one[1].view(torch.int32), top[1].view(torch.int32))
