"""A workspace may begin at any 4-byte boundary of a buffer, as a program that carves its memory by itself gives it:
the queue counters (64-bit) of the emitting pass, the work queue and the architecture sweep are placed at an 8-byte
boundary of the header. Results equal those of an aligned workspace bit for bit."""

import numpy as np
import pytest

from workloads import archs, gen

pytestmark = pytest.mark.gpu

TYPES = ("int32", "int32", "float32")


def run(offset):
    import torch

    import paper_1701_08547_gb300 as T

    ax, k = gen.axes(), 4
    a = archs.arch("sm_103")
    d = gen.descriptors(300, 11, "uneven")
    off = gen.point_offsets(d)
    dd, po = T.descs_to_device(d), torch.from_numpy(off).cuda()
    buf = torch.full((512,), 0xff, dtype=torch.uint8, device="cuda")
    ws = buf[offset:offset + 256]
    assert ws.data_ptr() % 8 == offset % 8
    pts = [torch.full((int(off[-1]),), 7, dtype=getattr(torch, t), device="cuda") for t in TYPES]
    out = list(T.tune_eval(a, ax, dd, k, flags=T.TUNE_EMIT_POINTS, pt_blocks=pts[0], pt_warps=pts[1], pt_cost=pts[2],
                           pt_offsets=po, workspace_buf=ws))
    T.tune_check(ws)
    queue = T.TUNE_SCHED_WARP | T.TUNE_SCHED_CHUNK(1)
    out += T.tune_eval(a, ax, dd, k, flags=queue, workspace_buf=ws)
    T.tune_check(ws)
    out += T.tune_eval_archs([archs.arch(n) for n in archs.ARCHS], ax, dd, k, flags=queue, workspace_buf=ws)
    out += T.tune_eval_noalloc(a, ax, dd, k)
    assert buf[:offset].eq(0xff).all() and buf[offset + 256:].eq(0xff).all()
    return [t.cpu().numpy().view(np.uint32) for t in out + pts]


@pytest.mark.parametrize("offset", [4, 8, 12, 60])
def test_workspace_offset(offset):
    for got, want in zip(run(offset), run(0)):
        assert np.array_equal(got, want)
