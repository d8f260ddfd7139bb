"""surrogate_infer with a workspace at an 8-byte boundary that is not a 16-byte one: the feature rows are stored by
words there. With the mma.sync forward the results equal those of an aligned workspace bit for bit; the fused
forward reads the rows through tensor maps, which such rows do not allow, and the call returns that error."""

import ctypes as C

import numpy as np
import pytest

from workloads import archs, gen
from workloads import mlp as L

pytestmark = pytest.mark.gpu


def infer(s, shift, n=90, k=7):
    import torch

    import paper_1701_08547_gb300 as T
    from paper_1701_08547_gb300 import native

    d = gen.descriptors(n, 21, "uneven")
    d["space_mask"][::4] = np.uint64(gen.mask_bits([3, 5, 30], [2], [0, 7], [1]))
    off = gen.point_offsets(d)
    dd = T.descs_to_device(d)
    nbytes = s.L.surrogate_infer_workspace_bytes(s.members, n, k)
    ws = torch.zeros(nbytes + 16, dtype=torch.uint8, device="cuda")[shift:shift + nbytes]
    assert ws.data_ptr() % 16 == shift
    idx = torch.empty((n, k), dtype=torch.int32, device="cuda")
    val = torch.empty((n, k), dtype=torch.float32, device="cuda")
    fb = torch.empty(n, dtype=torch.uint8, device="cuda")
    a, x = native.make_arch(archs.arch("sm_103")), native.make_axes(gen.axes())
    native.check(s.L.surrogate_infer(s.h, C.byref(a), C.byref(x), dd.data_ptr(), n, off.ctypes.data, k, 0.05,
                                     idx.data_ptr(), val.data_ptr(), fb.data_ptr(), ws.data_ptr(), nbytes, None))
    return [t.cpu().numpy() for t in (idx, val, fb)]


@pytest.fixture
def sur():
    from paper_1701_08547_gb300.surrogate import Surrogate

    s = Surrogate(members=2, batch=1024)
    s.set_params(L.init_params(2))
    return s


def test_rows_by_words(sur):
    sur.set_forward_mode(sur.FWD_LAYERED)
    sur.use_tcgen05(False)
    for got, want in zip(infer(sur, 8), infer(sur, 0)):
        assert np.array_equal(got, want)


def test_fused_forward_refuses(sur):
    from paper_1701_08547_gb300 import TuneError

    want = infer(sur, 0)
    with pytest.raises(TuneError, match="cuTensorMapEncodeTiled"):
        infer(sur, 8)
    for got, w in zip(infer(sur, 0), want):
        assert np.array_equal(got, w)
