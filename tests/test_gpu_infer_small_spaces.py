"""surrogate_infer over spaces of a few points, around the number of kernels among 32 points up to which their axis tables
are built: every row has to be the one tune_features writes, whichever way it is formed (one member, no fallback, k = 16,
so that a space's scores are exp(prediction) of all its rows; expf of CUDA is within 2 ulp of exp, hence 5e-7)."""

import numpy as np
import pytest

from workloads import archs, gen
from workloads import mlp as L

pytestmark = pytest.mark.gpu


def masks(n, points, rng):
    axis = [1, 1, 1, 1]
    axis[rng.integers(0, 2)] = points
    return np.array([gen.mask_bits(*[sorted(rng.choice(w, k, replace=False).tolist())
                                     for w, k in zip((32, 16, 8, 4), axis)]) for _ in range(n)], dtype=np.uint64)


@pytest.mark.parametrize("points", [1, 2, 5, 6, 7, 8, 10, 11, 16])
def test_small_spaces(points):
    import torch

    import paper_1701_08547_gb300 as T
    from paper_1701_08547_gb300.surrogate import Surrogate

    n, k = 211, 16
    rng = np.random.default_rng(points)
    a, ax = archs.arch("sm_35" if points % 2 else "sm_103"), gen.axes()
    d = gen.descriptors(n, 60 + points, "dense128")
    d["space_mask"] = masks(n, points, rng)
    d["space_mask"][::17] = 0
    d["space_mask"][n // 2] = np.uint64(gen.MASK_DENSE128)  # and back to tables
    d["r0"][::5], d["s0"][::7] = 250, 60000
    off = gen.point_offsets(d)
    s = Surrogate(members=1, batch=1024)
    s.set_params(L.init_params(1))
    dd = T.descs_to_device(d)
    idx, val, _ = [t.cpu().numpy() for t in s.infer(a, ax, dd, off, k, thresh=1e30)]
    kern = np.repeat(np.arange(n), np.diff(off))
    point = (np.arange(int(off[-1])) - off[kern]).astype(np.int32)
    feats = T.tune_features(a, ax, dd, torch.from_numpy(kern).cuda(), torch.from_numpy(point).cuda())
    pred = s.forward(feats)[0].double().cpu().numpy()
    want = np.where(feats[:, 29].float().cpu().numpy() > 0, np.exp(pred), np.inf)
    for j in range(n):
        w = want[off[j]:off[j + 1]]
        m = min(k, int(np.isfinite(w).sum()))
        assert np.all(idx[j, m:] == -1) and len(set(idx[j, :m].tolist())) == m
        np.testing.assert_allclose(val[j, :m], w[idx[j, :m]], rtol=5e-7)
        np.testing.assert_allclose(val[j, :m], np.sort(w)[:m], rtol=5e-7)


def test_malformed_among_small_spaces():
    import paper_1701_08547_gb300 as T
    from paper_1701_08547_gb300.surrogate import Surrogate

    d = gen.descriptors(100, 3, "dense128")
    d["space_mask"] = masks(100, 1, np.random.default_rng(1))
    d["d"][41] = 2.0
    s = Surrogate(members=1, batch=1024)
    s.set_params(L.init_params(1))
    with pytest.raises(T.TuneError, match="malformed"):
        s.infer(archs.arch("sm_103"), gen.axes(), T.descs_to_device(d), gen.point_offsets(d), 3)
