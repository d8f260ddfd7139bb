"""surrogate_infer builds its feature rows per kernel from axis tables; every row has to be
the one tune_features writes for that point.

One member, no fallback, k = 16: infer's scores are exp(prediction) of the k smallest
predictions, so spaces of at most 16 points show all their rows and larger ones their best
16. The same rows through tune_features and forward() give the same predictions to the bit
(one code path); expf of CUDA is within 2 ulp of exp, so the scores agree to 2.4e-7
relative (bound used: 5e-7) where one BF16 step in one feature moves a prediction by
orders of magnitude more."""

import numpy as np
import pytest

from workloads import archs, gen
from workloads import mlp as L

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def dev():
    import torch

    assert torch.cuda.is_available()
    return torch.device("cuda")


def _spaces(ax, rng, n):
    """Masks of sizes 1 .. 16, sizes around 32 and 256, empty spaces and a full one."""
    def bits(m, k):
        return sorted(rng.choice(m, k, replace=False).tolist())

    shapes = [(1, 1, 1, 1), (2, 1, 1, 1), (1, 3, 1, 1), (1, 1, 5, 1), (1, 1, 1, 4), (7, 1, 1, 2), (3, 5, 1, 1),
              (2, 2, 2, 2), (31, 1, 1, 1), (32, 1, 1, 1), (11, 1, 3, 1), (8, 4, 2, 4), (1, 16, 8, 2), (17, 5, 3, 1)]
    nt, ng, nu, nc = (len(ax[c]) for c in "tguc")
    out = []
    for i in range(n):
        if i % 13 == 12:
            out.append(0)
            continue
        t, g, u, c = shapes[i % len(shapes)] if i != n // 2 else (nt, ng, nu, nc)
        out.append(gen.mask_bits(bits(nt, min(t, nt)), bits(ng, min(g, ng)), bits(nu, min(u, nu)),
                                 bits(nc, min(c, nc))))
    return np.array(out, dtype=np.uint64)


@pytest.mark.parametrize("arch,n,seed", [("sm_103", 1, 1), ("sm_103", 61, 2), ("sm_20", 60, 3), ("sm_35", 60, 4),
                                         ("sm_103", 3000, 5)])
def test_infer_rows_equal_tune_features(dev, arch, n, seed):
    import torch

    import paper_1701_08547_gb300 as T
    from paper_1701_08547_gb300.surrogate import Surrogate

    rng = np.random.default_rng(seed)
    a, ax = archs.arch(arch), gen.axes()
    if seed % 2 == 0:  # axes off the warp size and off the powers of two
        ax = dict(ax, t=[1 + 33 * i for i in range(32)][:31], g=[3 ** i for i in range(10)], c=[0, 33, 90])
    d = gen.descriptors(n, 40 + seed, "dense128")
    d["space_mask"] = _spaces(ax, rng, n)
    d["r0"][::7] = 250
    d["s0"][::5] = rng.integers(0, 60000, len(d["s0"][::5]))
    off = gen.point_offsets(d)
    total, k = int(off[-1]), 16
    s = Surrogate(members=1, batch=1024)
    s.set_params(L.init_params(1, [seed]))
    dd = T.descs_to_device(d, dev)
    idx, val, fb = s.infer(a, ax, dd, off, k, thresh=1e30)
    idx, val = idx.cpu().numpy(), val.cpu().numpy()
    assert not fb.cpu().numpy().any()

    kern = np.repeat(np.arange(n), np.diff(off))
    point = np.arange(total) - off[kern]
    feats = T.tune_features(a, ax, dd, torch.from_numpy(kern).to(dev), torch.from_numpy(point.astype(np.int32)).to(dev))
    pred = s.forward(feats)[0].cpu().numpy().astype(np.float64)
    valid = feats[:, 29].float().cpu().numpy() > 0
    want = np.where(valid, np.exp(pred), np.inf)
    for j in range(n):
        w = want[off[j]:off[j + 1]]
        m = min(k, int(np.isfinite(w).sum()))
        assert np.all(idx[j, m:] == -1) and np.all(np.isinf(val[j, m:]))
        assert len(set(idx[j, :m].tolist())) == m
        np.testing.assert_allclose(val[j, :m], w[idx[j, :m]], rtol=5e-7)
        np.testing.assert_allclose(val[j, :m], np.sort(w)[:m], rtol=5e-7)
