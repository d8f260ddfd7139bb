"""The head's backward pass where the training forward does part of it.

With more 128-row units than SMs and a remainder, the CTAs with one unit less form the head's
slices of their own units; a one-member handle of the same batch has at most as many units as SMs,
so there the separate kernel forms them all. Both run the same arithmetic in the same order, and
no other part of a step mixes members, so losses and all gradients have to be equal bit for bit."""

import numpy as np
import pytest

from workloads import mlp as L

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("members,batch,n", [
    (5, 8192, 8192),   # 320 units: two or three per CTA of 152
    (3, 8192, 8191),   # 192 units, the last row not labelled
    (16, 1280, 1200),  # 160 units, the last tile half labelled
    (2, 9728, 9728),   # 152 units: one per CTA, nothing split off
    (4, 9728, 9600),   # 300 units
])
def test_gradients_equal_one_member_at_a_time(members, batch, n):
    import torch

    from paper_1701_08547_gb300.surrogate import Surrogate

    rng = np.random.default_rng(members)
    x = rng.uniform(-1, 1, (n, L.IN)).astype(np.float32)
    x[:, 48:] = 0
    feats = torch.from_numpy(x).cuda().bfloat16()
    labels = torch.from_numpy(rng.normal(size=n).astype(np.float32)).cuda()
    flat = L.init_params(members, list(range(3, 3 + members)))
    s = Surrogate(members=members, batch=batch)
    s.set_params(flat)
    s.train_step(feats, labels, apply_update=False)
    s.check()
    grads, loss = s.get(s.GET_GRADS).reshape(members, -1), s.get(s.GET_LOSS)
    one = Surrogate(members=1, batch=batch)
    for m in range(members):
        one.set_params(np.asarray(flat).reshape(members, -1)[m])
        one.train_step(feats, labels, apply_update=False)
        one.check()
        assert one.get(one.GET_LOSS)[0] == loss[m]
        g = one.get(one.GET_GRADS)
        assert np.any(g) and np.array_equal(g.view(np.uint32), grads[m].view(np.uint32))
