"""Mini-batch steps of the proposal's training against the FP64 oracle: batches
that leave a remainder of a 32-row tile and of the epoch, one that spans more
tiles than blocks, and the order of the rows.

Each Adam step moves a weight by at most about lr; the FP32 gradient's error
(1e-5 of its scale) can flip the sign of an entry that is zero in exact
arithmetic, so all but a thousandth of the weights are held to 1e-5 and the
rest to lr per step.  The sum over the tiles has a fixed order: two runs agree
bit for bit.
"""
import math

import numpy as np
import pytest

from oracle import mlp_oracle as M

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(97, 97), (200, 33), (1000, 321), (24001, 12000)])
def test_minibatch_steps_match_oracle(n, batch):
    from paper_1705_02876_gb300 import build, kf
    build.build()
    ctx = kf.Context(0)
    rng = np.random.default_rng(n)
    X = rng.normal(size=(n, 12)).astype(np.float32)
    y = (X[:, 0] - X[:, 2] + 0.3 * rng.normal(size=n) > 0).astype(np.float32)
    w = M.init_params(rng).astype(np.float32)
    cu = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    got = []
    for _ in range(2):
        wt = cu(w)
        loss = kf.proposal_train(ctx, wt, cu(X), cu(y), epochs=2, batch=batch, lr=1e-3)
        got.append((wt.cpu().numpy(), loss))
    assert np.array_equal(got[0][0], got[1][0]) and got[0][1] == got[1][1]
    p = w.astype(np.float64)
    m, v, t, P = np.zeros_like(p), np.zeros_like(p), 0, 1000003
    while math.gcd(P, n) != 1:
        P += 2
    for ep in range(2):
        order = (np.arange(n) * P + ep * 7919 % n) % n
        total = 0.0
        for a in range(0, n, batch):
            i = order[a:a + batch]
            total += M.loss(p, X[i], y[i]) * len(i)
            t += 1
            p, m, v = M.adam_step(p, M.backward(p, X[i], y[i]), m, v, t, lr=1e-3)
        assert abs(got[0][1][ep] - total / n) <= 1e-4 * total / n
    d = np.abs(got[0][0] - p)
    assert np.quantile(d, 0.999) <= 1e-5 and d.max() <= 1e-3 * t
    ctx.close()
