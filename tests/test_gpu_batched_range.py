"""The batched re-scoring at the ends of FP32's range, where its FP32 sums
overflow or its projections underflow: a power of two on V scales every value by
its square exactly and changes no decision, so the winner is that of V of
ordinary size (every candidate is selected)."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("exp2", [-146, -130, 118, 122])
def test_scaled_factor(exp2):
    probs, scaled = [], []
    for p, (n, r, K) in enumerate([(700, 1, 2), (1500, 2, 3), (300, 3, 4), (900, 4, 6), (700, 6, 8), (300, 8, 3)]):
        # small integers, so that the scaled V is exact down to 2^-149
        g = np.random.Generator(np.random.PCG64(p))
        V = (g.integers(-7, 8, (n, r)) + 1j * g.integers(-7, 8, (n, r)) + 20 * (g.random((n, r)) < 0.05)).astype(np.complex64)
        C = torch.from_numpy(inputs.directions(16, r, seed=p, dtype=np.complex64)).cuda()
        for q, e in ((probs, 0), (scaled, exp2)):
            W = torch.from_numpy(np.ldexp(V.view(np.float32), e).view(np.complex64)).cuda()
            q.append(dict(V=W, K=K, C=C))
    res = []
    for q in (probs, scaled):
        plan = lrq.BatchedPlan(q, top_m=16)
        plan.run()
        torch.cuda.synchronize()
        lrq.check_status(plan.status)
        res.append((plan.best_f.cpu().numpy(), plan.best_idx.cpu().numpy()))
    assert np.array_equal(res[0][1], res[1][1])
    assert np.allclose(res[1][0], np.ldexp(res[0][0], 2 * exp2), rtol=1e-12, atol=0)
