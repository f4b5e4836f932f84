"""The batched selection's re-scoring by unit sums (K = 2, 3, 4, 6, 8) and in FP64
(other K), with one warp, several warps and several rounds of candidates per
problem (top_m 1 to 16), at rows around a warp's 32.  Every candidate is
selected (S = top_m), so the winner is the oracle's.  The sums are exact to
2^-60 and end in FP64: 1e-13 relative per unit of |V^H z|^2 / (n sum |V_i|^2)
> 1e-2, so 1e-11."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 2, 3, 4, 5, 8, 9, 16])
def test_winner(m):
    probs, refs = [], []
    for p, (n, r, K) in enumerate([(1, 1, 2), (31, 2, 3), (33, 3, 4), (64, 4, 6), (255, 5, 8), (257, 6, 3), (513, 7, 2),
                                   (1000, 8, 8), (300, 3, 5), (300, 2, 11), (4001, 4, 8)]):
        V = inputs.factor(n, r, seed=p, dtype=np.complex64)
        C = inputs.directions(m, r, seed=100 * m + p, dtype=np.complex64)
        refs.append(oracle.score(V.astype(np.complex128), K, C.astype(np.complex128)))
        probs.append(dict(V=torch.from_numpy(V).cuda(), K=K, C=torch.from_numpy(C).cuda()))
    plan = lrq.BatchedPlan(probs, top_m=m)
    plan.run()
    torch.cuda.synchronize()
    lrq.check_status(plan.status)
    for p, ref in enumerate(refs):
        i, f = int(plan.best_idx[p].item()), float(plan.best_f[p].item())
        assert abs(f - ref[i]) <= 1e-11 * ref[i]
        assert ref[i] >= ref.max() * (1 - 1e-11)
