"""A batch whose longest items set its time runs one slot a thread, a batch
that fills the chip four: the same problem gives the same winner and value,
bit for bit, alone and among many, for every rank and alphabet class, and an
exact problem likewise."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


def _run(probs):
    plan = lrq.BatchedPlan(probs, top_m=4)
    plan.run()
    torch.cuda.synchronize()
    lrq.check_status(plan.status)
    return plan.best_f.clone(), plan.best_idx.clone()


@pytest.mark.parametrize("K", [2, 3, 4, 5, 6, 7, 8, 9, 64])
def test_alone_and_among_many(K):
    probs = []
    for r in range(1, 9):
        for n, S in ((1, 4), (127, 65), (129, 1000), (700, 257)):
            V = torch.from_numpy(inputs.factor(n, r, seed=n + r, dtype=np.complex64)).cuda()
            probs.append(dict(V=V, K=K, S=S, seed=7 * n + r))
    if K <= 8:
        probs.append(dict(V=torch.ones((1, 2), dtype=torch.complex64, device="cuda"), K=K, exact=True))
        probs.append(dict(V=torch.from_numpy(inputs.factor(7, 2, seed=3, dtype=np.complex64)).cuda(), K=K, exact=True))
    # 64 problems of 8192 directions on 700 rows: 4096 items of one size (and K = 3) fill the chip
    V = torch.from_numpy(inputs.factor(700, 8, seed=9, dtype=np.complex64)).cuda()
    f_many, i_many = _run(probs + [dict(V=V, K=3, S=8192, seed=p) for p in range(64)])
    f_few, i_few = _run(probs)
    assert torch.equal(f_many[:len(probs)], f_few) and torch.equal(i_many[:len(probs)], i_few)
