"""The re-scoring's final step (a warp per candidate, then the best of them)
at the edges of its ranges: one candidate, counts around a block of 256, the
largest m, one chunk and many, repeated indices (ties go to the earlier
position) and an index out of range.  Tolerance as for every re-scoring:
1e-9 relative of the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r,K,m", [(1, 1, 2, 1), (255, 4, 3, 255), (257, 4, 3, 257), (9000, 2, 5, 33),
                                     (300, 8, 12, 4096)])
def test_sums_and_best(n, r, K, m):
    S = 64
    V = inputs.factor(n, r, seed=n + m, dtype=np.complex64)
    C = inputs.directions(S, r, seed=3, dtype=np.complex64)
    idx = np.random.Generator(np.random.PCG64(m)).integers(0, S, m)
    out = lrq.rescore(torch.from_numpy(V).cuda(), K, torch.from_numpy(C).cuda(), torch.from_numpy(idx).cuda())
    lrq.check_status(out["dev_status"])
    f = out["f"].cpu().numpy()
    ref = oracle.score(V.astype(np.complex128), K, C.astype(np.complex128))[idx]
    assert np.all(np.abs(f - ref) <= 1e-9 * np.abs(ref))
    t = int(np.argmax(f))  # the earliest of equal values
    assert int(out["best"].item()) == idx[t] and float(out["best_f"].item()) == f[t]


def test_index_out_of_range():
    V = torch.from_numpy(inputs.factor(500, 3, seed=1, dtype=np.complex64)).cuda()
    C = torch.from_numpy(inputs.directions(4, 3, seed=2, dtype=np.complex64)).cuda()
    out = lrq.rescore(V, 3, C, torch.tensor([1, 9, -1, 2], device="cuda"))
    f = out["f"].cpu().numpy()
    assert f[1] == -1.0 and f[2] == -1.0 and int(out["best"].item()) in (1, 2)
    assert int(out["dev_status"].item()) == lrq.LRQ_EINVAL
