"""FP32 scoring for alphabets above 8 (scalar rows, one candidate a thread) and
below with one and two candidates a thread, for every rank: scores to 1e-5 of the
FP64 oracle on rows whose w keeps away from every boundary, and independent of the
number of blocks (the same direction in a small and in a large batch, bit for bit)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [3, 8, 9, 16, 64])
@pytest.mark.parametrize("r", range(1, 9))
def test_small_and_large_batches(K, r):
    n = 256  # one chunk of rows whatever the batch
    V = inputs.factor(n, r, seed=K + r, dtype=np.complex64)
    C = inputs.directions(512 * 700, r, seed=r, dtype=np.complex64)
    Vd, Cd = torch.from_numpy(V).cuda(), torch.from_numpy(C).cuda()
    few, many = (lrq.sample_score(Vd, K, C=c, mode=lrq.LRQ_MODE_FP32, top_m=1, want_scores=True)["scores"].cpu().numpy()
                 for c in (Cd[:300].contiguous(), Cd))
    assert np.array_equal(few, many[:300])
    C64 = C[:300].astype(np.complex128)
    w = V.astype(np.complex128) @ C64.T
    t = np.mod(np.angle(w) * K / (2 * np.pi) - 0.5, 1.0)
    tie = np.minimum(t, 1 - t) * 2 * np.pi / K * np.abs(w) < 1e-5 * np.abs(V).sum(1)[:, None]
    slack = 2 * np.sin(np.pi / K) * (tie * np.linalg.norm(V, axis=1)[:, None]).sum(0)
    ref = np.sqrt(oracle.score(V.astype(np.complex128), K, C64))
    assert np.all(np.abs(np.sqrt(few.astype(np.float64)) - ref) <= 5e-6 * ref + 1e-6 * ref.max() + slack)
