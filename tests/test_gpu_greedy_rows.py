"""Greedy rounds and the cut count with rows on both sides of a thread's share
(64 entries), parallel edges and self loops, and several rounds (marked
vertices only): labels, rounds, moves and cut equal the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,K", [(33, 2), (2500, 3), (2500, 8)])
def test_hubs(n, K):
    g = np.random.Generator(np.random.PCG64(n + K))
    a = np.concatenate([np.zeros(63, int), np.ones(64, int), np.full(65, 2), np.full(700, 3), g.integers(0, n, 4 * n)])
    b = np.concatenate([g.integers(4, n, 892), g.integers(0, n, 4 * n)])
    src, dst = np.concatenate([a, b]), np.concatenate([b, a])
    order = np.lexsort((dst, src))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int32)
    colidx = dst[order].astype(np.int32)
    rp, ci = torch.from_numpy(rowptr).cuda(), torch.from_numpy(colidx).cuda()
    z0 = g.integers(0, K, n).astype(np.uint8)
    for rounds in (0, 1, 1 << 20):
        out = lrq.greedy_cut(rp, ci, K, torch.from_numpy(z0).cuda(), rounds)
        z, nr, moves, conv = oracle.greedy_cut(rowptr, colidx, K, z0, rounds)
        assert np.array_equal(out["z"].cpu().numpy(), z)
        assert (out["rounds"], out["moves"], out["converged"]) == (nr, moves, conv)
        assert int(out["cut"].item()) == oracle.cut_count(rowptr, colidx, z)
