"""The greedy search on both sides of the vertex count where it goes from 8
lanes a row to a thread a row with marks, on graphs with long rows: labels,
rounds and moves equal to the rounds done in numpy."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [7, 31, 40959, 40960, 40961])
def test_rounds(n):
    K = 3
    g = np.random.Generator(np.random.PCG64(n))
    hubs = np.concatenate([np.zeros(63, int), np.full(65, 1), np.full(700, 2)]) if n > 1000 else np.zeros(40, int)
    a = np.concatenate([hubs, g.integers(0, n, 4 * n)])
    b = np.concatenate([g.integers(0, n, hubs.size), g.integers(0, n, 4 * n)])
    src, dst = np.concatenate([a, b]), np.concatenate([b, a])
    order = np.lexsort((dst, src))
    src, colidx = src[order], dst[order].astype(np.int32)
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int32)
    z0 = g.integers(0, K, n).astype(np.uint8)
    out = lrq.greedy_cut(torch.from_numpy(rowptr).cuda(), torch.from_numpy(colidx).cuda(), K, torch.from_numpy(z0).cuda())
    z, rounds, moves, own = z0.astype(np.int64), 0, 0, src != colidx
    while True:
        cnt = np.zeros((n, K), np.int64)
        np.add.at(cnt, (src[own], z[colidx[own]]), 1)
        same = cnt[np.arange(n), z]
        cnt[np.arange(n), z] = 1 << 40
        best = cnt.argmin(1)
        gain = np.maximum(same - cnt.min(1), 0)
        s, d = src[own], colidx[own]
        outranked = (gain[d] > gain[s]) | ((gain[d] == gain[s]) & (d < s))
        blocked = np.zeros(n, bool)
        blocked[s[outranked]] = True
        move = (gain > 0) & ~blocked
        if not move.any():
            break
        z[move] = best[move]
        rounds, moves = rounds + 1, moves + int(move.sum())
    assert np.array_equal(out["z"].cpu().numpy(), z.astype(np.uint8))
    assert (out["rounds"], out["moves"], out["converged"]) == (rounds, moves, True)
    assert int(out["cut"].item()) == oracle.cut_count(rowptr, colidx, z.astype(np.uint8))
