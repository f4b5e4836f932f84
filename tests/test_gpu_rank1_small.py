"""The sweep on graphs of some thousand vertices, where launches are what it
costs: no more of them than a bitonic network over the padded pairs takes,
and the same results from either sort (the largest network, the smallest radix
sort).  f to 1e-9 relative, cuts exact (the sweep tests' tolerances)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


def _ring(n):
    i = np.arange(n)
    colidx = np.sort(np.stack([(i - 1) % n, (i + 1) % n], 1), 1).astype(np.int32).reshape(-1)
    return (2 * np.arange(n + 1)).astype(np.int32), colidx


@pytest.mark.parametrize("n", [2049, 4096, 4097, 8192, 16384, 32768])
def test_launches(n):
    rowptr, colidx = _ring(n)
    q = torch.from_numpy(inputs.complex_gaussian((n,), seed=n)).cuda()
    rp, ci = torch.from_numpy(rowptr).cuda(), torch.from_numpy(colidx).cuda()
    before = lrq.lrq_kernel_launches()
    lrq.rank1_sweep(q, 3, rp, ci)
    taken = lrq.lrq_kernel_launches() - before
    sizes = int(np.ceil(np.log2(n / 2048)))  # merges above a block's 2048 pairs
    assert taken <= 1 + sizes * (sizes + 3) // 2 + 8


@pytest.mark.parametrize("n", [131072, 131073])
@pytest.mark.parametrize("equal", [False, True])
def test_both_sorts(n, equal):
    q = inputs.complex_gaussian((n,), seed=n)
    if equal:  # four phases only: the order is the index's
        q = np.abs(q) * np.exp(0.5j * np.pi * (np.arange(n) * 7 % 4) + 0.1j)
    rowptr, colidx = _ring(n)
    out = lrq.rank1_sweep(torch.from_numpy(q).cuda(), 3, torch.from_numpy(rowptr).cuda(), torch.from_numpy(colidx).cuda())
    z, order = oracle.rank1_sweep_states(q, 3)
    om = np.exp(2j * np.pi * np.arange(4) / 3)
    z = z.astype(np.int64)
    step = (q.conj() * (om[z + 1] - om[z]))[order]
    f_ref = (np.abs(np.concatenate([[0], np.cumsum(step)]) + (q.conj() * om[z]).sum()) ** 2).max()
    assert abs(float(out["f"].item()) - f_ref) <= 1e-9 * f_ref
    # every state's cut on the ring: an edge changes where its first end advances and back where the second does
    rank = np.empty(n, np.int64)
    rank[order] = np.arange(n)
    i = np.arange(n)
    j = (i + 1) % n
    first = rank[i] < rank[j]
    before = (z[i] != z[j]).astype(np.int64)
    between = ((z[i] + first) % 3 != (z[j] + ~first) % 3).astype(np.int64)
    diff = np.zeros(n + 1, np.int64)
    np.add.at(diff, np.minimum(rank[i], rank[j]) + 1, between - before)
    np.add.at(diff, np.maximum(rank[i], rank[j]) + 1, before - between)
    best = int((before.sum() + np.cumsum(diff)).max())
    assert int(out["cut"].item()) == best
    assert oracle.cut_count(rowptr, colidx, out["zcut"].cpu().numpy()) == best
