"""The sweep's sort and scans at the edges of their tiles: one block or radix
passes (n around 2048), a sort tile of 4096, a scan tile of 2048, many equal
phases (order by index), and long rows in the cut pass.  Tolerances of the
sweep tests: 1e-9 relative on f, cuts exact."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 2047, 2048, 2049, 4095, 4096, 4097, 12289])
@pytest.mark.parametrize("equal", [False, True])
def test_optimum(n, equal):
    q = inputs.complex_gaussian((n,), seed=n)
    if equal:  # four phases only
        q = np.abs(q) * np.exp(0.5j * np.pi * (np.arange(n) * 7 % 4) + 0.1j)
    out = lrq.rank1_sweep(torch.from_numpy(q).cuda(), 3)
    f_ref, _ = oracle.rank1_sweep(q, 3)
    f = float(out["f"].item())
    assert abs(f - f_ref) <= 1e-9 * f_ref
    assert abs(oracle.objective(q[:, None], 3, out["z"].cpu().numpy()) - f) <= 1e-9 * f


@pytest.mark.parametrize("K", [2, 3, 5])
def test_cut_with_hubs_and_parallel_edges(K):
    # hubs longer than a thread's share of a row (64 entries), parallel edges, self loops
    n = 2500
    g = np.random.Generator(np.random.PCG64(K))
    a = np.concatenate([np.zeros(63, int), np.ones(64, int), np.full(65, 2), np.full(900, 3), g.integers(0, n, 3000)])
    b = np.concatenate([g.integers(4, n, 63 + 64 + 65 + 900), g.integers(0, n, 3000)])
    src, dst = np.concatenate([a, b]), np.concatenate([b, a])
    order = np.lexsort((dst, src))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int32)
    colidx = dst[order].astype(np.int32)
    q = inputs.complex_gaussian((n,), seed=K)
    out = lrq.rank1_sweep(torch.from_numpy(q).cuda(), K, torch.from_numpy(rowptr).cuda(), torch.from_numpy(colidx).cuda())
    best, _, _ = oracle.rank1_sweep_cut(q, K, rowptr, colidx)
    assert int(out["cut"].item()) == best
    assert oracle.cut_count(rowptr, colidx, out["zcut"].cpu().numpy()) == best
