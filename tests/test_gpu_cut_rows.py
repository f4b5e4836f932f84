"""The cut count with 8 lanes a row and a thread a row (up to 40960 vertices and
above), rows on both sides of 64 entries, on a dense graph, against numpy."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(1, 0), (3, 2), (33, 400), (700, 140000), (40960, 200000), (40961, 200000)])
def test_count(n, m):
    g = np.random.Generator(np.random.PCG64(n))
    a, b = g.integers(0, n, m), g.integers(0, n, m)
    hub = g.integers(0, n, min(n, 900))
    a, b = np.concatenate([a, np.zeros(hub.size, int)]), np.concatenate([b, hub])
    src, dst = np.concatenate([a, b]), np.concatenate([b, a])
    order = np.lexsort((dst, src))
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(src, minlength=n))]).astype(np.int32)
    z = g.integers(0, 3, n).astype(np.uint8)
    cut = torch.empty(1, dtype=torch.int64, device="cuda")
    lrq.lrq_cut_count(torch.from_numpy(rowptr).cuda(), torch.from_numpy(dst[order].astype(np.int32)).cuda(),
                      torch.from_numpy(z).cuda(), cut)
    assert int(cut.item()) == int((z[a] != z[b]).sum())
