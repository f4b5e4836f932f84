"""Re-scoring by unit sums (K = 2, 3, 4, 6), by products (other K) and with
flushes in mid-chunk (rows per lane above 256), against the FP64 oracle.
Tolerance: a lane's double-float sum of 256 rows is off by at most 256 * 2^-47
of its terms' magnitudes, and f by twice that over |V^H z| / sum |V_i| > 0.05
for these inputs: 7e-11, so 1e-10."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r,K,m", [(1, 1, 4, 1), (33, 8, 6, 17), (257, 5, 2, 15), (255, 4, 6, 16), (256, 3, 7, 3),
                                     (700, 8, 3, 33), (700, 5, 8, 5), (513, 2, 9, 2), (200001, 2, 3, 512)])
def test_against_oracle(n, r, K, m):
    S = 24
    V = inputs.factor(n, r, seed=n + K, dtype=np.complex64)
    C = inputs.directions(S, r, seed=K, dtype=np.complex64)
    idx = np.random.Generator(np.random.PCG64(m)).integers(0, S, m)
    out = lrq.rescore(torch.from_numpy(V).cuda(), K, torch.from_numpy(C).cuda(), torch.from_numpy(idx).cuda(),
                      want_z=n < 1000)
    lrq.check_status(out["dev_status"])
    f = out["f"].cpu().numpy()
    ref = oracle.score(V.astype(np.complex128), K, C.astype(np.complex128))[idx]
    assert np.all(np.abs(f - ref) <= 1e-10 * np.abs(ref))
    if n < 1000:  # the codes give the same value
        z = np.exp(2j * np.pi * out["z"].cpu().numpy() / K)
        fz = (np.abs(z @ V.conj().astype(np.complex128)) ** 2).sum(1)
        assert np.all(np.abs(fz - f) <= 1e-10 * f)


def test_non_finite_row_is_reported():
    V = torch.from_numpy(inputs.factor(9000, 3, seed=1, dtype=np.complex64)).cuda()
    V[8999, 2] = float("inf")
    C = torch.from_numpy(inputs.directions(4, 3, seed=2, dtype=np.complex64)).cuda()
    out = lrq.rescore(V, 3, C, torch.tensor([1, 0], device="cuda"))
    assert int(out["dev_status"].item()) == lrq.LRQ_EINVAL
