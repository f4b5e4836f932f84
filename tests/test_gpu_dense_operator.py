"""The fixed-point dense operator's digits: Q = a p p^H + c I with |p_i| = 1 powers
of i has every entry's 53 bits add up in the same direction, so that a lost or
misplaced digit of Q shows in the largest eigenvalue n a + c (7 digits: the last
is worth 2^-48 of it; 16 2^-53 allowed, a few roundings of FP64), and its
eigenvector is p / sqrt(n).  One size gives the blocks a second trip over the
rows (n above 9728) and is no multiple of 4 or 128."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,a", [(1024, 1 + 21845 * 2.0 ** -52), (1531, (2.0 ** 53 - 1) * 2.0 ** -53),
                                 (1026, 4 / 3), (9731, 1 + 2 ** 40 / 3 * 2.0 ** -52)])
def test_largest_eigenpair(n, a):
    p = torch.tensor([1, 1j, -1, -1j], dtype=torch.complex128, device="cuda")
    k = torch.arange(n, device="cuda") * 7 % 11 % 4
    Q = p[(k[:, None] - k[None, :]) % 4] * a
    diag = a + 0.5
    Q.diagonal().fill_(diag)
    out = lrq.truncate(lrq.dense_matrix(Q), 1, max_iter=30, seed=3)
    lam = n * np.longdouble(a) + (np.longdouble(diag) - np.longdouble(a))
    assert abs(np.longdouble(out["lam"][0].item()) - lam) <= 16 * 2.0 ** -53 * lam
    v = out["V"][:, 0] / p[k]
    v = v / v[0]
    assert (v - 1).abs().max().item() <= 1e-12
