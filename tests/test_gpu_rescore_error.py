"""The re-scored values' error against extended precision, for the codes the
call reports.  The alphabets whose roots are products take them as pairs of FP32
numbers, off by up to 2^-50 a component: f is off by about twice a third of
that in the mean, and FP64 sums add some 2^-53, 9e-16 together; unit sums (K =
2, 3, 4, 6) are exact up to pairs of 48 bits, well below it."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu
ld = np.longdouble


@pytest.mark.skipif(np.finfo(ld).eps > 2.0 ** -60, reason="no extended precision")
@pytest.mark.parametrize("K", [2, 3, 4, 5, 6, 7, 8, 9, 16])
def test_error(K):
    turn = 2 * ld("3.14159265358979323846264338327950288") * np.arange(K).astype(ld) / K
    c, s, err = np.cos(turn), np.sin(turn), []
    for n, r in ((300, 2), (300, 4), (300, 6), (3000, 3)):
        m = 32
        V = inputs.factor(n, r, seed=n + r, dtype=np.complex64)
        C = inputs.directions(m, r, seed=K, dtype=np.complex64)
        out = lrq.rescore(torch.from_numpy(V).cuda(), K, torch.from_numpy(C).cuda(), torch.arange(m, device="cuda"),
                          want_z=True)
        z, f = out["z"].cpu().numpy(), out["f"].cpu().numpy()
        re, im = V.real.astype(ld), V.imag.astype(ld)
        for t in range(m):
            a = np.stack([re[z[t] == k].sum(0) for k in range(K)], 1)  # r x K sums per code
            b = np.stack([im[z[t] == k].sum(0) for k in range(K)], 1)
            ref = (((a * c + b * s).sum(1)) ** 2 + ((a * s - b * c).sum(1)) ** 2).sum()
            err.append(float((ld(f[t]) - ref) / ref))
    assert np.sqrt(np.mean(np.square(err))) <= 9e-16
