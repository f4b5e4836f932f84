"""The dense operator in fixed point (1024 <= n <= 32768) at its edges: rows and
columns past a multiple of 4 and 128, a leading dimension above n, rows of very
different size, zero rows, tiny and huge matrices.  Each entry and product is
off by at most about 2^-54 of its row's largest, so eigenvalues agree with
LAPACK's to n 2^-53 ||Q|| and residuals to Lanczos' own tolerance."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,r,exp2,spread", [(1023, 2, 0, 0), (1024, 3, 0, 0), (1025, 2, -300, 0), (1151, 1, 300, 0),
                                             (1153, 4, 0, 10), (1282, 2, 0, 25)])
def test_eigenpairs(n, r, exp2, spread):
    g = inputs.complex_gaussian((n, r), seed=n)
    Q = g @ g.conj().T + 0.05 * inputs.hermitian_gaussian(n, seed=n + 1)
    s = 2.0 ** np.random.Generator(np.random.PCG64(n)).integers(-spread, spread + 1, n) if spread else np.ones(n)
    s[n // 2] = 0.0  # a zero row and column
    Q = s[:, None] * Q * s[None, :] * 2.0 ** exp2
    Q = 0.5 * (Q + Q.conj().T)
    wide = torch.full((n, n + 3), complex("nan"), dtype=torch.complex128, device="cuda")
    wide[:, :n] = torch.from_numpy(Q).cuda()
    Qm = lrq.LrqMatrix(lrq.LRQ_MATRIX_DENSE_C128, n, wide.data_ptr(), n + 3, None, None, None, 0)
    out = lrq.truncate(Qm, r, seed=5)
    ref = np.linalg.eigvalsh(Q)
    norm = np.abs(ref).max()
    assert np.abs(out["lam"].cpu().numpy() - ref[::-1][:r]).max() <= 4 * n * 2.0 ** -53 * norm
    lam, V = out["lam"].cpu().numpy(), out["V"].cpu().numpy()
    U = V / np.sqrt(lam)[None, :]
    assert np.linalg.norm(Q @ U - U * lam[None, :], axis=0).max() <= 1e-8 * norm


def test_non_finite_entry_is_reported():
    Q = torch.eye(1100, dtype=torch.complex128, device="cuda")
    Q[1099, 3] = float("inf")
    with pytest.raises(Exception):
        lrq.truncate(lrq.dense_matrix(Q), 1)
