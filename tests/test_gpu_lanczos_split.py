"""Truncation at the edges of its kernels' splits: rows per warp of the dense
operator (n around 608), warps per row tile of the Gram-Schmidt update (n
around 155 648), groups of eight basis vectors, and operators scaled by
powers of two (the update's FP32 correction is taken relative to the vector's
norm).  Tolerances of the truncation tests: eigenvalues 1e-9 ||Q|| of LAPACK
or the closed form, residuals 1e-8 ||Q||, orthonormality 1e-9."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


def _check(Qv, out, norm):
    V, lam = out["V"].cpu().numpy(), out["lam"].cpu().numpy()
    U = V / np.sqrt(lam)[None, :]
    assert np.abs(U.conj().T @ U - np.eye(len(lam))).max() <= 1e-9
    assert np.linalg.norm(Qv(U) - U * lam[None, :], axis=0).max() <= 1e-8 * norm


@pytest.mark.parametrize("n,r,exp2", [(9, 1, 0), (33, 3, 0), (606, 4, 0), (607, 2, -120), (608, 4, 120), (609, 3, 0),
                                      (1025, 8, 0)])
def test_dense(n, r, exp2):
    g = inputs.complex_gaussian((n, r), seed=n)
    Q = (g @ g.conj().T + inputs.hermitian_gaussian(n, seed=n + 1)) * 2.0 ** exp2
    Q = 0.5 * (Q + Q.conj().T)
    Qd = torch.from_numpy(Q).cuda()
    out = lrq.truncate(lrq.dense_matrix(Qd), r, seed=5)
    ref = np.linalg.eigvalsh(Q)[::-1][:r]
    norm = np.abs(np.linalg.eigvalsh(Q)).max()
    assert np.abs(out["lam"].cpu().numpy() - ref).max() <= 1e-9 * norm
    _check(lambda U: Q @ U, out, norm)


@pytest.mark.parametrize("n", [155647, 155648, 155905])
@pytest.mark.parametrize("weight", [None, 2.0 ** -130])
def test_laplacian(n, weight):
    rowptr, colidx, _ = inputs.sbm_graph(n, 4.0, 8.0, seed=n)
    w = None if weight is None else np.full(len(colidx), weight)
    rp, ci = torch.from_numpy(rowptr).cuda(), torch.from_numpy(colidx).cuda()
    wd = None if w is None else torch.from_numpy(w).cuda()
    out = lrq.truncate(lrq.laplacian_matrix(rp, ci, wd), 2, max_iter=1000, seed=1)
    s = 1.0 if weight is None else weight
    deg = np.diff(rowptr).astype(float)

    def apply(U):
        rows = np.repeat(np.arange(n), np.diff(rowptr))
        return np.stack([s * (deg * u - np.bincount(rows, weights=u[colidx].real, minlength=n)) for u in U.T], axis=1)

    _check(apply, out, float(out["lam"][0]))
