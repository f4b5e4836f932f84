"""A dense truncation whose workspace leaves no room for the operator's digits
runs in FP64 from Q, as before there were any: same eigenvalues (to n 2^-53
||Q||, the tolerance of the dense operator's test) with the full workspace, with
14 n^2 bytes less, and through the binding when the full one cannot be had.  A
workspace below that is still refused."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1024, 1027])
def test_without_room_for_digits(n, monkeypatch):
    r = 3
    g = inputs.complex_gaussian((n, r), seed=n)
    Q = g @ g.conj().T + 0.05 * inputs.hermitian_gaussian(n, seed=n + 1)
    ref = np.linalg.eigvalsh(Q)
    dQ = torch.from_numpy(Q).cuda()
    Qm = lrq.dense_matrix(dQ)
    need = lrq.lrq_truncate_workspace_size(Qm, r, 0)
    lam, st = torch.empty(r, dtype=torch.float64, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    for size in (need, need - 14 * n * n):
        lam.zero_()
        lrq.lrq_truncate(Qm, r, 0.0, 0, 5, None, None, lam, lrq.workspace(size, "cuda"), st)
        assert np.abs(lam.cpu().numpy() - ref[::-1][:r]).max() <= 4 * n * 2.0 ** -53 * np.abs(ref).max()
    with pytest.raises(lrq.LrqError):
        lrq.lrq_truncate(Qm, r, 0.0, 0, 5, None, None, lam, lrq.workspace(need // 4, "cuda"), st)
    plain = lrq.workspace

    def short(nbytes, device):
        if nbytes >= need:
            raise torch.cuda.OutOfMemoryError("no room")
        return plain(nbytes, device)

    monkeypatch.setattr(lrq, "workspace", short)
    out = lrq.truncate(Qm, r, seed=5)
    assert np.abs(out["lam"].cpu().numpy() - ref[::-1][:r]).max() <= 4 * n * 2.0 ** -53 * np.abs(ref).max()
