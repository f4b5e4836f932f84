"""vMF loss and gradient where the split of the targets can go wrong: fewer
targets than lanes, counts around the groups of eight and the cluster sizes,
one instance and more than the chip holds, targets at an odd address, very
large and very small concentrations.  Tolerances of the loss kernel: 1e-9 on
the loss, float rounding on the gradient."""
import numpy as np
import pytest

from oracle import learned as OL
from paper_2602_20376_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("B,T,kscale,shift", [(1, 1, 0.0, 0), (1, 7, 0.0, 0), (3, 8, 2.0, 1), (2, 33, -6.0, 0),
                                              (5, 257, 40.0, 0), (64, 164, 0.0, 1), (400, 9, 3.0, 0),
                                              (1, 2100, 300.0, 0)])
def test_loss_and_gradient(B, T, kscale, shift):
    from paper_2602_20376_gb300 import lrq
    g = I.rng(100 * B + T)
    O = g.standard_normal((B, 160)).astype(np.float32)
    O.reshape(B, 16, 10)[:, :, 8] += kscale
    x = g.standard_normal((B, T, 8))
    x = (x / np.linalg.norm(x, axis=2, keepdims=True)).astype(np.float32)
    buf = torch.empty(B * T * 8 + shift, dtype=torch.float32, device="cuda")
    tx = buf[shift:].view(B, T, 8)
    tx.copy_(torch.from_numpy(x))
    loss = torch.empty(1, dtype=torch.float64, device="cuda")
    dO = torch.empty((B, 160), dtype=torch.float32, device="cuda")
    lrq.lrq_vmf_nll(torch.from_numpy(O).cuda(), tx, loss, dO)
    ref = OL.nll(O.astype(np.float64), x.astype(np.float64))
    gref = OL.nll_grad(O.astype(np.float64), x.astype(np.float64)).reshape(B, 160)
    assert abs(float(loss.item()) - ref) <= 1e-9 * max(1.0, abs(ref))
    assert np.abs(dO.cpu().numpy() - gref).max() <= 1e-6 * np.abs(gref).max()
