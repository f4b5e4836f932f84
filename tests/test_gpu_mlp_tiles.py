"""The network's BF16 GEMMs at the edges of their tiles: batches around 128
rows, batch sizes above one staged chunk of 256 (the reduction length of the
weight gradients), batches that take the wide tile, feature counts that are no
multiple of 4 or 16, and buffers off a 16-byte boundary.  Each layer is
checked on the kernel's own inputs: operands rounded to bfloat16, products
summed in FP64; bound: (K + 2) roundings of FP32 on the sum of magnitudes."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import lrq

pytestmark = pytest.mark.gpu
W, OUT = 256, 160


def _near(got, a, b, bias=None, mask=None, relu=False):
    a, b = a.to(torch.bfloat16).double(), b.to(torch.bfloat16).double()
    ref, mag = a @ b, a.abs() @ b.abs()
    if bias is not None:
        ref, mag = ref + bias.double(), mag + bias.double().abs()
    if relu:
        ref = torch.relu(ref)
    if mask is not None:
        ref = ref * (mask > 0)
    assert bool(((got.double() - ref).abs() <= (a.shape[1] + 2) * 2.0 ** -23 * mag).all())


@pytest.mark.parametrize("B,F,off", [(1, 24, 0), (64, 24, 1), (127, 7, 0), (128, 24, 0), (129, 30, 3), (257, 24, 0),
                                     (600, 9, 1), (5000, 24, 0), (20000, 24, 1)])
def test_layers(B, F, off):
    g = torch.Generator(device="cuda")
    g.manual_seed(B + F)

    def buf(*shape):
        n = int(np.prod(shape))
        return torch.randn(n + off, generator=g, device="cuda")[off:].view(*shape)

    P = lrq.lrq_proposal_num_params(F)
    params, X, dO = buf(P) * 0.1, buf(B, F), buf(B, OUT)
    params = torch.cat([torch.zeros(off, device="cuda"), params])[off:]
    H1, H2, O, grads, scratch = buf(B, W), buf(B, W), buf(B, OUT), buf(P), buf(2, B, W)
    lrq.lrq_mlp_forward(params, X, H1, H2, O, True)
    lrq.lrq_mlp_backward(params, X, H1, H2, dO, grads, scratch, True)
    sizes = [F * W, W, W * W, W, W * OUT, OUT]
    w1, b1, w2, b2, w3, b3 = torch.split(params, sizes)
    w1, w2, w3 = w1.view(F, W), w2.view(W, W), w3.view(W, OUT)
    d1, e1, d2, e2, d3, e3 = torch.split(grads, sizes)
    _near(H1, X, w1, b1, relu=True)
    _near(H2, H1, w2, b2, relu=True)
    _near(O, H2, w3, b3)
    dH2, dH1 = scratch[0], scratch[1]
    _near(d3.view(W, OUT), H2.T, dO)
    _near(dH2, dO, w3.T, mask=H2)
    _near(d2.view(W, W), H1.T, dH2)
    _near(dH1, dH2, w2.T, mask=H1)
    _near(d1.view(F, W), X.T, dH1)
