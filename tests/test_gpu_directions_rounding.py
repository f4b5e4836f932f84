"""Every component of a uniform direction is the FP32 rounding of its FP64 value:
against FP64 numpy on the same Philox stream, over some millions of components,
a component may differ from numpy's rounding only where the value lies within
2^-50 of the middle of two FP32 numbers (two FP64 evaluations of a unit vector's
component)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,S,seed", [(1, 400000, 3), (2, 300000, 2 ** 33 + 9), (4, 300000, 1), (7, 60000, 5), (64, 5000, 8)])
def test_rounding(r, S, seed):
    C = torch.empty((S, r), dtype=torch.complex64, device="cuda")
    lrq.lrq_sample_directions(seed, S, r, C)
    got, ref = C.cpu().numpy(), oracle.sphere_sample(seed, S, r)
    for g, x in ((got.real, ref.real), (got.imag, ref.imag)):
        half = np.maximum(np.spacing(np.abs(g)), np.abs(g - np.nextafter(g, np.float32(0)))).astype(np.float64) / 2
        assert np.all(np.abs(g.astype(np.float64) - x) <= half + 2.0 ** -50)
