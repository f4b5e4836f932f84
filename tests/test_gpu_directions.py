"""Uniform directions: ranks around the block's candidates per component
layout, and draws against the oracle's FP64 Philox + Box-Muller stream (1e-6
absolute, the sampler's tolerance; almost all components equal its FP32
rounding)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 2, 3, 5, 7, 8, 33, 64])
@pytest.mark.parametrize("S", [1, 63, 64, 65, 4099])
def test_matches_oracle(r, S):
    C = torch.empty((S, r), dtype=torch.complex64, device="cuda")
    lrq.lrq_sample_directions(2 ** 40 + 7, S, r, C)
    got = C.cpu().numpy()
    ref = oracle.sphere_sample(2 ** 40 + 7, S, r)
    assert np.abs(got - ref).max() <= 1e-6
    assert np.mean(got != ref.astype(np.complex64)) <= 0.01
