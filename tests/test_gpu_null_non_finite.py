"""The null-vector sampler on a V with NaN or infinite rows: a draw that meets
one is rejected, as a draw with a zero row is, so directions, draws and status
are those of V with these rows zeroed, for every rank's kernel."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("bad", [complex("nan"), complex(0.0, float("nan")), complex(float("inf"), 1.0)])
def test_rows_are_rejected(r, bad):
    V = inputs.factor(300, r, seed=r, dtype=np.complex64)
    rows = np.arange(5, 300, 29)
    V[rows, rows % r] = bad
    zeroed = V.copy()
    zeroed[rows] = 0
    got, ref = (lrq.sample_null_directions(torch.from_numpy(v).cuda(), 3, 3000, 11) for v in (V, zeroed))
    assert int(got["dev_status"].item()) == int(ref["dev_status"].item()) == 0
    assert int(got["draws"].item()) == int(ref["draws"].item()) > 3000
    assert torch.equal(torch.view_as_real(got["C"]), torch.view_as_real(ref["C"]))
