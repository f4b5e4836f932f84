"""Packing, finalize and selection around the scoring kernels, at the edges of
their tiles, blocks and segments.

* A power of two on V scales every tensor-core score by its square exactly:
  the row exponents, the global scale, the packed operands and the column sums
  do not depend on it.  Rows spread over 2^40, so that the exponents' clamp is
  reached.
* The selected list is the stable descending order of the scores of the same
  call.
* A non-finite entry anywhere is reported."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


def _factor(n, r, seed):
    V = torch.from_numpy(inputs.factor(n, r, seed=seed, dtype=np.complex64))
    g = torch.Generator().manual_seed(seed)
    return (V * torch.exp2(torch.randint(-20, 20, (n, 1), generator=g).float())).cuda()


@pytest.mark.parametrize("K", range(2, 9))
@pytest.mark.parametrize("n,r", [(1, 1), (16, 3), (79, 4), (81, 2), (129, 5), (641, 6), (20001, 8)])
def test_power_of_two_scales_out(n, r, K):
    V = _factor(n, r, n + K)
    C = torch.from_numpy(inputs.directions(130, r, seed=K, dtype=np.complex64)).cuda()
    ref = lrq.sample_score(V, K, C=C, mode=1, top_m=1, want_scores=True)["scores"]
    for e in (-17, 13):
        got = lrq.sample_score(V * 2.0 ** e, K, C=C, mode=1, top_m=1, want_scores=True)
        lrq.check_status(got["dev_status"])
        assert torch.equal(got["scores"], ref * 4.0 ** e)


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("S,m", [(1, 1), (31, 31), (33, 5), (1023, 512), (1024, 1), (1025, 17), (5000, 164)])
def test_selection_is_the_stable_order(S, m, mode):
    V = _factor(300, 3, S)
    C = torch.from_numpy(inputs.directions(S, 3, seed=m, dtype=np.complex64)).cuda()
    C[S // 2:] = C[:S - S // 2].clone()  # ties
    out = lrq.sample_score(V, 3, C=C, mode=mode, top_m=m, want_scores=True)
    s = out["scores"].cpu().numpy()
    order = np.argsort(-s, kind="stable")[:m]
    assert np.array_equal(out["top_idx"].cpu().numpy(), order)
    assert np.array_equal(out["top_f"].cpu().numpy(), s[order])


@pytest.mark.parametrize("mode", [0, 1])
@pytest.mark.parametrize("where", ["V first", "V last", "C last"])
def test_non_finite_is_reported(where, mode):
    V = _factor(5121, 5, 1)
    C = torch.from_numpy(inputs.directions(129, 5, seed=2, dtype=np.complex64)).cuda()
    (V if where[0] == "V" else C)[0 if "first" in where else -1, -1 if "last" in where else 0] = float("nan")
    out = lrq.sample_score(V, 3, C=C, mode=mode, top_m=1)
    assert int(out["dev_status"].item()) == lrq.LRQ_EINVAL
