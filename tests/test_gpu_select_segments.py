"""The top-m selection at the edges of its segments of 2048 keys, and where the
survivors of a pass fill more than one segment again (two and three passes)."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("S,m", [(2047, 512), (2048, 512), (2049, 512), (2049, 1), (4096, 17), (4097, 300),
                                 (20000, 512), (100003, 512)])
def test_stable_order(S, m):
    V = torch.from_numpy(inputs.factor(200, 3, seed=S, dtype=np.complex64)).cuda()
    C = torch.from_numpy(inputs.directions(S, 3, seed=m, dtype=np.complex64)).cuda()
    C[S // 2:] = C[:S - S // 2].clone()  # ties
    out = lrq.sample_score(V, 3, C=C, mode=lrq.LRQ_MODE_FP32, top_m=m, want_scores=True)
    s = out["scores"].cpu().numpy()
    order = np.argsort(-s, kind="stable")[:m]
    assert np.array_equal(out["top_idx"].cpu().numpy(), order)
    assert np.array_equal(out["top_f"].cpu().numpy(), s[order])
