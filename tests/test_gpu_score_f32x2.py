"""FP32 scoring with packed FMAs (one call and batched): every alphabet class
(sign tables, the run-time sign rule of the batched kernel, angles above 8)
and rank class (two candidates a thread or one), row counts around the
staging tiles and candidate counts around a block.  Bound: 1e-5 relative of
the FP64 oracle (FP32 scoring's), and for every coordinate whose FP64 value
lies within the FP32 projection's rounding of a decision boundary (where the
two may round to different roots) 2 sin(pi/K) |V_i| on ||V^H z||."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [2, 3, 4, 5, 6, 7, 8, 9, 64])
@pytest.mark.parametrize("n,r,S", [(1, 1, 1), (255, 2, 255), (257, 4, 257), (129, 5, 129), (513, 6, 128), (300, 8, 65)])
def test_scores(K, n, r, S):
    V = inputs.factor(n, r, seed=n + r, dtype=np.complex64)
    C = inputs.directions(S, r, seed=S, dtype=np.complex64)
    out = lrq.sample_score(torch.from_numpy(V).cuda(), K, C=torch.from_numpy(C).cuda(), mode=lrq.LRQ_MODE_FP32,
                           top_m=1, want_scores=True)
    lrq.check_status(out["dev_status"])
    V64, C64 = V.astype(np.complex128), C.astype(np.complex128)
    ref = oracle.score(V64, K, C64)
    w = V64 @ C64.T
    # distance of w to the nearest boundary ray's line against (2 r + 8) roundings of its terms
    dist = np.abs(w) * np.sin(np.minimum(np.pi / 2, _margin(w, K)))
    tie = dist <= (2 * r + 8) * 2.0 ** -23 * (np.abs(V64) @ np.abs(C64).T)
    slack = 2 * np.sin(np.pi / K) * (tie * np.linalg.norm(V64, axis=1)[:, None]).sum(0)
    got = np.sqrt(out["scores"].cpu().numpy().astype(np.float64))
    assert np.all(np.abs(got - np.sqrt(ref)) <= 5e-6 * np.sqrt(ref) + 1e-6 * np.sqrt(ref.max()) + slack)


def _margin(w, K):
    """Angle between w and the nearest decision boundary pi (2 m + 1) / K."""
    t = np.mod(np.angle(w) * K / (2 * np.pi) - 0.5, 1.0)
    return np.minimum(t, 1.0 - t) * 2 * np.pi / K


def test_batched_winners():
    probs, host = [], []
    for t, (n, r, K, S) in enumerate([(127, 1, 2, 64), (128, 2, 3, 65), (129, 3, 4, 130), (200, 4, 8, 257),
                                      (300, 5, 5, 100), (64, 6, 6, 33), (90, 7, 7, 511), (257, 8, 9, 300)]):
        V = inputs.factor(n, r, seed=50 + t, dtype=np.complex64)
        C = inputs.directions(S, r, seed=80 + t, dtype=np.complex64)
        host.append((V.astype(np.complex128), K, C.astype(np.complex128)))
        probs.append(dict(V=torch.from_numpy(V).cuda(), K=K, C=torch.from_numpy(C).cuda()))
    plan = lrq.BatchedPlan(probs, top_m=4)
    plan.run()
    lrq.check_status(plan.status)
    for (V, K, C), f, i in zip(host, plan.best_f.cpu().numpy(), plan.best_idx.cpu().numpy()):
        ref = oracle.score(V, K, C)
        assert abs(f - ref[i]) <= 1e-9 * ref[i] and ref[i] >= ref.max() * (1 - 1e-5)


def test_zero_direction_keeps_code_zero():
    V = inputs.factor(300, 3, seed=1, dtype=np.complex64)
    for K in (2, 3, 4, 5, 8):
        out = lrq.sample_score(torch.from_numpy(V).cuda(), K, C=torch.zeros((3, 3), dtype=torch.complex64, device="cuda"),
                               mode=lrq.LRQ_MODE_FP32, top_m=1, want_scores=True)
        ref = float((np.abs(V.astype(np.complex128).sum(0)) ** 2).sum())
        assert np.abs(out["scores"].cpu().numpy() - ref).max() <= 1e-5 * ref
