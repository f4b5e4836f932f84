"""Odd alphabets in the re-scoring: a coordinate opposite a boundary (a positive
real w, at the middle of its sector) is decided in FP32 like any other.  With a
non-negative real V and direction every coordinate is one: the call takes no
longer than on complex data (twice its time allowed; FP64 decisions took six times),
and codes and values are the oracle's."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


def _ms(V, K, C, idx, ws):
    best = float("inf")
    for _ in range(8):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        lrq.rescore(V, K, C, idx, ws=ws)
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


@pytest.mark.parametrize("K,r", [(3, 4), (5, 3), (7, 8)])
def test_positive_real(K, r):
    n, m = 1 << 17, 64
    V = torch.from_numpy(inputs.factor(n, r, seed=K, dtype=np.complex64)).cuda()
    C = torch.from_numpy(inputs.directions(m, r, seed=r, dtype=np.complex64)).cuda()
    idx = torch.arange(m, device="cuda")
    ws = lrq.workspace(lrq.lrq_rescore_workspace_size(n, r, m), "cuda")
    pos_V, pos_C = (x.real.abs().to(torch.complex64).contiguous() for x in (V, C))
    assert _ms(pos_V, K, pos_C, idx, ws) <= 2.0 * _ms(V, K, C, idx, ws)


@pytest.mark.parametrize("K", [3, 5, 7])
def test_codes_on_every_axis(K):
    # w on each boundary's far half (the middle of a sector), a hair to either side, and generic
    g = np.random.Generator(np.random.PCG64(K))
    mid = np.exp(2j * np.pi * np.arange(K) / K)
    turn = np.array([0.0, 1e-9, -1e-9, 1e-6, -1e-6, 1e-4, -1e-4])
    V = (np.exp(g.uniform(-3, 3, (40, 1, 1))) * mid[None, :, None] * np.exp(1j * turn)[None, None, :]).reshape(-1, 1)
    V = np.concatenate([V, g.standard_normal((500, 1)) + 1j * g.standard_normal((500, 1))]).astype(np.complex64)
    C = np.concatenate([np.ones((1, 1)), mid[:, None]]).astype(np.complex64)
    out = lrq.rescore(torch.from_numpy(V).cuda(), K, torch.from_numpy(C).cuda(),
                      torch.arange(K + 1, device="cuda"), want_z=True)
    w = V.astype(np.complex128) @ C.astype(np.complex128).T
    t = np.angle(w) * K / (2 * np.pi)
    assert np.abs(t - np.floor(t) - 0.5).min() > 1e-6  # no boundary tie among them
    assert np.array_equal(out["z"].cpu().numpy().T, np.mod(np.round(t), K).astype(np.uint8))
    ref = oracle.score(V.astype(np.complex128), K, C.astype(np.complex128))
    assert np.allclose(out["f"].cpu().numpy(), ref, rtol=1e-10, atol=0)
