"""The enumeration's FP32 bounds: instances of every alphabet and rank against
the oracle's enumeration (value, set count, codes that score the value), with
tiny and zero rows, exponents far from 1, and identical rows (every
vertex uncertain in FP32).  Tolerances of the enumeration tests: 1e-9 relative
on the optimum, set counts equal."""
import numpy as np
import pytest
import torch

import oracle
from paper_2602_20376_gb300 import inputs, lrq

pytestmark = pytest.mark.gpu


def _run(V, K):
    out = lrq.enumerate_exact(torch.from_numpy(np.ascontiguousarray(V)).cuda(), K)
    lrq.check_status(out["dev_status"])
    return float(out["f"].item()), out["z"].cpu().numpy(), int(out["n_sets"].item())


@pytest.mark.parametrize("n,r,K", [(1, 1, 2), (40, 1, 8), (9, 2, 2), (8, 2, 3), (8, 2, 4), (6, 2, 5), (6, 2, 6),
                                   (5, 2, 7), (6, 2, 8), (5, 3, 2), (4, 3, 3), (5, 4, 2)])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** -465, 2.0 ** 300])
def test_matches_bruteforce(n, r, K, scale):
    V = inputs.factor(n, r, seed=17 * n + K) * scale
    f, z, sets = _run(V, K)
    f1, z1, sets1 = _run(V / scale, K)
    assert sets == sets1 and np.array_equal(z, z1)
    if K ** n <= 300000:
        ref, _ = oracle.bruteforce(V / scale, K)
        assert abs(f1 - ref) <= 1e-9 * ref
    assert abs(oracle.objective(V, K, z) - f) <= 1e-12 * f


@pytest.mark.parametrize("kind", ["small_rows", "zero_rows", "equal_rows"])
@pytest.mark.parametrize("K", [2, 3, 4])
def test_structured(kind, K):
    V = inputs.factor(9, 2, seed=K)
    if kind == "small_rows":
        V[::3] *= 1e-45
        V[1] *= 1e-9
    elif kind == "zero_rows":
        V[[0, 4]] = 0
    else:
        V[3:6] = V[2]
    f, z, _ = _run(V, K)
    ref, _ = oracle.bruteforce(V, K)
    assert abs(f - ref) <= 1e-9 * ref
    assert abs(oracle.objective(V, K, z) - f) <= 1e-12 * f


@pytest.mark.parametrize("n,K", [(12, 3), (16, 2), (12, 4)])
def test_matches_oracle_enumeration(n, K):
    V = inputs.factor(n, 2, seed=n + K, scales=(2.0, 1.0))
    f, z, sets = _run(V, K)
    ref = oracle.enumerate_vertices(V, K)
    assert abs(f - ref[0]) <= 1e-9 * ref[0] and sets == ref[2]["full_rank"]
    assert abs(oracle.objective(V, K, z) - f) <= 1e-12 * f
