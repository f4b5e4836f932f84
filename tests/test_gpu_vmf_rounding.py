"""The proposal's draws and gauge-fixed factors are computed in pairs of FP32
numbers.  Against FP64 numpy on the same random numbers a draw's component is
the rounding of a value within 2^-40 (of a unit vector); a gauge-fixed entry is
the rounding of FP64's value, 2^-50 of the entry allowed for numpy's own."""
import numpy as np
import pytest
import torch

from paper_2602_20376_gb300 import inputs, lrq, proposal

pytestmark = pytest.mark.gpu


def _philox(c, seed):
    m32, sh = np.uint64(0xFFFFFFFF), np.uint64(32)
    c = [np.asarray(x).astype(np.uint64) for x in c]
    k0, k1 = np.uint64(seed & 0xFFFFFFFF), np.uint64(seed >> 32)
    for rnd in range(10):
        if rnd:
            k0, k1 = (k0 + np.uint64(0x9E3779B9)) & m32, (k1 + np.uint64(0xBB67AE85)) & m32
        a, b = np.uint64(0xD2511F53) * c[0], np.uint64(0xCD9E8D57) * c[2]
        c = [(b >> sh) ^ c[1] ^ k0, b & m32, (a >> sh) ^ c[3] ^ k1, a & m32]
    return [((((c[i] << sh) | c[i + 1]) >> np.uint64(11)).astype(np.float64) + 0.5) / 2.0 ** 53 for i in (0, 2)]


def _draws(O, b, S, K, seed):
    o = O[b].astype(np.float64).reshape(16, 10)
    mu = o[:, :8] / np.linalg.norm(o[:, :8], axis=1, keepdims=True)
    kap = np.log1p(np.exp(o[:, 8]))
    cdf = np.cumsum(np.exp(o[:, 9] - o[:, 9].max()))
    s, ctr = np.arange(S), np.zeros(S, np.int64)

    def uniforms(i):
        u = _philox((s[i], np.full(i.size, b), ctr[i], np.full(i.size, 0x564D46)), seed)
        ctr[i] += 1
        return u

    def normals(i):
        u, v = uniforms(i)
        rad = np.sqrt(-2 * np.log(u))
        return rad * np.cos(2 * np.pi * v), rad * np.sin(2 * np.pi * v)

    def gamma(i):
        (a, b2), (c, _) = uniforms(i), uniforms(i)
        return -np.log(a * b2 * c) + 0.5 * normals(i)[0] ** 2

    u, v = uniforms(s)
    m = np.minimum(np.searchsorted(cdf, u * cdf[-1]), 15)
    k = np.minimum(K - 1, (v * K).astype(int))
    kp = kap[m]
    bb = 7 / (2 * kp + np.sqrt(4 * kp ** 2 + 49))
    x0 = (1 - bb) / (1 + bb)
    w, todo = np.zeros(S), s
    while todo.size:
        g1, g2 = gamma(todo), gamma(todo)
        z, t = g1 / (g1 + g2), todo
        wt = (1 - (1 + bb[t]) * z) / (1 - (1 - bb[t]) * z)
        ok = kp[t] * (wt - x0[t]) + 7 * (np.log(1 - x0[t] * wt) - np.log(1 - x0[t] ** 2)) >= np.log(uniforms(todo)[0])
        w[t[ok]] = wt[ok]
        todo = t[~ok]
    n = np.stack([x for _ in range(4) for x in normals(s)], 1)
    n -= (n * mu[m]).sum(1, keepdims=True) * mu[m]
    n /= np.linalg.norm(n, axis=1, keepdims=True)
    x = w[:, None] * mu[m] + np.sqrt(1 - w ** 2)[:, None] * n
    return (x[:, ::2] + 1j * x[:, 1::2]) * np.exp(2j * np.pi * k / K)[:, None]


def _is_rounding(got, ref, tol):
    """got is the FP32 rounding of a value within tol of ref."""
    half = np.maximum(np.spacing(got), np.abs(got - np.nextafter(got, np.float32(0)))).astype(np.float64) / 2
    return np.abs(got.astype(np.float64) - ref) <= half + tol


@pytest.mark.parametrize("K,seed", [(8, 5), (3, 2 ** 40 + 1)])
def test_draws(K, seed):
    B, S = 2, 60000
    g = np.random.Generator(np.random.PCG64(K))
    O = g.standard_normal((B, 160)).astype(np.float32)
    O[:, 8::10] = g.uniform(-4, 60, (B, 16))
    C = torch.empty((B, S, 4), dtype=torch.complex64, device="cuda")
    st = torch.zeros(1, dtype=torch.int32, device="cuda")
    lrq.lrq_vmf_sample(torch.from_numpy(O).cuda(), S, K, seed, C, st)
    assert int(st.item()) == 0
    got = C.cpu().numpy()
    for b in range(B):
        ref = _draws(O, b, S, K, seed)
        for part in ("real", "imag"):
            assert np.all(_is_rounding(getattr(got[b], part), getattr(ref, part), 2.0 ** -40))


def test_gauge():
    B, n, r = 8, 32768, 4
    V = np.stack([inputs.factor(n, r, seed=b, dtype=np.complex64) for b in range(B)])
    lam = (np.abs(V.astype(np.complex128)) ** 2).sum(1)
    Vg, _ = proposal.features(torch.from_numpy(V).cuda(), torch.from_numpy(lam).cuda())
    got, V64 = Vg.cpu().numpy(), V.astype(np.complex128)
    a = np.take_along_axis(V64, (V64.real ** 2 + V64.imag ** 2).argmax(1)[:, None], 1)
    ref = V64 * (a.conj() / np.abs(a))
    for part in ("real", "imag"):
        assert np.all(_is_rounding(getattr(got, part), getattr(ref, part), 2.0 ** -50 * np.abs(V64)))
