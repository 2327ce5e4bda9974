"""The error of fixed-point solves against numpy's long double (64 or 113 bits), beside
the FP64 pipe's, at the units the size rule allows: 2^-52 at the end of the real range,
2^-51 above 2^18 complex sites."""
import numpy as np
import pytest

from paper_1105_5481_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


def _reference(L, hop, on, a, v0, M):
    """Per-vector doubling moments of -t sums plus the diagonal, periodic, in long double."""
    d, n = len(L), int(np.prod(L))
    T = np.longdouble if hop is None else np.clongdouble
    idx = np.arange(n).reshape(L[::-1])
    ends = [(np.roll(idx, -1, d - 1 - k).ravel(), np.roll(idx, 1, d - 1 - k).ravel()) for k in range(d)]

    def product(x):
        y = on.astype(np.longdouble) * x
        for k, (f, b) in enumerate(ends):
            y -= x[f] + x[b] if hop is None else hop[:, k].astype(T) * x[f] + np.conj(hop[b, k]).astype(T) * x[b]
        return y / np.longdouble(a)

    def dot(x, y):
        return (np.conj(x) * y).real.sum() / n

    out = np.zeros((v0.shape[1], M), np.longdouble)
    for r in range(v0.shape[1]):
        u = v0[:, r].astype(T)
        v = product(u)
        out[r, 0], out[r, 1] = dot(u, u), dot(u, v)
        for m in range(1, M // 2):
            u, v = v, 2 * product(v) - u
            out[r, 2 * m], out[r, 2 * m + 1] = 2 * dot(u, u) - out[r, 0], 2 * dot(u, v) - out[r, 1]
    return out


@pytest.mark.parametrize("L,cplx,M", [((511, 512), False, 16), ((65, 64, 64), True, 16), ((45, 29), True, 128),
                                      ((19, 18, 21), False, 128)])
def test_error_beside_the_fp64_pipe(K, monkeypatch, L, cplx, M):
    monkeypatch.setenv("KPM_COLRES", "0")
    n, R = int(np.prod(L)), 2
    hop = I.spin_hoppings(L, *I.spins(3, n)) if cplx else None
    on = I.onsite_disorder(3, n, 1.0)
    a = 2.02 * len(L) + 0.5
    ref = _reference(L, hop, on, a, I.random_block(7, n, R, cplx), M)
    rms = {}
    for fixed in ("0", "1"):
        monkeypatch.setenv("KPM_FIXED", fixed)
        with K.kpm_create_stencil(len(L), L, onsite=on, hop=hop, complex_=cplx) as h:
            per = K.kpm_moments(h, M, R, a, 0.0, seed=7, per_vec=True)[1]
        rms[fixed] = float(np.sqrt(((per - ref)[:, 1:] ** 2).mean()))
    # both are a few roundings of 2^-53 at random; the ratio of two such means over 2 M
    # values spreads by 1 / sqrt(M) about 1: at most 2 at M = 16
    assert rms["1"] <= 2 * rms["0"]
    assert rms["1"] <= 4 * 2.0**-53
