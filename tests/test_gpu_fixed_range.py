"""Fixed-point values that leave their range (bounds that miss the spectrum): the
moments of the products before are kept, as on the FP64 pipe, the later ones are NaN,
into device outputs too; and a spectrum outside the bounds by less than what
KPM_EDIVERGE allows is none of it."""
import numpy as np
import pytest
import torch

from paper_1105_5481_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


@pytest.mark.parametrize("L,S,R,form", [((150, 150), 1, 2, "fused step"), ((150, 150), 16, 4, "column strips"),
                                        ((10, 10, 10), 128, 14, "column strips")])
def test_moments_before_the_range_is_left(K, monkeypatch, L, S, R, form):
    if S == 1:
        monkeypatch.setenv("KPM_COLRES", "0")
    n, M = int(np.prod(L)), 96
    on = I.onsite_disorder(5, n, 2.0)

    def solve(fixed):
        mu = torch.full((M,), 7.0, device="cuda", dtype=torch.float64)
        with K.kpm_create_stencil(len(L), L, onsite=on) as h:
            # the spectrum reaches 1.6 times the bounds: T_n grows by e per product
            K.kpm_moments(h, M, R, 0.65 * (2 * len(L) + 1), 0.0, seed=2, S=S, out=mu)
            assert not fixed or K.kpm_testing_last_step_form(h) == form
            first = mu.cpu().numpy().copy()
            if S == 1:                                # a continued solve stays flagged
                ext = K.kpm_moments_extend(h, M + 8, out=torch.empty(M + 8, device="cuda", dtype=torch.float64))
                assert np.array_equal(ext.cpu().numpy()[:M], first, equal_nan=True)
            host = np.zeros(M)
            with pytest.raises(K.KPMError) as e:      # and host outputs report it, written
                K.kpm_moments(h, M, R, 0.65 * (2 * len(L) + 1), 0.0, seed=2, S=S, out=host)
            assert e.value.status == K.KPM_EDIVERGE
            assert np.array_equal(host, first, equal_nan=True)
        return first

    fix = solve(True)
    monkeypatch.setenv("KPM_FIXED", "0")
    pipe = solve(False)
    assert np.isfinite(pipe).all()
    ok = np.isfinite(fix)
    m = int(ok.sum())
    assert 8 <= m < M and ok[:m].all() and not ok[m:].any()
    assert np.abs(fix[:m] / pipe[:m] - 1).max() <= 1e-9


@pytest.mark.parametrize("cplx", [False, True])
def test_a_spectrum_just_outside_the_bounds(K, monkeypatch, cplx):
    """Sites without bonds, the first 1e-10 outside: its entry grows past sqrt(N) =
    2^6, the format's range, by 1e-7 while every moment stays within 1 + 1e-6."""
    monkeypatch.setenv("KPM_COLRES", "0")
    L, n, M = (64, 64), 4096, 64
    x = np.linspace(-0.9, 0.9, n)
    x[0] = 1.0 + 1e-10
    with K.kpm_create_stencil(2, L, onsite=x, t=0.0, complex_=cplx) as h:
        mu = K.kpm_ldos_moments(h, [0, 1, 4095], M, 1.0, 0.0, precision="fp64")
    k = np.arange(M)
    np.testing.assert_allclose(mu[0], np.cosh(k * np.arccosh(x[0])), rtol=0, atol=1e-12)
    for j, i in ((1, 1), (2, 4095)):
        np.testing.assert_allclose(mu[j], np.cos(k * np.arccos(x[i])), rtol=0, atol=1e-12)
