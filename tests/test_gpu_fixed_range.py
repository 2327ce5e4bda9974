"""Fixed-point values that leave their range (bounds that miss the spectrum): the
moments of the products before are kept, as on the FP64 pipe, the later ones are NaN,
into device outputs too."""
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
