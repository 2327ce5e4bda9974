"""CSR operators without entries: H = 0, moments T_n(-b / a) exactly, bounds [0, 0]."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n", [1, 2, 5, 300])
def test_operator_without_entries(K, n, cplx):
    a, b, M = 2.0, 0.5, 34
    want = np.cos(np.arange(M) * np.arccos(-b / a))
    with K.kpm_create_csr(n, np.zeros(n + 1, np.int64), np.zeros(0, np.int32),
                          np.zeros(0, complex if cplx else float), complex_=cplx) as h:
        for prec, tol in (("fp64", 1e-13), ("fp32", 1e-5)):
            for R in (1, 9):
                for _ in range(3):   # direct, captured and replayed
                    mu = K.kpm_moments(h, M, R, a, b, seed=3, precision=prec)
                    assert np.abs(mu - want).max() <= tol
            loc = K.kpm_ldos_moments(h, [0, n - 1], M, a, b, precision=prec)
            assert np.abs(loc - want).max() <= tol
        emin, emax, _, _ = K.kpm_bounds(h, 10, 0.01, seed=1)
        assert emin == 0.0 and emax == 0.0
