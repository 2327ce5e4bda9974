"""The per-vector DOS by a Cooley-Tukey step over a divisor of the node count,
against the oracle: divisors that do and do not divide M, more moments than
nodes, node counts without a divisor (the direct sums), and vector counts that
leave part of a group of eight; the temperature integrals spread over CTAs."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


def _pv(seed, nvec, M):
    rng = np.random.default_rng(seed)
    P = rng.standard_normal((nvec, M)) * np.exp(-np.arange(M) / (0.3 * M))
    P[:, 0] = 1.0
    return P


# K = 4096 = 32 x 128, 975 = 25 x 39, 64 = N1 itself, 6 and 97 (prime: direct), 1 (no node pair)
@pytest.mark.parametrize("nvec,M,Kn", [(17, 2048, 4096), (8, 300, 975), (3, 4000, 64), (9, 200, 6),
                                       (2, 600, 97), (5, 1001, 1287), (1, 64, 1), (7, 12, 512)])
def test_split_dos_matches_oracle(K, nvec, M, Kn):
    P = _pv(nvec + M, nvec, M)
    got = K.kpm_stats(P, 2.7, 0.2, Kn)
    ref = O.stats(P, 2.7, 0.2, Kn, "jackson", 0.0)
    for name, g, r in zip(["mu_mean", "mu_err", "E", "rho_mean", "rho_err"], got, ref):
        # an FP64 sum of M terms near the spectrum's edges (1 / sin theta)
        scale = max(1.0, np.abs(r).max())
        np.testing.assert_allclose(g, r, rtol=0, atol=1e-12 * scale * max(1, M / 64), err_msg=name)


@pytest.mark.parametrize("nT,Kn", [(1, 5), (3, 1000), (40, 4096), (400, 300)])
def test_thermo_spread_over_ctas_matches_oracle(K, nT, Kn):
    mu = _pv(5, 1, 128)[0]
    betas = np.geomspace(0.1, 300.0, nT)
    betas[-1] = np.inf if nT > 1 else betas[-1]
    got = K.kpm_thermo(mu, 3.0, 0.1, Kn, betas, 0.4)
    ref = O.thermo(mu, 3.0, 0.1, Kn, betas, 0.4)
    np.testing.assert_allclose(got, ref, rtol=1e-11, atol=1e-11)
