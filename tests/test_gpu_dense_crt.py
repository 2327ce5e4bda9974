"""The dense product on the tensor cores by residues (n <= 4096) and by slices
(above): odd sizes and vector counts (padded leading dimensions), rows and
columns of very different magnitude, and the last size of the residue form,
against the oracle."""
import numpy as np
import pytest

import oracle as O
from paper_1105_5481_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


@pytest.mark.parametrize("n,R,graded", [(7, 1, False), (33, 2, True), (515, 9, False), (512, 15, True),
                                        (1000, 33, True), (4096, 3, False), (4097, 3, False)])
def test_residue_products_match_oracle(K, monkeypatch, n, R, graded):
    monkeypatch.setenv("KPM_DENSE_TENSOR", "1")
    A = I.dense_hermitian(60 + n, n, False)
    if graded:  # rows and columns over twelve orders of magnitude, some exactly zero
        d = 10.0 ** (-6.0 * np.arange(n) / n)
        d[n // 3] = 0.0
        A = A * d[:, None] * d[None, :]
    H = O.from_dense(A)
    a, b = O.rescale(*O.gershgorin(H), 0.01)
    M, seed = 24, 5
    mu_o, per_o = O.moments_doubling(H, a, b, I.random_block(seed, n, R, False), M)
    with K.kpm_create_dense(A) as h:
        mu, per = K.kpm_moments(h, M, R, a, b, seed=seed, per_vec=True)
        assert K.kpm_testing_last_step_form(h) == "dense tensor cores"
    assert np.abs(per - per_o).max() <= 1e-10
    assert np.abs(mu - mu_o).max() <= 1e-10
