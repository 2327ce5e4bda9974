"""The dense tensor-core products where their exactness in FP32 ends: the slice form
above 4096 rows with its two slice counts, and the residue form with the largest
residues in every term."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


def _coherent(K, h, n, a, b, v0, M):
    """Moments of the n x n matrix of constant h with a constant start block, which is
    the eigenvector of h n, and the exact ones (of the start block's own length)."""
    with K.kpm_create_dense(np.full((n, n), h)) as hd:
        mu, per = K.kpm_moments(hd, M, v0.shape[1], a, b, user_v0=v0, per_vec=True)
        assert K.kpm_testing_last_step_form(hd) == "dense tensor cores"
    x = (np.longdouble(h) * n - b) / a
    exact = np.cos(np.arange(M) * np.arccos(x))
    return per, (v0[0].astype(np.longdouble) ** 2)[:, None] * exact[None, :]


@pytest.mark.parametrize("n", [
    16384,   # beta = 5, 11 slices: 16384 * 32 * 32 = 2^24 in the first slice product
    16392,   # beta = 4, 14 slices: 16392 * 16 * 16
    4104,    # the first sizes of the slice form: beta = 5
])
def test_slices_at_the_exactness_bound(K, monkeypatch, n):
    monkeypatch.setenv("KPM_DENSE_TENSOR", "1")
    # entries and start of 0.99: the first slice of either is 2^beta
    v0 = np.full((n, 8), 0.99) * np.where(np.arange(8) % 2, -1.0, 1.0)
    per, exact = _coherent(K, 0.99, n, 0.99 * n / 1.98, 0.99 * n / 2, v0, 12)
    # an inexact slice product would be off by 2^-24 relative, about 6e-8; FP64's own
    # rounding of n equal terms and 6 products stays below n 2^-53 * 36
    assert np.abs(per - exact).max() <= 36 * n * 2.0**-53


def test_residues_at_the_exactness_bound(K, monkeypatch):
    """Integers that are 64 modulo 128 and modulo 129, the largest balanced residue of
    both, in every element: 4096 * 64 * 64 = 2^24 in the FP32 sums of two products."""
    monkeypatch.setenv("KPM_DENSE_TENSOR", "1")
    n = 4096
    F = 64 + 128 * 129 * int(0.97 * 2**55 / (128 * 129))     # of 55 bits, a multiple of 4
    assert F % 129 == 64 and F % 128 == 64 and F % 4 == 0 and 2**54 < F < 2**55
    h = F * 2.0**-68                     # 2 h = F 2^-67; n h = F 2^-56 < 1
    v = F * 2.0**-55
    assert h * 2.0**68 == F and v * 2.0**55 == F
    v0 = np.full((n, 6), v) * np.where(np.arange(6) % 2, -1.0, 1.0)
    per, exact = _coherent(K, h, n, 1.0, 0.0, v0, 12)
    # a residue off by one moves the product by at least 2^-7 of its largest value
    assert np.abs(per - exact).max() <= 36 * n * 2.0**-53
