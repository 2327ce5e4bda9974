"""Long CSR rows in 64-bit fixed point.  The low words of the coefficients do not
shrink with them, so a long row's sum of low-word products passes 64 bits unless it is
carried on the way.  Operators with a closed form drive that sum to its largest value:
k sites all joined by c u_i conj(u_j), with 2 c 2^56 an integer whose low 28 bits are
close to 2^27 and a unit vector as the start, whose image has low words close to 2^31
in every entry.  The spectrum is {0, c k}: mu_3 of a site of the block is T_3(c k) / k.

A carry lost once in every row moves each entry of v_2 by 256 units 2^-q and mu_3 by
2 * 256 * 2^-q * c k / sqrt(N); the moments must be right to a quarter of that."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


def _block(k, n, cplx):
    """Rows of k entries on the sites 0 .. k-1 of n (the others empty), and 2 c 2^56."""
    h = int(1.8 / k * 2.0**56) >> 28 << 28 | 0x7FFFFF0   # low word 2^27 - 16
    c = h * 2.0**-57
    assert c * 2.0**57 == h
    assert k * 0x7FFFFF0 * 16 * 0x7FFFFF0 > 2**63         # what the row's low words add up to
    u = np.array([1, 1j, -1, -1j])[np.arange(k) % 4] if cplx else np.where(np.arange(k) % 3, 1.0, -1.0)
    val = c * np.outer(u, np.conj(u))
    rowptr = np.minimum(np.arange(n + 1), k) * k
    return rowptr.astype(np.int64), np.tile(np.arange(k, dtype=np.int32), k), val.ravel(), h


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("nsites", [1, 64])   # rows fetched ahead, and the general form
@pytest.mark.parametrize("k,n", [(33, 4096), (40, 4096), (64, 64), (200, 4096), (1000, 4096),
                                 (2048, 4096), (4000, 4096)])
def test_low_words_of_long_rows_are_carried(K, k, n, nsites, cplx):
    rowptr, col, val, h = _block(k, n, cplx)
    x = np.longdouble(h) * k / 2**57
    sites = [j % k for j in range(nsites)]
    with K.kpm_create_csr(n, rowptr, col, val, complex_=cplx) as hd:
        mu = K.kpm_ldos_moments(hd, sites, 4, 1.0, 0.0, precision="fp64")
    q = 61 - (int(np.log2(n)) + 1) // 2
    lost = 2 * 256 * 2.0**-q * float(x) / np.sqrt(n)
    assert np.abs(mu[:, 3] - (4 * x**3 - 3 * x) / k).max() <= lost / 4
    assert np.abs(mu[:, 1] - x / k).max() <= lost / 4
