"""CSR rows longer than the padded form takes, FP32 vectors: an
empty row and lengths on every side of the batches of four that are fetched ahead,
real and complex, against the oracle per vector."""
import numpy as np
import pytest

import oracle as O
from paper_1105_5481_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


def _matrix(n, cplx):
    """Hermitian; row 5 is empty, the others hold 3 to 19 entries."""
    rng = np.random.default_rng(n)
    A = np.zeros((n, n), dtype=complex)
    for i in range(n):
        for s in range(1, 1 + i % 13):
            j = (i + 3 * s * s) % n
            if j != i and i != 5 and j != 5:
                A[i, j] = rng.uniform(-1, 1) + (1j * rng.uniform(-1, 1) if cplx else 0)
                A[j, i] = np.conj(A[i, j])
    i, j = np.nonzero(A)
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(i, minlength=n))])
    return O.CSR(n, rowptr, j, A[i, j] if cplx else A[i, j].real)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,R", [(97, 1), (257, 9), (640, 40), (61, 270)])
def test_csr_rows_fetched_ahead(K, n, R, cplx):
    H = _matrix(n, cplx)
    lengths = np.diff(H.rowptr)
    assert lengths.min() == 0 and lengths.max() > 8
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    with K.kpm_create_csr(n, H.rowptr, H.col, H.val, complex_=cplx) as h:
        _, per = K.kpm_moments(h, 40, R, a, b, seed=7, precision="fp32", per_vec=True)
    _, per_o = O.moments_doubling(H, a, b, I.random_block(7, n, R, cplx), 40)
    assert np.abs(per - per_o).max() <= 1e-5
