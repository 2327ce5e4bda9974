"""The density of states next to the edges of the spectrum: with mu_0 alone it is
1 / (pi a sin theta_k), whose smallest sines, of order 1 / K, must keep their relative
accuracy.  Tolerance: the sine two ulp and its argument half a one, pi half a one, and
the two products and two divisions one rounding each: 10 * 2^-53."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
TOL = 10 * 2.0**-53
PI = np.longdouble("3.14159265358979323846264338327950288")


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


# split sums, direct sums (97 prime, 6 small), odd counts, one node
@pytest.mark.parametrize("M,Kn", [(2048, 4096), (500, 8000), (600, 97), (64, 6), (1001, 1287), (12, 1), (30, 2)])
def test_edges_keep_their_relative_accuracy(K, M, Kn):
    a, b = 4.0, 0.0
    k = np.arange(Kn)
    near = np.minimum(k, Kn - 1 - k)          # the edge's distance in nodes
    s = np.sin(PI * (2 * near + 1).astype(np.longdouble) / (2 * Kn))
    rho = 1 / (PI * a * s)
    pv = np.zeros((3, M))
    pv[:, 0] = 1.0
    for got in (K.kpm_stats(pv, a, b, Kn)[3], K.kpm_dos(pv[0], a, b, Kn)[1],
                -K.kpm_green(pv[0], a, b, Kn)[1].imag.astype(np.longdouble) / PI):
        assert np.abs(got / rho - 1).max() <= TOL
