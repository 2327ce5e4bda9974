"""Lattices whose rows are taken in natural order (coordinates worked out from the
row index): sides of one, primes, and one past and one short of powers of two, and
start blocks whose column count does not divide the writers' stride, per vector
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


@pytest.mark.parametrize("prec,tol", [("fp32", 1e-5), ("fp64", 1e-10)])
@pytest.mark.parametrize("L,R,cplx", [((1, 9), 3, False), ((2, 3), 1, True), ((3, 1, 5), 7, False),
                                      ((5, 7, 1), 2, True), ((701, 3), 5, False), ((127, 129), 40, True),
                                      ((13, 11, 7), 24, False), ((64, 5, 3), 3, True), ((1, 1, 2), 2, False),
                                      ((40009,), 11, False)])
def test_rows_in_natural_order(K, monkeypatch, L, R, cplx, prec, tol):
    monkeypatch.setenv("KPM_COLRES", "0")
    n = int(np.prod(L))
    on = I.onsite_disorder(3, n, 2.0)
    hop = I.spin_hoppings(L, *I.spins(3, n)) if cplx else None
    H = O.lattice_hamiltonian(L, onsite=on, hop=hop)
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    with K.kpm_create_stencil(len(L), L, onsite=on, hop=hop, complex_=cplx) as h:
        _, per = K.kpm_moments(h, 40, R, a, b, seed=7, precision=prec, per_vec=True)
    _, per_o = O.moments_doubling(H, a, b, I.random_block(7, n, R, cplx), 40)
    assert np.abs(per - per_o).max() <= tol
