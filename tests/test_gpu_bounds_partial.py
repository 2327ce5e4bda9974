"""Lanczos bounds of large operators, whose vectors are reorthogonalised only in
the steps that need it: against the oracle's Lanczos with full
reorthogonalisation, at the smallest dimension of that path, with Ritz values
that converge early (every step after that needs it) and late (none does), and
on an operator whose Krylov space ends at once."""
import numpy as np
import pytest

import oracle as O
from paper_1105_5481_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


@pytest.mark.parametrize("L,cplx,W,k", [((256, 256), False, 1.0, 30), ((256, 256), True, 0.0, 50),
                                        ((64, 32, 40), True, 30.0, 120), ((300, 301), False, 60.0, 80)])
def test_partial_reorthogonalisation_matches_full(K, L, cplx, W, k):
    n = int(np.prod(L))
    hop = I.spin_hoppings(L, *I.spins(4, n)) if cplx else None
    on = I.onsite_disorder(4, n, W) if W else None
    H = O.lattice_hamiltonian(L, onsite=on, hop=hop)
    with K.kpm_create_stencil(len(L), L, onsite=on, hop=hop, complex_=cplx) as h:
        emin, emax, _, _ = K.kpm_bounds(h, k, 0.0, seed=9)
    omin, omax, _ = O.lanczos_bounds(H, k, I.lanczos_start(9, n))
    gmin, gmax = O.gershgorin(H)
    omin, omax = max(omin, gmin), min(omax, gmax)
    assert abs(emin - omin) <= 1e-9 * (gmax - gmin)
    assert abs(emax - omax) <= 1e-9 * (gmax - gmin)


def test_invariant_start_vector(K):
    # H = 2.5 on every site and no bonds: the first step ends the Krylov space
    n = 1 << 16
    with K.kpm_create_stencil(2, (256, 256), onsite=np.full(n, 2.5), t=0.0) as h:
        emin, emax, _, _ = K.kpm_bounds(h, 20, 0.0, seed=1)
    assert emin == pytest.approx(2.5, abs=1e-12) and emax == pytest.approx(2.5, abs=1e-12)
