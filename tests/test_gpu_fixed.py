"""FP64 calls on stencils and CSR operators in 64-bit fixed point: against the oracle and against
the FP64 pipe (KPM_FIXED=0), per vector, on ragged lattices, wraps of length 1
and 2, open edges, dilution and disorder, one to many columns, start blocks
written on the device, several realisations, continued solves, and calls that
stay on the FP64 pipe (a user's start block, coefficients out of range); bounds
that miss the spectrum are still reported."""
import numpy as np
import pytest

import oracle as O
from paper_1105_5481_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


@pytest.fixture(autouse=True)
def chain(monkeypatch):
    monkeypatch.setenv("KPM_COLRES", "0")   # small lattices too take the step chain


CASES = [
    # L, periodic, complex, on-site, dilution, R
    ((64, 64, 33), (True, True, True), True, False, False, 3),
    ((17, 9, 12), (True, False, True), True, True, True, 5),
    ((2, 1, 7), (True, True, True), True, True, False, 4),
    ((150, 90), (True, True), False, True, False, 8),
    ((31, 40), (False, True), False, False, False, 13),
    ((40, 25), (True, False), True, False, True, 1),
    ((300,), (False,), False, True, False, 2),
    ((1, 2, 1), (False, False, False), False, True, False, 3),
]


def _make(K, L, per, cplx, onsite, dilute, seed=3):
    n, d = int(np.prod(L)), len(L)
    hop = I.spin_hoppings(L, *I.spins(seed, n)) if cplx else None
    on = I.onsite_disorder(seed, n, 2.0) if onsite else None
    mask = I.dilution_mask(seed, n, d, 0.2) if dilute else None
    H = O.lattice_hamiltonian(L, periodic=per, onsite=on, hop=hop, mask=mask)
    h = K.kpm_create_stencil(d, L, periodic=per, onsite=on, hop=hop, bond_mask=mask, complex_=cplx)
    return H, h


@pytest.mark.parametrize("case", range(len(CASES)))
def test_fixed_point_matches_oracle_and_fp64_pipe(K, monkeypatch, case):
    L, per, cplx, onsite, dilute, R = CASES[case]
    H, h = _make(K, L, per, cplx, onsite, dilute)
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    M = 64
    v0 = I.random_block(7, H.n, R, cplx)
    mu_o, per_o = O.moments_doubling(H, a, b, v0, M)
    with h:
        runs = [K.kpm_moments(h, M, R, a, b, seed=7, per_vec=True)[1] for _ in range(3)]
        assert np.array_equal(runs[0], runs[1]) and np.array_equal(runs[0], runs[2])
        # a continued solve is the uninterrupted one's bits
        K.kpm_moments(h, 20, R, a, b, seed=7)
        _, ext = K.kpm_moments_extend(h, M, R=R, per_vec=True)
        assert np.array_equal(ext, runs[0])
        # realisations in turn
        _, pv = K.kpm_moments(h, M, R, a, b, seed=7, S=2, per_vec=True)
        assert np.abs(pv[:R] - runs[0]).max() <= 1e-13
        # a user's start block stays on the FP64 pipe, and the next call goes back
        _, usr = K.kpm_moments(h, M, R, a, b, user_v0=v0, per_vec=True)
        assert np.abs(usr - per_o).max() <= 1e-10
        assert np.array_equal(K.kpm_moments(h, M, R, a, b, seed=7, per_vec=True)[1], runs[0])
        # another (a, b): the fixed-point operator follows
        a2, b2 = 1.3 * a, b + 0.1 * a
        _, sc = K.kpm_moments(h, M, R, a2, b2, seed=7, per_vec=True)
    assert np.abs(runs[0] - per_o).max() <= 1e-10
    assert np.abs(sc - O.moments_doubling(H, a2, b2, v0, M)[1]).max() <= 1e-10
    monkeypatch.setenv("KPM_FIXED", "0")
    H, h = _make(K, L, per, cplx, onsite, dilute)
    with h:
        pipe = K.kpm_moments(h, M, R, a, b, seed=7, per_vec=True)[1]
    # both carry rounding of order 2^-53 per product; 64 moments of one vector
    assert np.abs(runs[0] - pipe).max() <= 1e-12


def test_local_moments_in_fixed_point(K):
    L = (23, 19, 5)
    H, h = _make(K, L, (True, True, False), True, True, False)
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    sites = [0, 5, 17, H.n - 1]
    with h:
        mu = K.kpm_ldos_moments(h, sites, 96, a, b, precision="fp64")
    assert np.abs(mu - O.ldos_exact(H, a, b, sites, 96)).max() <= 1e-10


def test_out_of_range_calls(K):
    L = (40, 30)
    H, h = _make(K, L, (True, True), False, True, False)
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    with h:
        for f in (0.5, 0.3, 0.05):        # the spectrum outside the bounds, mildly to absurdly
            with pytest.raises(K.KPMError) as e:
                K.kpm_moments(h, 200, 4, f * a, b, seed=1)
            assert e.value.status == K.KPM_EDIVERGE
        mu = K.kpm_moments(h, 64, 4, a, b, seed=1)   # and the handle is fine afterwards
    mu_o, _ = O.moments_doubling(H, a, b, I.rademacher_block(1, H.n, 4), 64)
    assert np.abs(mu - mu_o).max() <= 1e-10


@pytest.mark.parametrize("big", [3.0, 300.0])
def test_bonds_that_cancel(K, big):
    """A periodic side of length 2: both bonds join the same pair, and their sum
    (which bounds the spectrum) says nothing about either.  The large pair is out
    of the format's range and stays on the FP64 pipe."""
    L = (2, 37)
    n = 74
    rng = np.random.default_rng(5)
    hop = rng.uniform(-1, 1, (n, 2)) + 1j * rng.uniform(-1, 1, (n, 2))
    hop[0::2, 0] += big
    hop[1::2, 0] -= big           # t_f + conj(t_b) stays of order one
    H = O.lattice_hamiltonian(L, hop=hop)
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    M, R = 64, 3
    mu_o, per_o = O.moments_doubling(H, a, b, I.random_block(7, n, R, True), M)
    with K.kpm_create_stencil(2, L, hop=hop, complex_=True) as h:
        _, per = K.kpm_moments(h, M, R, a, b, seed=7, per_vec=True)
    assert np.abs(per - per_o).max() <= 1e-10


def _csr(n, row, cplx, seed):
    """A Hermitian matrix with up to `row` entries in a row (row 3 has none), a
    diagonal on every second row."""
    rng = np.random.default_rng(seed)
    A = np.zeros((n, n), dtype=complex)
    for s in range(1, (row - 1) // 2 + 1):
        v = rng.uniform(-1, 1, n) + (1j * rng.uniform(-1, 1, n) if cplx else 0)
        for i in range(n):
            j = (i + 1 + 7 * (s - 1)) % n
            if i != j and i != 3 and j != 3:
                A[i, j] += v[i]
                A[j, i] += np.conj(v[i])
    A += np.diag(np.where(np.arange(n) % 2 == 0, rng.uniform(-2, 2, n), 0.0))
    A[3, 3] = 0.0
    i, j = np.nonzero(A)
    rowptr = np.concatenate([[0], np.cumsum(np.bincount(i, minlength=n))])
    return O.CSR(n, rowptr, j, A[i, j] if cplx else A[i, j].real)


@pytest.mark.parametrize("cplx", [False, True])
@pytest.mark.parametrize("n,row,R", [(301, 1, 5), (301, 3, 1), (509, 5, 13), (150, 7, 64), (77, 9, 3),
                                     (400, 13, 8), (333, 21, 2)])
def test_csr_in_fixed_point(K, monkeypatch, cplx, n, row, R):
    """Padded rows of every width and general rows, against the oracle and the FP64 pipe."""
    H = _csr(n, row, cplx, seed=n)
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    M = 64
    _, per_o = O.moments_doubling(H, a, b, I.random_block(7, n, R, cplx), M)

    def solve():
        with K.kpm_create_csr(n, H.rowptr, H.col, H.val, complex_=cplx) as h:
            runs = [K.kpm_moments(h, M, R, a, b, seed=7, per_vec=True)[1] for _ in range(3)]
        assert np.array_equal(runs[0], runs[1]) and np.array_equal(runs[0], runs[2])
        return runs[0]

    fix = solve()
    monkeypatch.setenv("KPM_FIXED", "0")
    assert np.abs(fix - per_o).max() <= 1e-10
    assert np.abs(fix - solve()).max() <= 1e-12


@pytest.mark.parametrize("S", [1, 2])
def test_an_allocation_that_fails(K, S, monkeypatch):
    """Each allocation of the first call in turn: an error or the right moments
    (the operator's fixed-point copy is done without), and then the right moments."""
    if S > 1:
        monkeypatch.delenv("KPM_COLRES")      # the column tasks of several realisations
    L, M, R = (21, 22), 32, 3
    H, h = _make(K, L, (True, True), False, True, False)
    h.close()
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    mu_o = np.mean([O.moments_doubling(H, a, b, I.random_block(7, H.n, R, False, s=s), M)[0]
                    for s in range(S)], axis=0)
    done = 0
    for after in range(14):
        _, h = _make(K, L, (True, True), False, True, False)
        with h:
            K.kpm_testing_fail_allocations(after)
            try:
                mu = K.kpm_moments(h, M, R, a, b, seed=7, S=S)
                assert np.abs(mu - mu_o).max() <= 1e-10
                done += 1
            except K.KPMError as e:
                assert e.status == K.KPM_ENOMEM
            finally:
                K.kpm_testing_fail_allocations(-1)
            for _ in range(2):
                mu = K.kpm_moments(h, M, R, a, b, seed=7, S=S)
                assert np.abs(mu - mu_o).max() <= 1e-10
    assert done > 0


@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("where", ["onsite", "hop", "csr"])
def test_coefficients_that_are_not_finite(K, where, value):
    """They give moments that are not finite, and the error that reports them."""
    L, n = (20, 15), 300
    on = I.onsite_disorder(3, n, 1.0)
    hop = np.ones((n, 2))
    if where == "onsite":
        on[17] = value
    elif where == "hop":
        hop[17, 1] = value
    if where == "csr":
        H = O.lattice_hamiltonian(L, onsite=on)
        val = H.val.copy()
        val[40] = value
        h = K.kpm_create_csr(n, H.rowptr, H.col, val)
    else:
        h = K.kpm_create_stencil(2, L, onsite=on, hop=hop)
    with h:
        with pytest.raises(K.KPMError) as e:
            K.kpm_moments(h, 64, 4, 5.0, 0.0, seed=1)
    assert e.value.status == K.KPM_EDIVERGE
