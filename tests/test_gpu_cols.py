"""The column-strip form: every instance against the oracle and against the
global-memory form, at the edges of its layouts (one-row lattices, wraps of
length 1 and 2, open edges, strips of one row, planes of exactly one CTA's
threads, bands split among the CTAs of a cluster, columns that leave part of a
task empty)."""
import numpy as np
import pytest

import oracle as O
from paper_1105_5481_gb300 import inputs as I

pytestmark = pytest.mark.gpu
TOL = {"fp64": 1e-10, "fp32": 1e-5}
# FP32: the global-memory form's dots in its default configuration, in its
# order; FP64: another order of the dot sums
SUMS = {"fp64": 1e-13, "fp32": 0.0}


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


CASES = [
    # lattices, periodic, on-site, R
    ([(5, 5), (16, 16), (13, 7), (1, 9), (9, 1), (2, 3), (31, 33), (40, 64)], (True, True), True, 16),
    ([(5, 5), (17, 4), (64, 3), (33, 31)], (False, True), False, 13),
    ([(512, 5), (100, 129), (3, 300), (511, 2)], (True, False), True, 3),
    ([(5, 4, 3), (8, 8, 8), (1, 1, 7), (2, 2, 2), (16, 32, 9)], (True, True, True), True, 5),
    ([(7, 3, 20), (22, 23, 10)], (False, True, False), False, 17),
    ([(128, 128), (97, 131), (64, 256)], (True, True), True, 32),  # line traversal
    ([(16, 16, 33), (20, 24, 24)], (True, True, False), True, 64),
    ([(250, 260), (300, 200)], (True, True), True, 4),             # more than one CTA holds
    ([(20, 25, 60), (21, 20, 70)], (True, True, False), True, 2),
]


@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_column_strips_match_oracle_and_global_form(K, prec, case):
    Ls, per, onsite, R = CASES[case]
    hs, Hs, ab, Ms, seeds = [], [], [], [], []
    for i, L in enumerate(Ls):
        n = int(np.prod(L))
        on = I.onsite_disorder(50 + i, n, 2.0) if onsite else None
        H = O.lattice_hamiltonian(L, periodic=per, onsite=on)
        Hs.append(H)
        hs.append(K.kpm_create_stencil(len(L), L, periodic=per, onsite=on))
        ab.append(O.rescale(*O.gershgorin(H), eps=0.01))
        Ms.append((2, 32, 34, 70)[i % 4])
        seeds.append(9 + i)
    a, b = [x[0] for x in ab], [x[1] for x in ab]
    with K.kpm_batch_create(hs, Ms, R, a, b, seeds, precision=prec) as bt:
        # FP32 runs a column on one CTA; FP64 splits a large one
        assert K.kpm_batch_get_columns(bt) == (prec == "fp64" or case < len(CASES) - 2)
        mu = K.kpm_batch_run(bt)
        assert np.array_equal(mu, K.kpm_batch_run(bt))   # replays are bitwise equal
        parts = bt.split(mu)
        K.kpm_batch_set_config(bt, 4, 4, 100)            # the global-memory form
        assert not K.kpm_batch_get_columns(bt)
        ref = bt.split(K.kpm_batch_run(bt))
    for i, H in enumerate(Hs):
        mu_o, _ = O.moments_doubling(H, a[i], b[i], I.rademacher_block(seeds[i], H.n, R), Ms[i])
        assert np.abs(parts[i] - mu_o).max() <= TOL[prec], Ls[i]
        assert np.abs(parts[i] - ref[i]).max() <= SUMS[prec], Ls[i]


def test_column_strips_report_divergence(K):
    with K.kpm_create_stencil(2, (24, 24)) as h, \
            K.kpm_batch_create([h], [64], 8, [2.0], [0.0], [1]) as bt:   # the spectrum is [-4, 4]
        with pytest.raises(K.KPMError) as e:
            K.kpm_batch_run(bt)
        assert e.value.status == K.KPM_EDIVERGE


@pytest.mark.parametrize("fixed", ["1", "0"], ids=["fixed point", "fp64 pipe"])
@pytest.mark.parametrize("L,per,onsite,R,S,M", [
    ((10, 10, 10), (True, True, True), False, 14, 128, 32),
    ((33, 17), (True, False), True, 3, 5, 70),
    ((9, 8, 31), (False, True, True), True, 20, 40, 34),
    ((3, 300), (True, True), False, 1, 700, 2),
])
def test_realisations_in_one_launch_match_single_solves(K, monkeypatch, L, per, onsite, R, S, M, fixed):
    monkeypatch.setenv("KPM_FIXED", fixed)
    n = int(np.prod(L))
    on = I.onsite_disorder(8, n, 2.0) if onsite else None
    H = O.lattice_hamiltonian(L, periodic=per, onsite=on)
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    with K.kpm_create_stencil(len(L), L, periodic=per, onsite=on) as h:
        for s0 in (0, 2):  # and twice with the same plan
            mu, pv = K.kpm_moments(h, M, R, a, b, seed=11, S=S, s0=s0, per_vec=True)
            assert K.kpm_testing_last_step_form(h) == "column strips"
            np.testing.assert_allclose(mu, pv.mean(0), rtol=0, atol=1e-13)
            for s in (0, 1, S // 2, S - 1):
                mu_o, per_o = O.moments_doubling(H, a, b, I.rademacher_block(11, n, R, s=s0 + s), M)
                assert np.abs(pv[s * R:(s + 1) * R] - per_o).max() <= TOL["fp64"]
        # another S on the handle, and a single realisation that can be extended
        mu2, pv2 = K.kpm_moments(h, M, R, a, b, seed=11, S=2, s0=2, per_vec=True)
        assert np.abs(pv2 - pv[:2 * R]).max() <= 1e-12  # another form may take two
        K.kpm_moments(h, M, R, a, b, seed=11, s0=2)
        ext, _ = K.kpm_moments_extend(h, M + 2, R=R, per_vec=True)
        assert np.abs(ext[:M] - pv[:R].mean(0)).max() <= 1e-12
