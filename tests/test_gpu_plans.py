"""Plans that stand beside each other: calls that alternate the realisations S, or
the vectors R within one padded width, or start blocks of the caller's and of the
library's making, replace none of them (nothing is allocated when a shape comes again)
and keep their bits; the column tasks of an operator too
large for their fixed-point unit run beside a step chain in fixed point."""
import numpy as np
import pytest

import oracle as O
from paper_1105_5481_gb300 import inputs as I

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


@pytest.mark.parametrize("L,onsite,strips", [((150, 150), True, True), ((24, 25, 26), False, False)])
def test_alternating_shapes_keep_their_plans(K, L, onsite, strips):
    n = int(np.prod(L))
    on = I.onsite_disorder(5, n, 2.0) if onsite else None
    H = O.lattice_hamiltonian(L, onsite=on)
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    M = 48
    shapes = [(16, 4), (1, 4), (16, 3), (1, 3), (2, 4)]
    with K.kpm_create_stencil(len(L), L, onsite=on) as h:
        def call(S, R):
            return K.kpm_moments(h, M, R, a, b, seed=3, S=S, per_vec=True)[1], K.kpm_testing_last_step_form(h)

        first = [call(*s) for s in shapes]
        assert {f for _, f in first} == ({"column strips", "fused step"} if strips else {"fused step"})
        K.kpm_testing_fail_allocations(0)
        try:
            for _ in range(3):
                for s, (pv, form) in zip(shapes, first):
                    again, f = call(*s)
                    assert f == form and np.array_equal(again, pv), s
        finally:
            K.kpm_testing_fail_allocations(-1)
        # more shapes than are kept, and the first ones again
        for S in range(3, 11):
            assert np.abs(call(S, 4)[0] - first[0][0][:4 * S]).max() <= 1e-12
        for s, (pv, _) in zip(shapes, first):
            assert np.array_equal(call(*s)[0], pv), s
    # each S against the same realisations alone
    assert np.abs(first[0][0][:4] - first[1][0]).max() <= 1e-12
    assert np.abs(first[0][0][:8] - first[4][0]).max() <= 1e-12


@pytest.mark.parametrize("user_first", [False, True])
def test_alternating_start_blocks_keep_their_plans(K, user_first):
    """A user's start block on the FP64 pipe, one of sites in fixed point."""
    L, M = (150, 150), 48
    on = I.onsite_disorder(5, 22500, 2.0)
    H = O.lattice_hamiltonian(L, onsite=on)
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    v0 = I.random_block(7, H.n, 4, False)
    sites = [0, 77, 11111, 22499]
    with K.kpm_create_stencil(2, L, onsite=on) as h:
        def call(user):
            if user:
                return K.kpm_moments(h, M, 4, a, b, user_v0=v0, per_vec=True)[1]
            return K.kpm_ldos_moments(h, sites, M, a, b, precision="fp64")

        first = {user: call(user) for user in (user_first, not user_first)}
        K.kpm_testing_fail_allocations(0)
        try:
            for _ in range(3):
                for user in (True, False):
                    assert np.array_equal(call(user), first[user])
        finally:
            K.kpm_testing_fail_allocations(-1)
    assert np.abs(first[True] - O.moments_doubling(H, a, b, v0, M)[1]).max() <= 1e-10
    unit = np.zeros((H.n, 4))
    unit[sites, np.arange(4)] = np.sqrt(H.n)
    assert np.abs(first[False] - O.moments_doubling(H, a, b, unit, M)[1]).max() <= 1e-10


def test_kept_launches_give_way_without_memory(K):
    """An allocation that fails while another (S, R) is kept: the kept one goes, the call
    takes its form all the same, and the other one comes back when it is asked for."""
    L, M, R = (10, 10, 10), 32, 4
    with K.kpm_create_stencil(3, L) as h:
        def call(S):
            pv = K.kpm_moments(h, M, R, 6.1, 0.0, seed=3, S=S, per_vec=True)[1]
            return pv, K.kpm_testing_last_step_form(h)

        big, form = call(64)
        assert form == "column strips"
        want = call(32)
        for after in range(3):
            assert np.array_equal(call(64)[0], big)
            K.kpm_testing_fail_allocations(after)
            try:
                pv, form = call(33 + after)      # a shape that is not kept
            finally:
                K.kpm_testing_fail_allocations(-1)
            assert form == "column strips"
            assert np.abs(pv - big[:(33 + after) * R]).max() <= 1e-13
        assert np.array_equal(call(32)[0], want[0])


@pytest.mark.parametrize("S", [2, 16])
def test_large_lattice_beside_a_fixed_point_chain(K, S):
    """90,000 sites: a chain in fixed point (unit 2^-52), column tasks on the FP64 pipe."""
    L, M, R = (300, 300), 24, 2
    on = I.onsite_disorder(6, 90000, 2.0)
    H = O.lattice_hamiltonian(L, onsite=on)
    a, b = O.rescale(*O.gershgorin(H), eps=0.01)
    with K.kpm_create_stencil(2, L, onsite=on) as h:
        for _ in range(2):
            _, pv = K.kpm_moments(h, M, R, a, b, seed=4, S=S, per_vec=True)
            _, one = K.kpm_moments(h, M, R, a, b, seed=4, per_vec=True)
            assert np.abs(pv[:R] - one).max() <= 1e-12
    for s in (0, S - 1):
        per = O.moments_doubling(H, a, b, I.rademacher_block(4, H.n, R, s=s), M)[1]
        assert np.abs(pv[s * R:(s + 1) * R] - per).max() <= 1e-10
