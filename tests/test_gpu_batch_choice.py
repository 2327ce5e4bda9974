"""The form a batch starts with: the column strips on batches of few or large
instances, the global-memory form where many instances with many vectors fill the
chip (measured 1.2 to 1.5 times as fast there); FP32 moments have the same bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def K(gpu_lib):
    from paper_1105_5481_gb300 import kpm

    return kpm


@pytest.mark.parametrize("L,count,R,strips", [
    ((32, 32), 256, 32, False), ((16, 16, 16), 256, 32, False), ((10, 10, 10), 256, 32, False),
    ((32, 32), 8, 32, True), ((96, 96), 40, 16, True), ((16, 16), 256, 8, True), ((20, 20, 20), 8, 16, True),
])
def test_form_of_a_new_batch(K, L, count, R, strips):
    with K.kpm_create_stencil(len(L), L) as h:
        a = 2.1 * len(L)
        with K.kpm_batch_create([h] * count, [32] * count, R, [a] * count, [0.0] * count,
                                list(range(count))) as bt:
            assert K.kpm_batch_get_columns(bt) == strips
            mu = K.kpm_batch_run(bt)
            K.kpm_batch_set_columns(bt, not strips)
            assert np.array_equal(K.kpm_batch_run(bt), mu)


def test_form_of_a_mixed_batch(K):
    """Large instances run together spill the L2: the strips, although many are small."""
    rng = np.random.default_rng(3)
    sides, Ms = rng.integers(16, 129, 256), 2 * rng.integers(64, 1025, 256)
    hs = {int(L): K.kpm_create_stencil(2, (int(L), int(L))) for L in np.unique(sides)}
    with K.kpm_batch_create([hs[int(L)] for L in sides], [int(m) for m in Ms], 16, [4.2] * 256,
                            [0.0] * 256, list(range(256))) as bt:
        assert K.kpm_batch_get_columns(bt)
    for h in hs.values():
        h.close()


@pytest.mark.parametrize("count,lo,hi,Mlo,Mhi,seed", [(201, 29, 96, 190, 812, 2694),
                                                      (158, 31, 66, 162, 536, 692656)])
def test_form_of_a_ragged_batch(K, count, lo, hi, Mlo, Mhi, seed):
    """Sides between the two kinds: the strips are 1.12 to 1.15 times as fast here."""
    rng = np.random.default_rng(seed)
    sides = rng.integers(lo, hi + 1, count)
    Ms = Mlo + 2 * rng.integers(0, (Mhi - Mlo) // 2 + 1, count)
    hs = {int(L): K.kpm_create_stencil(2, (int(L), int(L))) for L in np.unique(sides)}
    with K.kpm_batch_create([hs[int(L)] for L in sides], [int(m) for m in Ms], 16, [4.2] * count,
                            [0.0] * count, list(range(count))) as bt:
        assert K.kpm_batch_get_columns(bt)
    for h in hs.values():
        h.close()
