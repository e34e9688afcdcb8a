"""A batch created without a tile shape starts on the tiles that suit its first
replicas and moves to larger ones when it outgrows them; the chains do not
change. The shape a batch is on shows in the bytes it asks for a replica."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

BETA_C = 0.44068679


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


def bytes_on(sw, shape, L=300, sweeps=10):
    b = sw.sw_batch_create([], [], [], shape=shape)
    try:
        return sw.sw_batch_footprint(b, L, sweeps)
    finally:
        sw.sw_batch_destroy(b)


def test_large_replicas_join_a_small_batch(sw):
    b = sw.sw_batch_create([100, 333], [BETA_C, 0.5], [1, 2])
    reps = {0: (100, BETA_C, 1, 7), 1: (333, 0.5, 2, 7)}
    try:
        assert sw.sw_batch_footprint(b, 300, 10) == bytes_on(sw, 7)
        sw.sw_batch_sweep(b, 3)
        for k in range(5):  # 640 tiles of 128 x 64
            before = sw.sw_batch_info(b)[2]
            need = sw.sw_batch_footprint(b, 1024, 1)
            slot = sw.sw_batch_add(b, 1024, 0.43 + 0.01 * k, 10 + k)
            assert sw.sw_batch_info(b)[2] - before <= need
            reps[slot] = (1024, 0.43 + 0.01 * k, 10 + k, 4)
        assert sw.sw_batch_footprint(b, 300, 10) == bytes_on(sw, 6)
        sw.sw_batch_sweep(b, 4)
        for slot, (L, beta, seed, n) in reps.items():
            want_s, want_E, want_M, _ = oracle.run(L, beta, seed, n)
            assert sw.sw_batch_get_sweep(b, slot) == n
            assert np.array_equal(sw.sw_batch_spins(b, slot, L), want_s), slot
            E, M = sw.sw_batch_observables(b, slot, 0, n)
            assert np.array_equal(E, want_E) and np.array_equal(M, want_M), slot
    finally:
        sw.sw_batch_destroy(b)


def test_many_small_replicas(sw):
    n0, n1 = 600, 20
    b = sw.sw_batch_create([16] * n0, [BETA_C] * n0, list(range(n0)))
    try:
        sw.sw_batch_sweep(b, 2)
        for k in range(n1):
            sw.sw_batch_add(b, 16, BETA_C, n0 + k)
        assert sw.sw_batch_footprint(b, 300, 10) == bytes_on(sw, 2)
        sw.sw_batch_remove(b, 5)
        sw.sw_batch_sweep(b, 3)
        for slot in (0, 4, 6, 599, 600, 619):
            n = 5 if slot < n0 else 3
            want_s, want_E, _, _ = oracle.run(16, BETA_C, slot, n)
            assert np.array_equal(sw.sw_batch_spins(b, slot, 16), want_s), slot
            assert np.array_equal(sw.sw_batch_observables(b, slot, 0, n)[0], want_E), slot
    finally:
        sw.sw_batch_destroy(b)


@pytest.mark.parametrize("shape", [7, 6])
def test_a_named_shape_stays(sw, shape):
    b = sw.sw_batch_create([64], [BETA_C], [1], shape=shape)
    try:
        for k in range(6):
            sw.sw_batch_add(b, 1024, BETA_C, k)
        assert sw.sw_batch_footprint(b, 300, 10) == bytes_on(sw, shape)
    finally:
        sw.sw_batch_destroy(b)
