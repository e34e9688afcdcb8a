"""Which batches take the fused schedule: by their tile shape, the same whether
it was named, tuned or set in the environment; a batch on the default's small
tiles moves to the large ones for it."""
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


def accepts(sw, b):
    try:
        sw.sw_batch_set_schedule(b, sw.SW_SCHEDULE_FUSED)
        return True
    except sw.SWError as e:
        assert e.status == sw.SW_EINVAL
        return False
    finally:
        sw.sw_batch_destroy(b)


@pytest.mark.parametrize("shape", range(10))
def test_one_answer_a_shape(sw, shape, monkeypatch):
    want = shape in (4, 6)
    assert accepts(sw, sw.sw_batch_create([100], [0.4], [1], shape=shape)) == want
    sw.sw_tune_shape(7, shape)
    try:
        assert accepts(sw, sw.sw_batch_create([100], [0.4], [1])) == want
    finally:
        sw.sw_tune_shape(7, -1)
    monkeypatch.setenv("SW_TILE_SHAPE", str(shape))
    assert accepts(sw, sw.sw_batch_create([100], [0.4], [1])) == want


def test_the_default_moves(sw):
    reps = [(100, BETA_C, 1), (65, 0.3, 2), (300, 0.5, 3)]
    L, beta, seed = (list(x) for x in zip(*reps))
    b = sw.sw_batch_create(L, beta, seed)
    try:
        sw.sw_batch_sweep(b, 3)
        sw.sw_batch_set_schedule(b, sw.SW_SCHEDULE_FUSED)
        sw.sw_batch_sweep(b, 4)
        sw.sw_batch_set_schedule(b, sw.SW_SCHEDULE_PHASES)
        sw.sw_batch_sweep(b, 2)
        for slot, (Lr, br, sr) in enumerate(reps):
            want_s, want_E, want_M, _ = oracle.run(Lr, br, sr, 9)
            assert np.array_equal(sw.sw_batch_spins(b, slot, Lr), want_s), slot
            E, M = sw.sw_batch_observables(b, slot, 0, 9)
            assert np.array_equal(E, want_E) and np.array_equal(M, want_M), slot
    finally:
        sw.sw_batch_destroy(b)
    assert not accepts(sw, sw.sw_batch_create([64, 32], [0.4, 0.4], [1, 2]))
