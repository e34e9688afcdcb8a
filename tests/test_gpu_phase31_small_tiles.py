"""The fused launch (phase 3 with the next phase 1) on 128 x 32 tiles, the
default of lattices up to L = 1024: the checks that test_gpu_phase31 makes on
the taller tiles, the assignment rule and a trace that grows between calls."""
import numpy as np
import pytest

import oracle
import test_gpu_phase31 as base
from test_gpu_phase31 import sw  # noqa: F401  (the fixture)

pytestmark = pytest.mark.gpu

SHAPE = 7


@pytest.mark.parametrize("L", [33, 130, 257, 500, 1001])
def test_split_calls_with_queries_between(sw, L):  # noqa: F811
    base.test_split_calls_with_queries_between(sw, SHAPE, L)


@pytest.mark.parametrize("asynchronous", [False, True])
def test_set_state_between_fused_calls(sw, asynchronous):  # noqa: F811
    base.test_set_state_between_fused_calls(sw, SHAPE, asynchronous)


def test_every_call_length(sw):  # noqa: F811
    base.test_every_call_length(sw, SHAPE)


@pytest.mark.parametrize("L", [130, 300])
def test_assignment_rule_and_trace_growth(sw, L):  # noqa: F811
    seed, n = 5, 1030
    with base.make(sw, L, base.BETA_C, seed, SHAPE) as lat:
        lat.set_rule(sw.SW_RULE_ASSIGN)
        for c in (2, 1021, 1, 6):  # the trace holds 1024 sweeps at first
            lat.sweep(c)
        E, M = lat.observables(0, n)
        spins = lat.spins()
    want_s, want_E, want_M, _ = oracle.run(L, base.BETA_C, seed, n, rule="assign")
    assert np.array_equal(E, want_E) and np.array_equal(M, want_M)
    assert np.array_equal(spins, want_s)
