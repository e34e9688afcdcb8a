"""The one-CTA path (whole sweeps of a small lattice in one launch), bit for
bit against the oracle at the sides where its pieces change: row words one to
32 columns wide, segments of one to 32 rows and several segments a warp, odd
sides (Philox pairs straddle rows), both new-spin rules, clusters from single
sites to the whole lattice, and calls of one and of several sweeps."""
import numpy as np
import pytest

import oracle
from workloads import random_spins, striped_spins

pytestmark = pytest.mark.gpu

BETA_C = 0.44068679
SIDES = [2, 3, 4, 5, 31, 32, 33, 63, 64, 65, 95, 96, 97, 127, 128, 129, 144, 145, 160, 161, 180, 181, 192, 193, 223,
         224, 225, 255, 256, 257]


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


@pytest.mark.parametrize("rule", ["flip", "assign"])
@pytest.mark.parametrize("L", SIDES)
def test_chain(sw, L, rule):
    seed = 70 + L
    for beta, s0 in [(BETA_C, random_spins(L, seed=L)), (0.1, random_spins(L, seed=L + 1)),
                     (0.6, random_spins(L, seed=L + 2, p_minus=0.03)), (3.0, striped_spins(L, 3))]:
        with sw.Lattice(L, beta, seed) as lat:
            lat.set_rule(sw.SW_RULE_ASSIGN if rule == "assign" else sw.SW_RULE_FLIP)
            lat.set_state(s0, 9)
            lat.sweep(1)
            lat.sweep(4)
            want_s, want_E, want_M, _ = oracle.run(L, beta, seed, 5, spins=s0, t0=9, rule=rule)
            E, M = lat.observables(9, 5)
            assert np.array_equal(E, want_E) and np.array_equal(M, want_M), (L, beta)
            assert np.array_equal(lat.spins(), want_s), (L, beta)
