"""The one-CTA path above the sides where sw_sweep takes it, bit for bit
against the oracle: from L = 161 on a warp has several segments, and 181 is
the largest side. Reached through a batch's small replicas (both rules,
several sides in one launch, several sweeps and one a chunk) and through
sw_sweep_noalloc."""
import numpy as np
import pytest

import oracle
from workloads import random_spins

pytestmark = pytest.mark.gpu

BETA_C = 0.44068679
SIDES = [2, 31, 33, 64, 97, 105, 128, 133, 144, 145, 157, 160, 161, 162, 165, 170, 176, 177, 180, 181]


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


@pytest.mark.parametrize("rule", ["flip", "assign"])
@pytest.mark.parametrize("beta", [0.1, BETA_C, 0.6, 3.0])
def test_batch(sw, beta, rule):
    n = len(SIDES)
    b = sw.sw_batch_create(SIDES, [beta] * n, [70 + L for L in SIDES], [L % 2 for L in SIDES])
    try:
        sw.sw_batch_set_small(b, 181)
        for slot in range(n):
            sw.sw_batch_set_rule(b, slot, sw.SW_RULE_ASSIGN if rule == "assign" else sw.SW_RULE_FLIP)
        for chunk in (1, 4, 1, 2):
            sw.sw_batch_sweep(b, chunk)
        for slot, L in enumerate(SIDES):
            want_s, want_E, want_M, _ = oracle.run(L, beta, 70 + L, 8, cold=bool(L % 2), rule=rule)
            E, M = sw.sw_batch_observables(b, slot, 0, 8)
            assert np.array_equal(E, want_E) and np.array_equal(M, want_M), L
            assert np.array_equal(sw.sw_batch_spins(b, slot, L), want_s), L
    finally:
        sw.sw_batch_destroy(b)


@pytest.mark.parametrize("L", [161, 165, 176, 180, 181])
def test_noalloc(sw, L):
    import torch
    s0 = random_spins(L, seed=L, p_minus=0.3)
    spins = torch.from_numpy(s0).cuda()
    em = torch.zeros((5, 2), dtype=torch.int64, device="cuda")
    err = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    sw.sw_sweep_noalloc(spins.data_ptr(), L, BETA_C, 9, 3, 5, em.data_ptr(), err.data_ptr())
    torch.cuda.synchronize()
    want_s, want_E, want_M, _ = oracle.run(L, BETA_C, 9, 5, spins=s0, t0=3)
    assert err.item() == 0 and np.array_equal(spins.cpu().numpy(), want_s)
    assert np.array_equal(em[:, 0].cpu().numpy(), want_E) and np.array_equal(em[:, 1].cpu().numpy(), want_M)
