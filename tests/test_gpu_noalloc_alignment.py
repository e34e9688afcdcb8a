"""sw_sweep_noalloc on a caller's lattice that starts on any byte: the wide
loads and stores of the tiled path (L > 181) stay inside the lattice and the
chain is the oracle's."""
import numpy as np
import pytest

import oracle
from workloads import random_spins

pytestmark = pytest.mark.gpu

BETA_C = 0.44068679
GUARD = 64


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


@pytest.mark.parametrize("offset", list(range(16)))
@pytest.mark.parametrize("L", [182, 192, 193, 257, 400])
def test_any_byte(sw, L, offset):
    import torch
    n, seed, t0 = 3, 11 + L, 5
    s0 = random_spins(L, seed=L + offset)
    buf = torch.full((GUARD + 16 + L * L + GUARD,), 77, dtype=torch.int8, device="cuda")
    at = GUARD + offset
    buf[at:at + L * L] = torch.from_numpy(s0.reshape(-1)).cuda()
    em = torch.zeros((n, 2), dtype=torch.int64, device="cuda")
    err = torch.full((1,), -1, dtype=torch.int32, device="cuda")
    torch.cuda.synchronize()
    sw.sw_sweep_noalloc(buf.data_ptr() + at, L, BETA_C, seed, t0, n, em.data_ptr(), err.data_ptr())
    torch.cuda.synchronize()
    got = buf.cpu().numpy()
    want_s, want_E, want_M, _ = oracle.run(L, BETA_C, seed, n, spins=s0, t0=t0)
    assert err.item() == 0
    assert (got[:at] == 77).all() and (got[at + L * L:] == 77).all()
    assert np.array_equal(got[at:at + L * L].reshape(L, L), want_s)
    assert np.array_equal(em[:, 0].cpu().numpy(), want_E) and np.array_equal(em[:, 1].cpu().numpy(), want_M)
