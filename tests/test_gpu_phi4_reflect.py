"""The reflection fma(-2 a, r, phi) of the phi^4 update at every magnitude of
the projection a: zero, subnormal, ordinary, and so large that 2 a leaves the
binary64 range."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


@pytest.mark.parametrize("magnitude", [0.0, 5e-324, 1e-310, 2.0 ** -1022, 1e-200, 1.0, 1e150, 8e307, 1.5e308])
def test_field(sw, magnitude):
    L, kappa, seed, t = 4, 0.304, 31, 2
    r = oracle.phi4_direction(seed, t)
    rng = np.random.default_rng(3)
    phi = np.ascontiguousarray(magnitude * rng.choice([-1.0, 1.0], size=(L, L, L, L, 1)) * r)
    with np.errstate(all="ignore"):
        want = oracle.phi4_run(L, kappa, seed, 1, phi=phi, t0=t)[0]
    with sw.Phi4(L, kappa, seed) as f:
        f.set_field(phi, t)
        f.sweep(1)
        assert np.array_equal(f.field(), want, equal_nan=True)
