"""Clusters of phi^4 bricks whose unions fill a warp's list: fields that
alternate in sign along one axis have no bonds along it and, for x0, no
neighbour whose bond would make a union redundant, so a warp of the small
brick (8 x 4 x 4 x 2, below 2^20 sites) lists up to 88 unions in one round
over its 32 sites. Labels and fields against the oracle, bit for bit, with
bond probabilities from 0.5 to 0.95 along the other axes, and a long chain of
an ordered field."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

KAPPA = 0.304


@pytest.fixture(scope="module")
def sw():
    from conftest import build_libsw
    build_libsw()
    import paper_2302_14720_gb300 as sw
    return sw


def staggered(L, axis, p, r, seed):
    """A field along +-r, the sign alternating along x_axis, with lengths that
    bond equal signs with probability about p."""
    rng = np.random.default_rng(seed)
    a = np.sqrt(-np.log1p(-p) / (4.0 * KAPPA)) * (1.0 + 0.1 * rng.normal(size=(L, L, L, L, 1)))
    x = np.indices((L, L, L, L))[3 - axis][..., None]
    return np.ascontiguousarray(a * np.where(x % 2, -1.0, 1.0) * np.asarray(r))


@pytest.mark.parametrize("axis", [0, 1, 2, 3])
@pytest.mark.parametrize("L", [8, 9, 16, 31, 32])
def test_alternating_signs(sw, L, axis):
    seed, t = 5 + L, 3
    r = oracle.phi4_direction(seed, t)
    for p in ([0.5, 0.7, 0.85, 0.95] if L <= 16 else [0.8]):
        phi = staggered(L, axis, p, r, L + axis)
        bonds = oracle.phi4_bonds(phi, KAPPA, seed, t, r)
        want, _ = oracle.phi4_labels(bonds)
        with sw.Phi4(L, KAPPA, seed) as f:
            f.set_field(phi, t)
            assert np.array_equal(f.labels(), want), p
            f.sweep(1)
            assert np.array_equal(f.field(), oracle.phi4_run(L, KAPPA, seed, 1, phi=phi, t0=t)[0]), p


def test_ordered_chain(sw):
    L, seed, n = 12, 21, 60
    with sw.Phi4(L, 0.35, seed, sw.SW_INIT_COLD) as f:
        f.sweep(n)
        assert np.array_equal(f.field(), oracle.phi4_run(L, 0.35, seed, n, cold=True)[0])
